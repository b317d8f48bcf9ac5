// Device side of the DBaS-Log-MPPI step (arXiv 2504.06437), sm_103a.
//
// One controller's K samples are cut into tiles of S <= 32 samples; a CTA
// processes one tile or a few in a row (batched step: persistent CTAs pull
// (controller, first tile) work items).  Per tile:
//   noise      all threads draw the NLN perturbations of every (sample, step)
//              (Eq. 11) from Philox4x32-10 with counter (k, t, iter) -- no
//              noise crosses HBM -- and keep the clamped controls v = u + du;
//   dynamics   one warp per sample, lanes over steps: explicit Euler for both
//              models is triangular (heading rate -> heading -> velocities
//              -> positions), so a whole trajectory is a few warp prefix
//              scans over time, segment by segment, with one sincos per step;
//              the warp also sums the stage and control costs (Eq. 9);
//   barrier    all threads evaluate the fused barrier sum over every
//              (step, sample) unit, its P shape points and every obstacle
//              (Eq. 5, 13/15): each thread keeps whole units (NPOS world
//              points) in registers as packed pairs, streams the obstacle
//              set from shared memory (broadcast reads), evaluates two points
//              per packed two-lane FP32 instruction, adds two obstacles per
//              approximate reciprocal, and sums each unit's points exactly
//              into a float pair, written over the unit's pose; in large
//              problems only the obstacles near a cell of poses are streamed
//              and the others enter through one polynomial per cell (FarCell);
//   costs      one warp per sample adds the barrier-state and collision costs;
//   partials   the tile's minimum cost, its exponentiated weights, their sum Z
//              and the 2T weighted column sums of the perturbations (Eq. 4);
//   merge      the last tile to finish (a ticket per group of tiles) merges
//              the partials log-sum-exp style against the exact minimum over
//              the tiles, sums the barriers of the samples that carry the
//              weights directly once more if cells were used, then runs the
//              final stage (U*, nominal rollout, S_e, shift).
// The one-controller kernels exist in a 96- and an 80-register form (the
// host picks per launch); the batch kernel's tiles take a padded row stride
// and the one-batch merge (BATCHED in run_tile).  All forms give the same
// results bit for bit.
// The DBaS recursion of Eq. 7, w_t = b_t + gamma (w_{t-1} - beta_d), is
// linear, so its cost sum is evaluated in unrolled form:
//   sum_{t=1..T} w_t = sum_s c_s b_s + beta_0 g1 - gamma beta_d csum,
//   c_s = (1 - gamma^(T-s+1)) / (1 - gamma),  g1 = gamma (1 - gamma^T) / (1 - gamma),
//   csum = sum_s c_s,
// which removes the rounding of the running state w; the sample-independent
// part is formed once in FP64.
//
// Precision: the rollout runs in FP32 in a frame whose origin is the
// measured position (obstacles and reference are moved into it in FP64 then
// rounded), so coordinates stay small; the per-sample cost is an unevaluated
// float pair (TwoSum / TwoProd) relative to a base, the part of the cost
// common to all samples, formed in FP64; the minima, the normaliser Z and the
// weighted sums of perturbations are float pairs, merged across tiles with
// float-pair arithmetic; U* is formed in FP64 from them.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace dbm {

constexpr int kMaxShape = 8;
constexpr int kMaxN = 6;
constexpr int kStatusOk = 0;
constexpr int kStatusTimeout = 1;

// Controller state resident on the device between steps.
struct DevState {
  double S_e;        // exploration rate used by the next step
  double beta;       // barrier state of the last measured state
  double rho, Z;     // last step: global minimum cost and normaliser
  double CB_star;    // last step: barrier cost of the nominal rollout of U*
  double beta_used;  // last step: barrier state the rollouts started from
  double beta_d;     // last step: barrier summed at the goal pose
  double S_e_used;   // last step: exploration rate of the draws
  double u0[2];      // last step: u*_0
  double x1[6];      // last step: state after applying u*_0 (model prediction)
  double C0;         // sum_t gamma u_t^T (S_e Sigma)^-1 u_t of the next step
  double csum, g1;   // DBaS unrolling constants (see above)
  float L00, L10, L11;  // chol(S_e Sigma) of the next step
  unsigned near;     // sum over the cells of their near obstacles' share, in 256ths; zero between steps
  unsigned long long iter;  // Philox counter words 2..3
  int first;         // 1 until the first step
  int status;        // kStatus*
  // grid map, set by the host (mppi_set_grid) and read by the grid form of
  // the step kernels: signed distances (m), sample (i, j) at
  // (grid_ox + i res, grid_oy + j res), stored at grid[j grid_nx + i]; or null
  const float* grid;
  int grid_nx, grid_ny;
  double grid_ox, grid_oy, grid_res;
  float grid_inv_res, grid_pad;
};

// Outputs of a step that the host reads after every step, written by the
// final stage straight into mapped pinned host memory (one-controller
// contexts; null elsewhere), followed there by the shifted sequence (T x 2
// doubles).  seq is stored last, after a system-scope fence, so a host that
// sees the step's seq also sees its u0, sequence and status.  The sequence
// goes out as it is formed, before the nominal rollout, so its way over the
// host link is hidden; copying it after the step cost 10 to 13 us of a small
// controller's 40 us call (unicycle K 256 with u0 alone: 27.5 us).
struct __align__(16) HostOut {
  double u0[2];  // u*_0
  int status;    // kStatus*
  int seq;       // the launch's number (CtrlDesc::seq)
};

// Everything a CTA needs to process one tile of one controller.
struct CtrlDesc {
  int model, K, T, J, P, n;
  int S, NPOS, nTiles, GT, nGroups;
  int chunk;                 // tiles of a CTA of the one-controller kernels
  int nc;                    // far-field cells of a tile (far_cells), 0 = every pair directly
  float r_body;              // largest distance of a shape point from the body's position
  int look_max;              // samples of the second look at most (look_samples)
  float dt, h_eps, C_coll, ln_mu, ln_sigma;
  float umin[2], umax[2];
  float Q[kMaxN], Qf[kMaxN];
  float shape[2 * kMaxShape];
  float g, inv_mass;
  float k_turn;              // arm / I (6-state quadrotor) or 1 / wheelbase (Ackermann)
  float inv_lambda_f;
  double mu_coarse, gamma_bas, R_B_d;
  double umin_d[2], umax_d[2];
  int nscl;
  int sgf_wp;                // Savitzky-Golay window | order << 8, 0 = off (weights: cw)
  double Lsig[3];            // chol(Sigma): l00, l10, l11
  double Sinv[4];            // gamma * Sigma^-1 (row-major; zero when gamma = 0)
  double x_goal[kMaxN];
  uint32_t key0, key1;
  double* U;                 // T x 2 nominal sequence
  float2* cU;                // T: U in FP32 for the next step
  float2* cA;                // T: gamma Sigma^-1 u_t in FP32 (divided by S_e where used)
  float* cw;                 // T: R_B c_{t+1}, weight of step t's barrier sum (then the
                             // smoothing weights, see sgf_table_offset)
  DevState* st;
  const double* obst;        // J x 3 (cx, cy, r), padded to 16 bytes
  const double* x0;          // n (may be overridden per launch)
  const double* xref;        // (T+1) x n
  float* part;               // nTiles x 2T tile weighted sums
  float4* part_rz;           // nTiles x (rho_c hi, lo, Z_c hi, lo), rho relative to base
  float* gpart;              // nGroups x 2T
  float4* gpart_rz;          // nGroups
  unsigned* counters;        // 2 (nGroups + 1): tickets, then minimum words (zero between steps)
  double* costs;             // K
  uint8_t* coll;             // K
  double* Ustar;             // T x 2
  HostOut* host_out;         // device alias of the host mirror, or null
  int seq;                   // what the step leaves there when its outputs are in it
  double* ctl_out;           // the allocation-free step: where the caller keeps its state
  double* u0_out;            // and its control; null elsewhere
};

// The Savitzky-Golay weights (W x W floats, row q: the fit's value at window
// position q) follow the T barrier weights cw at the next 16-byte boundary
// of the same buffer, when the controller smooths its update.
__host__ __device__ inline int sgf_table_offset(int T) { return (T + 3) & ~3; }

// Shared-memory layout of one tile; host and device compute it alike.
// region: poses (overwritten in place by the unit barrier sums) and clamped
// controls of the whole horizon; reused as the raw obstacle staging buffer
// before the rollout, as the per-warp column sums of a merge and as the
// nominal-rollout buffers in the final stage.
struct SmemLayout {
  int obs4, cell, list, region, pose, V, red, Us, Usf, Uf, Af, colhi, collo, scl, xrf, shp, eS, cw, Sk, scH,
      scL, collf, xi, total;
};

__host__ __device__ inline int align_up(int x, int a) { return (x + a - 1) / a * a; }

// Tile merge geometry (merge_partials): row groups over the CTA's threads
// and the bytes of their float-pair column sums.
constexpr int kMergeLoads = 16;   // float2 loads in flight per thread
constexpr int kMergeGroups = 32;  // row groups at most
__host__ __device__ inline int merge_row_groups(int ncol, int nthreads) {
  const int ncp = ncol / 2;
  int rg = ncp > 0 ? nthreads / ncp : nthreads;
  if (rg < 1) rg = 1;
  if (rg > kMergeGroups) rg = kMergeGroups;
  return rg;
}
__host__ __device__ inline int merge_buf_bytes(int ncol, int nthreads) {
  return align_up(8 * merge_row_groups(ncol, nthreads) * (ncol + 1), 16);  // + Z
}

// ---- Far-field cells of the barrier.  A tile's (step, sample) units, in
// step order, are cut into nc cells of consecutive units.  The poses of a
// cell lie in a disc (centre p0, radius R, body included), and over that disc
// the sum of 1 / h_j of the obstacles far from it is a smooth function: its
// Taylor polynomial of degree kFarN about p0, built once per cell, replaces
// one evaluation per point and obstacle.  The obstacles near the cell are
// evaluated one by one as before.  With a_j = |p0 - c_j| - r_j the clearance
// of the centre and t = R / a_j, the terms of degree n of 1 / h_j are at most
// (n + 1) t^n / h_j(p0) anywhere in the disc, so the remainder is at most
// (N + 2) t^(N+1) (1 + t)^2 / (1 - t)^2 of the term itself: 1.2e-7 (one FP32
// rounding) at t = kFarRatio, reached only on the disc's rim by an obstacle at
// the limit, and 2^-9 of that half way in.  A trajectory tile is small beside
// the world: of 200 obstacles about 10 are near a cell of the 65536-sample
// unicycle, of 500 about 40 near one of the crowded quadrotor.  Without and
// with cells, a whole call, all else as it was then: unicycle K 65536, T 100, J 200
// 608 and 365 us; quadrotor K 32768, T 100, J 500, P 7 3090 and 830 us; vehicle
// K 9973, T 73, J 117, P 8 305 and 162 us; 512 mixed controllers in one launch
// 29.2 and 13.8 ms.  Degree 8 against 6 and 10, and cells of 1024 points against one or
// sixteen per tile, come from counting the operations over the presets'
// rollouts (least at 8 and 800 to 2800 points).
constexpr int kFarN = 8;
constexpr int kFarCoef = (kFarN + 1) * (kFarN + 2) / 2;
constexpr float kFarRatio = 0.125f;
constexpr int kFarMin = 12;       // fewer far obstacles than this cost less one by one
constexpr int kFarMaxCells = 8;
constexpr int kFarListMax = 512;  // near obstacles listed per cell at most
struct __align__(16) FarCell {
  float cx, cy, inv_R;
  int n_near;               // obstacles listed, or -1: no polynomial, every obstacle directly
  float2 c[kFarCoef + 1];   // coefficients in the order far_eval takes them, each twice
};
__host__ __device__ inline int far_list_cap(int J) {
  const int c = J < kFarListMax ? J : kFarListMax;
  return (c + 7) & ~7;
}
// Cells of a tile: about kFarCellPoints world points each (a cell's set-up
// takes as long as evaluating some 50 points against every obstacle, and more
// points make it wider), at most one per warp.  None where they would save too
// little: in units of one point against one obstacle, a point costs J directly
// and with cells about 9 (the polynomial), 8 + J / 10 near obstacles (what the
// presets' densities give) and its share of the set-up.  The line of 4e7 over
// the whole step is about 8 us of the GPU, what the last CTA's second look
// (refine_samples) takes when it is needed: the quadrotor at K 4096, T 50,
// J 40 (2e7) took 71.5 us a call without cells, 72 to 80 us with them; at
// K 8192, T 40, J 60 (7e7) 104 us without, 86 to 92 us with them.  None either
// with fewer than kFarMinPerSm samples per SM: there two samples of the second
// look take half as long as the whole step without cells, and cells save
// little (0.72 to 0.99 of the time over 14 drawn problems).
constexpr int kFarCellPoints = 1024;
constexpr int kFarMinPerSm = 4;
constexpr float kFarMinSaved = 4.0e7f;
__host__ __device__ inline float far_setup_ops(int nc, int J, int pts) {
  return nc * (2800.0f + 53.0f * J) / pts;
}
__host__ __device__ inline int far_cells(int K, int T, int S, int P, int J, int npos,
                                         int nthreads, int sms) {
  if (K < kFarMinPerSm * sms) return 0;
  const int gsz = 32 * (npos / P);
  const int groups = (T * S + gsz - 1) / gsz;
  const int pts = T * S * P;
  int nc = pts / kFarCellPoints;
  if (nc > kFarMaxCells) nc = kFarMaxCells;
  if (nc > nthreads / 32) nc = nthreads / 32;
  if (nc > groups) nc = groups;
  if (nc < 1) nc = 1;
  return (float)K * T * P * (0.9f * J - 17.0f - far_setup_ops(nc, J, pts)) >= kFarMinSaved ? nc : 0;
}

// Row stride of the tile's (step, sample) arrays (poses, clamped controls,
// unit sums): element (t, s) sits at t SP + s.  The rollout scans and the
// per-sample cost loops step through a sample's row with lanes on
// consecutive t, so an even S folds the lanes' float4 and float2 accesses
// onto a few banks (S = 32: all onto one).  The persistent batch kernel
// rounds SP up to an odd number, which spreads them (a 64-controller mix
// at S = 32: 3.31 -> 3.00 ms); the one-controller kernels keep SP = S,
// which measured faster there (their autotuned S avoid the worst strides).
__host__ __device__ inline int row_stride(int S, bool batched) { return batched ? (S | 1) : S; }

__host__ __device__ inline SmemLayout smem_layout(int T, int S, int P, int J, int n, int nscl,
                                                  int nwarps, int nc, bool batched) {
  SmemLayout L;
  int off = 0;
  L.obs4 = off;
  off += 16 * (J > 0 ? J : 1);
  off = align_up(off, 16);
  L.cell = off;
  off += nc * (int)sizeof(FarCell);
  L.list = off;
  off += align_up(2 * nc * far_list_cap(J), 16);
  L.region = off;
  const int SP = row_stride(S, batched);
  int main_b = 16 * T * SP + 8 * T * SP;
  int raw_b = align_up(24 * J, 16);
  int nom_b = 16 * T + 4 * T * P;
  int merge_b = merge_buf_bytes(2 * T, 32 * nwarps) + 8 * (nscl > 1 ? nscl : 1);
  int reg = main_b;
  if (raw_b > reg) reg = raw_b;
  if (nom_b > reg) reg = nom_b;
  if (merge_b > reg) reg = merge_b;
  L.pose = off;
  L.V = off + 16 * T * SP;
  off += align_up(reg, 16);
  L.red = off;
  off += 8 * 4 * 32;
  L.Us = off;
  off += 16 * T;
  L.Sk = off;
  off += 8 * 32;
  L.Usf = off;
  off += 8 * T;
  L.Uf = off;
  off += 8 * T;
  L.Af = off;
  off += 8 * T;
  L.colhi = off;
  off += 8 * T;
  L.collo = off;
  off += 8 * T;
  L.scl = off;
  off += 4 * (nscl > 32 ? nscl : 32);
  L.xrf = off;
  off += 4 * (T + 1) * n;
  off = align_up(off, 8);
  L.shp = off;
  off += 8 * kMaxShape;
  L.eS = off;
  off += 4 * 32;
  L.cw = off;
  off += 4 * T;
  L.scH = off;
  off += 4 * 32;
  L.scL = off;
  off += 4 * 32;
  L.xi = off;
  off += 4 * kMaxN;
  L.collf = off;
  off += 32;
  L.total = align_up(off, 16);
  return L;
}

// ------------------------------------------------------------------ Philox
// Philox4x32-10 from the published description (Salmon et al., SC'11):
// ten rounds of two 32x32->64 multiplies with the key bumped by the Weyl
// constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t a0 = 0xD2511F53u, a1 = 0xCD9E8D57u;
    uint32_t hi0 = __umulhi(a0, c.x), lo0 = a0 * c.x;
    uint32_t hi1 = __umulhi(a1, c.z), lo1 = a1 * c.z;
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

// The top 23 bits k of r as an odd multiple (2 k + 1) of 2^-24, times `scale`
// (1 or 2): exactly representable, so 1 + k 2^-23, whose bits are put
// together, less 1 - 2^-24 is exact (no integer conversion, which runs at a
// quarter of the rate).
template <int SCALE>
__device__ __forceinline__ float unit_open(uint32_t r) {
  static_assert(SCALE == 1 || SCALE == 2, "one exponent up at most");
  const uint32_t one = SCALE == 1 ? 0x3f800000u : 0x40000000u;
  return __fadd_rn(__uint_as_float(one | (r >> 9)), -SCALE * (1.0f - 5.9604644775390625e-8f));
}

// Square root by the approximate instruction (relative error about one ulp).
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// One NLN perturbation (Eq. 11): (chol(S_e Sigma) z_n) .* exp(mu + sigma z_ln).
// Box-Muller radii sqrt(-2 ln u) with u >= 2^-24 and 1 - u >= 2^-24, so the
// argument of the square root is at least 1.1e-7; the log-normal factor's
// exponent is bounded by |mu| + 5.8 sigma, where the intrinsic exponential is
// within a few ulp.
__device__ __forceinline__ float2 nln_draw(uint4 r, float L00, float L10, float L11,
                                           float ln_mu, float ln_sigma) {
  float ra = sqrt_approx(-2.0f * logf(unit_open<1>(r.x)));
  float sa, ca;
  sincospif(unit_open<2>(r.y), &sa, &ca);
  float rb = sqrt_approx(-2.0f * logf(unit_open<1>(r.z)));
  float sb, cb;
  sincospif(unit_open<2>(r.w), &sb, &cb);
  float zn0 = ra * ca, zn1 = ra * sa;
  float g0 = __expf(ln_mu + ln_sigma * (rb * cb));
  float g1 = __expf(ln_mu + ln_sigma * (rb * sb));
  return make_float2(L00 * zn0 * g0, (L10 * zn0 + L11 * zn1) * g1);
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// min(a, b, c) in one instruction (three-input PTX min, sm_100 and later);
// exact, as min(min(a, b), c).
__device__ __forceinline__ float fmin3(float a, float b, float c) {
  float y;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}

// Unevaluated float pair accumulated with Knuth's TwoSum.
struct FF {
  float hi, lo;
};
__device__ __forceinline__ void ff_add(FF& a, float x) {
  float s = __fadd_rn(a.hi, x);
  float bp = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
  a.hi = s;
  a.lo = __fadd_rn(a.lo, e);
}

// TwoProd: c * (bh + bl) = ph + pe (+ c bl) added to the float pair.
__device__ __forceinline__ void ff_add_prod(FF& a, float c, float bh, float bl) {
  float ph = c * bh;
  float pe = fmaf(c, bh, -ph);
  ff_add(a, ph);
  a.lo += fmaf(c, bl, pe);
}

// Renormalise a float pair so that |lo| <= ulp(hi) / 2 (Fast2Sum).
__device__ __forceinline__ FF ff_norm(FF a) {
  const float s = __fadd_rn(a.hi, a.lo);
  return FF{s, __fsub_rn(a.lo, __fsub_rn(s, a.hi))};
}
// Lexicographic order of normalised float pairs = order of their values.
__device__ __forceinline__ bool ff_less(FF a, FF b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}
// (a - b) rounded to float, for normalised pairs a >= b.
__device__ __forceinline__ float ff_diff(FF a, FF b) {
  return __fadd_rn(__fsub_rn(a.hi, b.hi), __fsub_rn(a.lo, b.lo));
}
__device__ __forceinline__ FF warp_min_ff(FF a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    FF b;
    b.hi = __shfl_xor_sync(0xffffffffu, a.hi, o);
    b.lo = __shfl_xor_sync(0xffffffffu, a.lo, o);
    if (ff_less(b, a)) a = b;
  }
  return a;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_min_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------------------ mbarrier / TMA
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Bulk (non-tensor) TMA copy global -> shared, completion on the mbarrier.
// dst, src 16-byte aligned; bytes a multiple of 16.
__device__ __forceinline__ void tma_bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                             uint64_t* bar) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// One arrival on an mbarrier (no transaction bytes).
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait on an mbarrier phase: at most max_polls tries and max_cycles
// SM clock cycles (a try may suspend the thread for a while); false if a
// bound ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int max_polls,
                                          long long max_cycles) {
  uint32_t a = smem_u32(bar);
  const long long t0 = clock64();
  for (int i = 0; i < max_polls; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > max_cycles) break;
  }
  return false;
}

// ------------------------------------------------------------------ dynamics
// State dimension of each model (the Euler steps themselves are evaluated in
// scan form, see scan_trajectory).
// Models: 0 unicycle, 1 planar quadrotor (6 states, two thrusts), 2 Ackermann
// vehicle (Eq. 14), 3 the paper's planar quadrotor (5 states, Eq. 12).
template <int MODEL>
struct Dyn {
  static constexpr int n = MODEL == 0 ? 3 : MODEL == 1 ? 6 : MODEL == 2 ? 4 : 5;
};

// ------------------------------------------------------------ tile kernel body
// Samples with a weight of at least 1 / kRefShare are summed directly once
// more (refine_samples); at most kRefShare samples can have one (their weights
// add up to 1 at most; the last roundings of 128 weights of 1 / 128 each can
// not make room for another).  Their numbers and the changes of their costs
// lie in the reduction scratch.
constexpr int kRefShare = 128;
constexpr int kRefMax = kRefShare;
static_assert(8 * kRefMax <= 8 * 4 * 32, "the list lies in the reduction scratch");
struct TileScratch {
  uint64_t mbar;
  int flag;
  double beta0, beta_d, Kconst, base;  // base = C0 + Kconst
  FF rho, Z;                           // merge results
  float ref;                           // common reference of a merge (minimum of the sources' rho)
  double S_e_used, S_e_next;           // exploration rate of this step and the next
  unsigned long long iter;             // iteration counter of this step
  double x0[2];                        // measured position: origin of the tile's frame
  int n_ref, n_tile;                   // samples whose costs the last CTA takes again (refine_list)
};

// The grid map as a tile reads it.  The tile's frame is centred on the
// measured position x0, whose grid coordinates are split (in FP64) into the
// integer cell (ci, cj) and the remainder (ru, rv) in [0, 1): a point X of
// the tile's frame has grid coordinate ci + (ru + X / res), and the FP32
// part stays small, so its rounding is that of a few cells, not of the
// whole map.
struct GridView {
  const float* g;
  int nx, ny, ci, cj;
  float ru, rv, inv_res;
};

// One axis of the lookup: cell index in [0, n - 2] and weight in [0, 1] of
// grid coordinate c + l, with the coordinate clamped to [0, n - 1] first.
// The first clamp bounds l to just beyond the map (fminf / fmaxf return the
// number when the other operand is NaN), so the index is finite for any
// input.
__device__ __forceinline__ int grid_axis(int c, float l, int n, float& f) {
  l = fminf(fmaxf(l, (float)(-1 - c)), (float)(n - c));
  const float fl = floorf(l);
  int i = c + (int)fl;
  f = l - fl;
  if (i < 0) {
    i = 0;
    f = 0.0f;
  } else if (i >= n - 1) {
    i = n - 2;
    f = 1.0f;
  }
  return i;
}

// The grid map's h at a point of the tile's frame (Sec. V-C grid map):
// bilinear interpolation of the four samples around it, the grid
// coordinates first clamped to [0, nx - 1] x [0, ny - 1]; nx, ny >= 2.
__device__ __forceinline__ float grid_h(const GridView& gv, float X, float Y) {
  float fx, fy;
  const int i = grid_axis(gv.ci, fmaf(X, gv.inv_res, gv.ru), gv.nx, fx);
  const int j = grid_axis(gv.cj, fmaf(Y, gv.inv_res, gv.rv), gv.ny, fy);
  const float* r0 = gv.g + (size_t)j * gv.nx + i;
  const float* r1 = r0 + gv.nx;
  const float g00 = __ldg(r0), g10 = __ldg(r0 + 1), g01 = __ldg(r1), g11 = __ldg(r1 + 1);
  const float a = fmaf(fx, g10 - g00, g00), b = fmaf(fx, g11 - g01, g01);
  return fmaf(fy, b - a, a);
}

// Minimum and maximum of a float over the warp, in one instruction each.
__device__ __forceinline__ float warp_min_f(float v) {
  float y;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(v));
  return y;
}
__device__ __forceinline__ float warp_max_f(float v) {
  float y;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(v));
  return y;
}

// Place of unit u = t S + s in the tile's (step, sample) arrays: t SP + s =
// u + (SP - S) floor(u / S), SP = row_stride(S, BATCHED); the quotient by one
// multiply-high with m = ceil(2^32 / S), exact while u (m S - 2^32) < 2^32
// (here u < T S <= 2^13 and m S - 2^32 < S <= 32).
template <bool BATCHED>
struct UnitIndex {
  unsigned pad, mS;
  __device__ __forceinline__ explicit UnitIndex(int S) {
    pad = (unsigned)(row_stride(S, BATCHED) - S);
    mS = pad ? 0xffffffffu / (unsigned)S + 1u : 0u;
  }
  __device__ __forceinline__ int operator()(int u) const {
    if constexpr (BATCHED) return (int)((unsigned)u + pad * __umulhi((unsigned)u, mS));
    else return u;
  }
};

// Place of the coefficient of x^i y^k (i + k <= kFarN) in FarCell::c: Horner
// in y from the highest power, inside it Horner in x from the highest power.
__host__ __device__ constexpr int far_pos(int i, int k) {
  return (kFarN - k) * (kFarN + 1 - k) / 2 + (kFarN - k - i);
}

// Set-up of one cell by one warp: the disc around the poses of units
// [u0, u1), the obstacles near it (list, in order) and the Taylor
// coefficients of the others' sum of 1 / h.  With D = p0 - c, H = |D|^2 - r^2
// and d = R (x, y) the offset from p0,
//   1 / h = 1 / (H + 2 D.d + |d|^2) = sum_n Q_n,  Q_0 = 1 / H,
//   Q_{n+1} = -(2 D.d / H) Q_n - (|d|^2 / H) Q_{n-1},
// the three-term recurrence of 1 / (1 - 2 x t + t^2); Q_n is homogeneous of
// degree n, so its n + 1 coefficients follow from the two rows before.  Lanes
// take obstacles; their sums are added across the warp with a transposing
// butterfly (each lane ends with three of the coefficients).  The cell's share
// of near obstacles goes to *near_share, if given (look_samples).
template <bool BATCHED>
__device__ __noinline__ void far_setup(int cell_off, int list_off, int pose_off, int obs_off, int u0,
                                       int u1, int S, int J, float r_body, float h_eps,
                                       unsigned* near_share, int lane) {
  extern __shared__ __align__(16) char smem[];
  FarCell* cell = reinterpret_cast<FarCell*>(smem + cell_off);
  unsigned short* list = reinterpret_cast<unsigned short*>(smem + list_off);
  const float4* pose = reinterpret_cast<const float4*>(smem + pose_off);
  const float4* obs4 = reinterpret_cast<const float4*>(smem + obs_off);
  const int cap = far_list_cap(J);
  const UnitIndex<BATCHED> at(S);
  const float inf = __int_as_float(0x7f800000);
  float x0 = inf, x1 = -inf, y0 = inf, y1 = -inf;
  for (int u = u0 + lane; u < u1; u += 32) {
    const float2 p = *reinterpret_cast<const float2*>(pose + at(u));
    x0 = fminf(x0, p.x);
    x1 = fmaxf(x1, p.x);
    y0 = fminf(y0, p.y);
    y1 = fmaxf(y1, p.y);
  }
  const float cx = 0.5f * (warp_min_f(x0) + warp_max_f(x1));
  const float cy = 0.5f * (warp_min_f(y0) + warp_max_f(y1));
  float m = 0.0f;
  bool fine = true;  // every pose finite (and not so far that squares overflow)
  for (int u = u0 + lane; u < u1; u += 32) {
    const float2 p = *reinterpret_cast<const float2*>(pose + at(u));
    const float dx = p.x - cx, dy = p.y - cy;
    const float d2 = fmaf(dx, dx, dy * dy);
    fine = fine && d2 < 1.0e30f;
    m = fmaxf(m, d2);
  }
  const float R = (sqrt_approx(warp_max_f(m)) + r_body) * 1.00001f;
  fine = __all_sync(0xffffffffu, fine);
  // near obstacles: those whose clearance a is below R / kFarRatio, or whose h
  // could come down to h_eps (h >= (a - R)^2 over the disc)
  auto far = [&](int j, float& dx, float& dy, float& H) {
    const float4 o = obs4[j];
    dx = cx - o.x;
    dy = cy - o.y;
    const float d2 = fmaf(dx, dx, dy * dy);
    H = fmaf(dx, dx, fmaf(dy, dy, o.z));
    const float a = sqrt_approx(d2) - o.w, b = a - R;
    return fine && R <= kFarRatio * a && b * b >= h_eps;
  };
  int nn = 0;
  for (int j0 = 0; j0 < J; j0 += 32) {
    const int j = j0 + lane;
    float dx, dy, H;
    const bool near = j < J && !far(j, dx, dy, H);
    const unsigned b = __ballot_sync(0xffffffffu, near);
    const int at_ = nn + __popc(b & ((1u << lane) - 1u));
    if (near && at_ < cap) list[at_] = (unsigned short)j;
    nn += __popc(b);
  }
  const bool direct = nn > cap || J - nn < kFarMin;
  const float inv_R = R > 1.0e-30f ? 1.0f / R : 0.0f;
  if (lane == 0) {
    cell->cx = cx;
    cell->cy = cy;
    cell->inv_R = inv_R;
    cell->n_near = direct ? -1 : nn;
    if (near_share) atomicAdd(near_share, direct ? 256u : 256u * (unsigned)nn / (unsigned)J);
  }
  if (direct) return;
  float acc[48];
#pragma unroll
  for (int i = 0; i < 48; ++i) acc[i] = 0.0f;
  for (int j = lane; j < J; j += 32) {
    float dx, dy, H;
    // (an obstacle so far away that H overflows, as pads a set of fixed size,
    // adds nothing; its offset times 1 / H = 0 would be no number)
    if (!far(j, dx, dy, H) || H > 3.0e38f) continue;
    const float q = 1.0f / H, g = -2.0f * R * q;
    const float ax = g * dx, ay = g * dy, b = -R * R * q;
    float r0[kFarN + 1], r1[kFarN + 1];  // rows n - 1 and n
    r0[0] = q;
    r1[0] = ax * q;
    r1[1] = ay * q;
    acc[far_pos(0, 0)] += q;
    acc[far_pos(1, 0)] += r1[0];
    acc[far_pos(0, 1)] += r1[1];
#pragma unroll
    for (int n = 1; n < kFarN; ++n) {
      float r2[kFarN + 1];
#pragma unroll
      for (int k = 0; k <= n + 1; ++k) {  // coefficient of x^(n+1-k) y^k
        float v = k <= n ? ax * r1[k] : 0.0f;
        if (k >= 1) v = k <= n ? fmaf(ay, r1[k - 1], v) : ay * r1[k - 1];
        if (k <= n - 1) v = fmaf(b, r0[k], v);
        if (k >= 2) v = fmaf(b, r0[k - 2], v);
        r2[k] = v;
        acc[far_pos(n + 1 - k, k)] += v;
      }
#pragma unroll
      for (int k = 0; k <= n + 1; ++k) {
        if (k <= n) r0[k] = r1[k];
        r1[k] = r2[k];
      }
    }
  }
  __syncwarp();
  int base = 0;
#pragma unroll
  for (int o = 16, n = 24; o >= 2; o >>= 1, n >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float send = up ? acc[i] : acc[i + n];
      const float keep = up ? acc[i + n] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    base += up ? n : 0;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float v = acc[i] + __shfl_xor_sync(0xffffffffu, acc[i], 1);
    if (!(lane & 1) && base + i < kFarCoef) cell->c[base + i] = make_float2(v, v);
  }
}

// The far obstacles' sum of 1 / h at a thread's packed points: the cell's
// polynomial by Horner's rule in two variables, 44 two-lane FMAs per pair of
// points (as much as nine obstacles one by one).
template <int NP2>
__device__ __forceinline__ void far_eval(const FarCell* __restrict__ cell, const float2 (&X2)[NP2],
                                         const float2 (&Y2)[NP2], float2 (&acc2)[NP2]) {
  const float2 ncx = make_float2(-cell->cx, -cell->cx), ncy = make_float2(-cell->cy, -cell->cy);
  const float2 ir = make_float2(cell->inv_R, cell->inv_R);
  float2 x[NP2], y[NP2];
#pragma unroll
  for (int k = 0; k < NP2; ++k) {
    x[k] = __fmul2_rn(__fadd2_rn(X2[k], ncx), ir);
    y[k] = __fmul2_rn(__fadd2_rn(Y2[k], ncy), ir);
    acc2[k] = cell->c[0];
  }
  int at = 1;
#pragma unroll
  for (int ky = kFarN - 1; ky >= 0; --ky) {
    float2 r[NP2];
    const float2 c0 = cell->c[at++];
#pragma unroll
    for (int k = 0; k < NP2; ++k) r[k] = c0;
#pragma unroll
    for (int i = kFarN - ky - 1; i >= 0; --i) {
      const float2 c = cell->c[at++];
#pragma unroll
      for (int k = 0; k < NP2; ++k) r[k] = __ffma2_rn(r[k], x[k], c);
    }
#pragma unroll
    for (int k = 0; k < NP2; ++k) acc2[k] = __ffma2_rn(acc2[k], y[k], r[k]);
  }
}

template <bool B>
struct BoolC {
  static constexpr bool value = B;
};

// Fused barrier over nunits = T S (step, sample) units; unit u = t S + s has
// its pose at pose[t SP + s] (SP = row_stride(S, BATCHED)) and P shape
// points shp[0..P).  A warp takes groups of 32 (NPOS / P) consecutive units
// (NPOS >= P), each lane the units base + 32 k + lane (k < NPOS / P) so that
// neighbouring lanes read neighbouring poses, keeps their world points in
// registers and streams the obstacles of the group's cell, or all of them
// (nc = 0, or a cell without a polynomial): h = |p - c|^2 - r^2 evaluated as
// fma(dx, dx, fma(dy, dy, -r^2)), terms 1 / max(h, h_eps) added two obstacles
// at a time as (h1 + h2) / (h1 h2) with the approximate reciprocal.  The
// points are held in packed pairs and the subtractions, fmas, sums and
// products are packed two-lane FP32 instructions (each lane the same
// round-to-nearest operation as the scalar one): one issue slot for two
// points, where the loop is bound by instruction issue.  A unit's points
// are summed exactly (TwoSum) into (hi, lo), stored at uB[u * ustride]; the
// sign bit of hi marks a unit in which some h <= 0 (collision; a far obstacle
// has h >= h_eps all over its cell).  A lane reads the poses of its units
// before it writes their sums, so uB may overlay pose.  GRID: each point also
// adds the grid map's term (grid_h) and counts its h in the collision test.
template <int NPOS, bool BATCHED, bool FAR, bool GRID = false>
__device__ __forceinline__ void barrier_units(int nunits, int S, int P, int J, const float4* pose,
                                              const float2* __restrict__ shp,
                                              const float4* __restrict__ obs4, float h_eps,
                                              float2* uB, int ustride, int tid, int nthreads, int nc,
                                              const FarCell* __restrict__ cells,
                                              const unsigned short* __restrict__ lists,
                                              const GridView* gv = nullptr) {
  const UnitIndex<BATCHED> at(S);
  static_assert(NPOS % 2 == 0, "points are held in packed pairs");
  constexpr int NP2 = NPOS / 2;
  const int upt = NPOS / P;  // units per lane
  const int used = upt * P;
  const int lane = tid & 31, nwarps = nthreads >> 5;
  const int gsz = 32 * upt, NG = (nunits + gsz - 1) / gsz;
  for (int g = tid >> 5; g < NG; g += nwarps) {
    const int ub = g * gsz + lane;  // this lane's first unit
    float2 X2[NP2], Y2[NP2], acc2[NP2];  // points 2k and 2k + 1
    float mn[NPOS];
    int uu = 0, p = 0;
#pragma unroll
    for (int i = 0; i < NPOS; ++i) {
      const int u = ub + uu * 32;
      const bool ok = (i < used) && (u < nunits);
      const float4 ps = pose[at(ok ? u : nunits - 1)];
      const float2 sh = shp[ok ? p : 0];
      const float X = fmaf(ps.z, sh.x, fmaf(-ps.w, sh.y, ps.x));
      const float Y = fmaf(ps.w, sh.x, fmaf(ps.z, sh.y, ps.y));
      if (i & 1) {
        X2[i >> 1].y = X;
        Y2[i >> 1].y = Y;
      } else {
        X2[i >> 1].x = X;
        Y2[i >> 1].x = Y;
      }
      mn[i] = __int_as_float(0x7f800000);
      if (++p == P) {
        p = 0;
        ++uu;
      }
    }
#pragma unroll
    for (int k = 0; k < NP2; ++k) acc2[k] = make_float2(0.0f, 0.0f);
    auto one = [&](const float4 o) {
      const float2 nox = make_float2(-o.x, -o.x), noy = make_float2(-o.y, -o.y);
      const float2 noz = make_float2(o.z, o.z);
#pragma unroll
      for (int k = 0; k < NP2; ++k) {
        const float2 dx = __fadd2_rn(X2[k], nox), dy = __fadd2_rn(Y2[k], noy);
        const float2 h = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, noz));
        mn[2 * k] = fminf(mn[2 * k], h.x);
        mn[2 * k + 1] = fminf(mn[2 * k + 1], h.y);
        acc2[k] = __fadd2_rn(acc2[k], make_float2(rcp_approx(fmaxf(h.x, h_eps)),
                                                  rcp_approx(fmaxf(h.y, h_eps))));
      }
    };
    // obstacles in pairs: 1/h1 + 1/h2 = (h1 + h2) / (h1 h2), one reciprocal
    // for two terms (h1 h2 stays finite for |p - c| < 4e9 m and h_eps >= 1e-18).
    // At 14 points per lane only the lists of near obstacles do so (a call at
    // K 32768, J 500 829 -> 786 us: one reciprocal per pair of point and obstacle
    // binds the special-function pipe); the loop over all obstacles keeps one
    // each, whose sums barrier_refine forms bit for bit.
    auto two = [&](const float4 o, const float4 q, auto paired) {
      if constexpr (decltype(paired)::value) {
        const float2 nox = make_float2(-o.x, -o.x), noy = make_float2(-o.y, -o.y);
        const float2 noz = make_float2(o.z, o.z);
        const float2 nqx = make_float2(-q.x, -q.x), nqy = make_float2(-q.y, -q.y);
        const float2 nqz = make_float2(q.z, q.z);
#pragma unroll
        for (int k = 0; k < NP2; ++k) {
          const float2 dx = __fadd2_rn(X2[k], nox), dy = __fadd2_rn(Y2[k], noy);
          const float2 ex = __fadd2_rn(X2[k], nqx), ey = __fadd2_rn(Y2[k], nqy);
          float2 h1 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, noz));
          float2 h2 = __ffma2_rn(ex, ex, __ffma2_rn(ey, ey, nqz));
          mn[2 * k] = fmin3(mn[2 * k], h1.x, h2.x);
          mn[2 * k + 1] = fmin3(mn[2 * k + 1], h1.y, h2.y);
          h1 = make_float2(fmaxf(h1.x, h_eps), fmaxf(h1.y, h_eps));
          h2 = make_float2(fmaxf(h2.x, h_eps), fmaxf(h2.y, h_eps));
          const float2 pr = __fmul2_rn(h1, h2);
          const float2 r = make_float2(rcp_approx(pr.x), rcp_approx(pr.y));
          acc2[k] = __ffma2_rn(__fadd2_rn(h1, h2), r, acc2[k]);
        }
      } else {
        one(o);
        one(q);
      }
    };
    bool direct = true;
    if constexpr (FAR) {
      const int c = nc > 0 ? g * nc / NG : 0;
      const int nn = nc > 0 ? cells[c].n_near : -1;
      if (nn >= 0) {
        direct = false;
        far_eval<NP2>(cells + c, X2, Y2, acc2);
        const unsigned short* l = lists + c * far_list_cap(J);
        int j = 0;
        for (; j + 1 < nn; j += 2) {
          const unsigned jj = *reinterpret_cast<const unsigned*>(l + j);
          two(obs4[jj & 0xffffu], obs4[jj >> 16], BoolC<true>());
        }
        if (j < nn) one(obs4[l[j]]);
      }
    }
    if (direct) {
      int j = 0;
      for (; j + 1 < J; j += 2) two(obs4[j], obs4[j + 1], BoolC<(NPOS <= 8)>());
      if (j < J) one(obs4[j]);
    }
    if constexpr (GRID) {
      if (gv->g) {
#pragma unroll
        for (int k = 0; k < NP2; ++k) {
          const float hx = grid_h(*gv, X2[k].x, Y2[k].x), hy = grid_h(*gv, X2[k].y, Y2[k].y);
          mn[2 * k] = fminf(mn[2 * k], hx);
          mn[2 * k + 1] = fminf(mn[2 * k + 1], hy);
          acc2[k] = __fadd2_rn(acc2[k], make_float2(rcp_approx(fmaxf(hx, h_eps)),
                                                    rcp_approx(fmaxf(hy, h_eps))));
        }
      }
    }
    FF f = {0.0f, 0.0f};
    bool coll = false;
    uu = 0;
    p = 0;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NPOS; ++i) {
      if (i < used) {
        ff_add(f, (i & 1) ? acc2[i >> 1].y : acc2[i >> 1].x);
        coll |= (mn[i] <= 0.0f);
        if (++p == P) {
          const int u = ub + uu * 32;
          if (u < nunits) uB[(size_t)at(u) * ustride] = make_float2(coll ? -f.hi : f.hi, f.lo);
          f.hi = 0.0f;
          f.lo = 0.0f;
          coll = false;
          p = 0;
          ++uu;
        }
      }
    }
  }
}

// The barrier of a few samples (Sc of them, their poses at pose[t SP + s]),
// every obstacle directly, with the points spread over the lanes: the points
// of a unit on 1, 2, 4 or 8 neighbouring lanes, two units per lane as a packed
// pair.  Each point's sum and each unit's sum are formed by the operations of
// barrier_units without cells, in the same order, so they are the same bits.
// For the last CTA of a step, which runs it alone: the time is that of one
// lane's loop over the obstacles.
template <int NPOS, bool GRID>
__device__ __forceinline__ void barrier_refine(int Sc, int T, int SP, int P, int J,
                                               const float4* pose, const float2* __restrict__ shp,
                                               const float4* __restrict__ obs4, float h_eps,
                                               float2* uB, int ustride, int tid, int nthreads,
                                               const GridView* gv) {
  const int lp = P <= 1 ? 1 : P <= 2 ? 2 : P <= 4 ? 4 : 8;  // lanes per unit
  const int lane = tid & 31, upw = 32 / lp, p = lane & (lp - 1), first = lane - p;
  const int nunits = Sc * T;
  const float2 sh = shp[min(p, P - 1)];
  for (int u0 = (tid >> 5) * 2 * upw; u0 < nunits; u0 += (nthreads >> 5) * 2 * upw) {
    int at[2];
    float2 X, Y, acc = make_float2(0.0f, 0.0f);
    float mn[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int u = min(u0 + q * upw + lane / lp, nunits - 1);
      const int t = u / Sc;
      at[q] = t * SP + (u - t * Sc);
      const float4 ps = pose[at[q]];
      (q ? X.y : X.x) = fmaf(ps.z, sh.x, fmaf(-ps.w, sh.y, ps.x));
      (q ? Y.y : Y.x) = fmaf(ps.w, sh.x, fmaf(ps.z, sh.y, ps.y));
      mn[q] = __int_as_float(0x7f800000);
    }
    auto h_of = [&](const float4 o) {
      const float2 dx = __fadd2_rn(X, make_float2(-o.x, -o.x)), dy = __fadd2_rn(Y, make_float2(-o.y, -o.y));
      return __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, make_float2(o.z, o.z)));
    };
    int j = 0;
    if constexpr (NPOS <= 8) {
#pragma unroll 2
      for (; j + 1 < J; j += 2) {
        float2 h1 = h_of(obs4[j]), h2 = h_of(obs4[j + 1]);
        mn[0] = fmin3(mn[0], h1.x, h2.x);
        mn[1] = fmin3(mn[1], h1.y, h2.y);
        h1 = make_float2(fmaxf(h1.x, h_eps), fmaxf(h1.y, h_eps));
        h2 = make_float2(fmaxf(h2.x, h_eps), fmaxf(h2.y, h_eps));
        const float2 pr = __fmul2_rn(h1, h2);
        acc = __ffma2_rn(__fadd2_rn(h1, h2), make_float2(rcp_approx(pr.x), rcp_approx(pr.y)), acc);
      }
    }
#pragma unroll 4
    for (; j < J; ++j) {
      const float2 h = h_of(obs4[j]);
      mn[0] = fminf(mn[0], h.x);
      mn[1] = fminf(mn[1], h.y);
      acc = __fadd2_rn(acc, make_float2(rcp_approx(fmaxf(h.x, h_eps)), rcp_approx(fmaxf(h.y, h_eps))));
    }
    if constexpr (GRID) {
      if (gv->g) {
        const float hx = grid_h(*gv, X.x, Y.x), hy = grid_h(*gv, X.y, Y.y);
        mn[0] = fminf(mn[0], hx);
        mn[1] = fminf(mn[1], hy);
        acc = __fadd2_rn(acc, make_float2(rcp_approx(fmaxf(hx, h_eps)), rcp_approx(fmaxf(hy, h_eps))));
      }
    }
    __syncwarp();
    FF f[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
    for (int i = 0; i < P; ++i) {
      ff_add(f[0], __shfl_sync(0xffffffffu, acc.x, first + i));
      ff_add(f[1], __shfl_sync(0xffffffffu, acc.y, first + i));
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const unsigned hit = __ballot_sync(0xffffffffu, mn[q] <= 0.0f);
      const bool coll = (hit >> first) & ((1u << lp) - 1u);
      if (p == 0 && u0 + q * upw + lane / lp < nunits)
        uB[(size_t)at[q] * ustride] = make_float2(coll ? -f[q].hi : f[q].hi, f[q].lo);
    }
  }
}

// Two float pairs added exactly up to the final rounding of the low part.
__device__ __forceinline__ FF ff_sum(FF a, FF b) {
  FF r = a;
  ff_add(r, b.hi);
  r.lo += b.lo;
  return r;
}

// Sum of a float pair over the 32 lanes (fixed butterfly order).
__device__ __forceinline__ FF warp_sum_ff(FF a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    FF b;
    b.hi = __shfl_xor_sync(0xffffffffu, a.hi, o);
    b.lo = __shfl_xor_sync(0xffffffffu, a.lo, o);
    a = ff_sum(a, b);
  }
  return a;
}

// Sums of four float pairs over the 32 lanes at once: the first two rounds of
// the butterfly each hand half of the pairs to the partner, so six pair sums
// take the place of twenty.  Lane 8 q returns the sum of v[sum4_of_lane(8 q)],
// formed in the order in which warp_sum_ff forms lane 0's (the lower lane's low
// part first): the same bits.
__device__ __forceinline__ FF ff_exchange_sum(FF a, FF b, int o, int lane) {
  const bool up = lane & o;
  const FF keep = up ? b : a, send = up ? a : b;
  FF got;
  got.hi = __shfl_xor_sync(0xffffffffu, send.hi, o);
  got.lo = __shfl_xor_sync(0xffffffffu, send.lo, o);
  return up ? ff_sum(got, keep) : ff_sum(keep, got);
}
__device__ __forceinline__ FF warp_sum_ff4(const FF (&v)[4], int lane) {
  FF a = ff_exchange_sum(ff_exchange_sum(v[0], v[1], 16, lane),
                         ff_exchange_sum(v[2], v[3], 16, lane), 8, lane);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    FF b;
    b.hi = __shfl_xor_sync(0xffffffffu, a.hi, o);
    b.lo = __shfl_xor_sync(0xffffffffu, a.lo, o);
    a = ff_sum(a, b);
  }
  return a;
}
__device__ __forceinline__ int sum4_of_lane(int lane) {
  return ((lane >> 4) & 1) | ((lane >> 2) & 2);
}

// Minimum of floats by an integer atomic: key(f) = ~u(f), u the
// order-preserving unsigned image of f, so that a larger key is a smaller f
// and 0 (the cleared word) is below every key of a number.  atomicMax over
// keys is an exact, order-independent minimum.
__device__ __forceinline__ unsigned min_key(float f) {
  const int i = __float_as_int(f);
  return ~((unsigned)(i >= 0 ? i : i ^ 0x7fffffff) ^ 0x80000000u);
}
__device__ __forceinline__ float key_min(unsigned k) {
  const int i = (int)(~k ^ 0x80000000u);
  return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff);
}

// Merge n partial results (rho_i, Z_i, cols_i[ncol]), each taken relative to
// its own minimum rho_i, into one relative to ref = min_i rho_i.hi: the
// log-sum-exp merge of Eq. 4's numerator and denominator.  ref is read from
// *minw, the key (min_key) into which every source put its rho_i.hi with an
// atomic maximum before its ticket; thread 0 clears the word for the next
// step once every thread has read it, and stores ref at *ref_out.  Source i
// is scaled by s_i = exp(-(rho_i - ref) / lambda) <= 1.  Every load of the
// merge (the word, a thread's first source row, its column pairs) is issued
// before the first of them is used: one memory round trip, which is most of
// what a merge costs when one CTA runs it alone at the end of a step.  The
// ncol columns are read as ncp = ncol / 2 float pairs: thread tid takes the
// cell (row group rg, column pair cp) = (tid / ncp, tid % ncp), i.e. rows
// rg, rg + RG, ... of that pair, up to kMergeLoads rows in flight; the
// threads with cp = 0 also add s_i Z_i.  The row groups are then added in
// order.  All threads of the CTA call it.
// PIPELINED: the rows in flight are two batches of kMergeLoads / 2, the next
// loading while one is added; otherwise one batch of kMergeLoads, added
// before the next is loaded.  Both add the rows in the same order (the same
// bits).  The two-batch form is faster in the one-controller step kernels
// (a 256-sample step: 24.2 against 26.4 us); the one-batch form in the
// persistent batch kernel (64 mixed controllers: 3.31 against 4.04 ms).
// Shared memory: scl (n floats), zi (n float2), buf (merge_buf_bytes).
// Outputs in shared memory: *Z_out, col_hi/col_lo[ncol].
template <bool PIPELINED>
__device__ inline void merge_partials(int n, const float4* rz, const float* cols, int ncol,
                                      unsigned* minw, float inv_lambda, float* scl, float2* zi,
                                      FF* buf, float* ref_out, FF* Z_out, float* col_hi,
                                      float* col_lo, int tid, int nthreads) {
  const int ncp = ncol >> 1;
  const int RG = merge_row_groups(ncol, nthreads);
  const int ncell = RG * ncp;
  const int ldb = ncol + 1;  // buf row: the columns, then Z
  const float2* cols2 = reinterpret_cast<const float2*>(cols);
  constexpr int KB = PIPELINED ? kMergeLoads / 2 : kMergeLoads;
  float2 va[KB], vb[KB];  // vb: the second batch (PIPELINED only)
  auto load = [&](float2 (&v)[KB], int cell, int r0) {
    const int rg = cell / ncp, cp = cell - rg * ncp;
#pragma unroll
    for (int q = 0; q < KB; ++q) {
      const int i = rg + (r0 + q) * RG;
      v[q] = (cell < ncell && i < n) ? __ldcg(cols2 + (size_t)i * ncp + cp) : make_float2(0.0f, 0.0f);
    }
  };
  auto add = [&](const float2 (&v)[KB], int rg, int cp, int r0, FF& a0, FF& a1, FF& z) {
#pragma unroll
    for (int q = 0; q < KB; ++q) {
      const int i = rg + (r0 + q) * RG;
      if (i < n) {
        const float sc = scl[i];
        ff_add(a0, v[q].x * sc);
        ff_add(a1, v[q].y * sc);
        if (cp == 0) {
          const float2 zz = zi[i];
          ff_add_prod(z, sc, zz.x, zz.y);
        }
      }
    }
  };
  const unsigned kmin = __ldcg(minw);
  const float4 c0 = tid < n ? __ldcg(rz + tid) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  load(va, tid, 0);
  if constexpr (PIPELINED) load(vb, tid, KB);
  const float ref = key_min(kmin);
  if (tid < n) {
    scl[tid] = expf(-((c0.x - ref) + c0.y) * inv_lambda);
    zi[tid] = make_float2(c0.z, c0.w);
  }
  for (int i = tid + nthreads; i < n; i += nthreads) {  // more sources than threads
    const float4 c = __ldcg(rz + i);
    scl[i] = expf(-((c.x - ref) + c.y) * inv_lambda);
    zi[i] = make_float2(c.z, c.w);
  }
  __syncthreads();
  if (tid == 0) {
    *ref_out = ref;
    *minw = 0u;
  }
  for (int cell = tid; cell < ncell; cell += nthreads) {
    const int rg = cell / ncp, cp = cell - rg * ncp;
    FF a0 = {0.0f, 0.0f}, a1 = {0.0f, 0.0f}, z = {0.0f, 0.0f};
    if constexpr (PIPELINED) {
      for (int r0 = 0;; r0 += 2 * KB) {
        add(va, rg, cp, r0, a0, a1, z);
        if (rg + (r0 + KB) * RG >= n) break;
        if (rg + (r0 + 2 * KB) * RG < n) load(va, cell, r0 + 2 * KB);
        add(vb, rg, cp, r0 + KB, a0, a1, z);
        if (rg + (r0 + 2 * KB) * RG >= n) break;
        if (rg + (r0 + 3 * KB) * RG < n) load(vb, cell, r0 + 3 * KB);
      }
    } else {
      for (int r0 = 0;; r0 += KB) {
        add(va, rg, cp, r0, a0, a1, z);
        if (rg + (r0 + KB) * RG >= n) break;
        load(va, cell, r0 + KB);
      }
    }
    buf[rg * ldb + 2 * cp] = a0;
    buf[rg * ldb + 2 * cp + 1] = a1;
    if (cp == 0) buf[rg * ldb + ncol] = z;
    if (cell + nthreads < ncell) {
      load(va, cell + nthreads, 0);
      if constexpr (PIPELINED) load(vb, cell + nthreads, KB);
    }
  }
  __syncthreads();
  for (int c = tid; c <= ncol; c += nthreads) {
    FF a = buf[c];
    for (int g = 1; g < RG; ++g) a = ff_sum(a, buf[g * ldb + c]);
    if (c < ncol) {
      col_hi[c] = a.hi;
      col_lo[c] = a.lo;
    } else {
      *Z_out = ff_norm(a);
    }
  }
  __syncthreads();
}

// Fused barrier over npos positions, one position per thread at a time
// (position i = unit i / P, shape point i % P): the fully parallel form used
// for the single nominal trajectory.  out[i] = +-sum_j 1/max(h, h_eps), the
// sign bit marking some h <= 0.  GRID: plus the grid map's term.
template <bool GRID = false>
__device__ __forceinline__ void barrier_flat(int npos, int P, int J, const float4* __restrict__ pose,
                                             const float2* __restrict__ shp,
                                             const float4* __restrict__ obs4, float h_eps,
                                             float* __restrict__ out, int tid, int nthreads,
                                             const GridView* gv = nullptr) {
  for (int i = tid; i < npos; i += nthreads) {
    const int u = i / P, p = i - u * P;
    const float4 ps = pose[u];
    const float2 sh = shp[p];
    const float X = fmaf(ps.z, sh.x, fmaf(-ps.w, sh.y, ps.x));
    const float Y = fmaf(ps.w, sh.x, fmaf(ps.z, sh.y, ps.y));
    float acc = 0.0f, mn = __int_as_float(0x7f800000);
    for (int j = 0; j < J; ++j) {
      const float4 o = obs4[j];
      float dx = X - o.x, dy = Y - o.y;
      float h = fmaf(dx, dx, fmaf(dy, dy, o.z));
      mn = fminf(mn, h);
      acc += rcp_approx(fmaxf(h, h_eps));
    }
    if constexpr (GRID) {
      if (gv->g) {
        const float h = grid_h(*gv, X, Y);
        mn = fminf(mn, h);
        acc += rcp_approx(fmaxf(h, h_eps));
      }
    }
    out[i] = mn <= 0.0f ? -acc : acc;
  }
}

// Warp inclusive prefix sum over the 32 lanes.
__device__ __forceinline__ float warp_incl_scan(float v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    float y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}
// The value of lane - 1; lane 0 receives `first`.
__device__ __forceinline__ float from_prev_lane(float v, float first, int lane) {
  float y = __shfl_up_sync(0xffffffffu, v, 1);
  return lane == 0 ? first : y;
}
__device__ __forceinline__ float lane31(float v) { return __shfl_sync(0xffffffffu, v, 31); }

}  // namespace dbm
