// Batched step kernel: persistent CTAs pull (controller, tile) work items
// from an atomic counter; each item's descriptor is copied to shared memory
// and the item runs the same tile body as the one-controller kernels.
#include "kernels.cuh"

namespace dbm {

// (two CTAs per SM: without the bound the allocation rises to 255 registers)
__global__ void __launch_bounds__(kBatchThreads, 2) batch_kernel(const CtrlDesc* __restrict__ descs,
                                                              unsigned char* stage,
                                                              double* __restrict__ u0_out) {
  TileScratch& ts = tile_scratch();
  CtrlDesc& Ds = tile_desc();
  __shared__ int s_item;
  BatchHdr* hdr = reinterpret_cast<BatchHdr*>(stage);
  const StepEntry* steps = reinterpret_cast<const StepEntry*>(stage + sizeof(BatchHdr));
  const WorkItem* items = reinterpret_cast<const WorkItem*>(steps + hdr->n_steps);
  const double* inputs = reinterpret_cast<const double*>(stage + hdr->inputs_off);
  const int tid = threadIdx.x;
  if (tid == 0) mbar_init(&ts.mbar);
  __syncthreads();
  uint32_t phase = 0u;
  const int n_items = hdr->n_items, chunk = hdr->chunk;
  for (;;) {
    if (tid == 0) s_item = (int)atomicAdd(&hdr->next, 1u);
    __syncthreads();
    const int it = s_item;
    if (it >= n_items) break;
    const WorkItem w = items[it];
    const StepEntry e = steps[w.ctrl];
    const int* src = reinterpret_cast<const int*>(descs + e.slot);
    int* dst = reinterpret_cast<int*>(&Ds);
    for (int i = tid; i < (int)(sizeof(CtrlDesc) / 4); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    const double* x0 = inputs + e.x0_off;
    const double* xref = inputs + e.xref_off;
    double* uo = u0_out + 8 * w.ctrl;  // u0 and the predicted next state
    // the batched form of the tile: see run_tile
    switch (Ds.model * 2 + npos_code(Ds.NPOS)) {
      case 0: run_tile<0, 8>(w.tile, chunk, x0, xref, phase, uo); break;
      case 1: run_tile<0, 14>(w.tile, chunk, x0, xref, phase, uo); break;
      case 2: run_tile<1, 8>(w.tile, chunk, x0, xref, phase, uo); break;
      default: run_tile<1, 14>(w.tile, chunk, x0, xref, phase, uo); break;
    }
    __syncthreads();  // Ds and s_item are reused by the next item
  }
}

// Resident serving kernel over the same tile instantiations (see
// serve_body in kernels.cuh).
__global__ void __launch_bounds__(kBatchThreads, 2) serve_kernel(const CtrlDesc* __restrict__ descs,
                                                              ServeRing R) {
  serve_body<false>(descs, R);
}

}  // namespace dbm
