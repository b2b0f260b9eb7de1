// Instantiation of the persistent blocked NDFT kernel that writes spectra to
// global memory (ddhf_power_spectrum with DDHF_FORM_BLOCKED).
#include "ndft_blocked.cuh"

namespace ddhf {
namespace {

__global__ void k_list_pixels(const SlotView *view, int list_min, int big_min, uint64_t *list,
                              int64_t cap, uint32_t *count, uint32_t *flags) {
  const SlotView &v = *view;
  const int64_t n_act = (int64_t)v.counters[2];
  for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < n_act;
       a += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t key = v.active[a], cnt = v.offsets[key + 1] - v.offsets[key];
    if (cnt < (uint32_t)list_min) continue;
    const bool big = cnt >= (uint32_t)big_min;
    const uint32_t pos = atomicAdd(&count[big ? 1 : 0], 1u);
    if ((int64_t)pos < cap)
      list[big ? cap - 1 - pos : pos] = (uint32_t)a;  // slot 0
    else
      atomicOr(flags, DDHF_FLAG_CAPACITY);
  }
}

// The work list of slot 0's pixels under the tuning of this call, and the kernel's
// cursors zeroed. The list that the last binning or detection left may be of another
// tuning (ddhf_set_tuning came since), of the last window of a batch, or of all its
// windows: it is filled again unless the host knows that it is the right one. A
// captured call always fills it (what precedes its replays is not known here). A
// listed pixel has at least 32 events, so the list's capacity (a 32nd of the events)
// holds both ends. Filling costs 5 us on 307,200 pixels, 11 in calls so small that
// their launches bound them.
ddhf_status list_slot0(Ctx *c, cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  DDHF_CUDA_TRY(c, cudaStreamIsCapturing(s, &cs));
  if (cs == cudaStreamCaptureStatusNone && !c->list_in_graph &&
      c->listed_min == list_min(c->tuning) && c->listed_big == big_min(c->tuning)) {
    DDHF_CUDA_TRY(c, cudaMemsetAsync(c->qctl + 5, 0, 3 * sizeof(uint32_t), s));
    return DDHF_OK;
  }
  c->listed_min = c->listed_big = 0;
  // with word 4, which every soft comb zeroes itself
  DDHF_CUDA_TRY(c, cudaMemsetAsync(c->qctl, 0, 8 * sizeof(uint32_t), s));
  const int blocks = (int)std::min<int64_t>(ceil_div(c->npx, 256), (int64_t)c->num_sms * 8);
  k_list_pixels<<<blocks, 256, 0, s>>>(c->d_views, list_min(c->tuning), big_min(c->tuning),
                                       c->work, c->heavy_cap, c->qctl, c->flags);
  DDHF_CUDA_TRY(c, cudaGetLastError());
  DDHF_CUDA_TRY(c, note_list(c, true, s));
  return DDHF_OK;
}

}  // namespace

ddhf_status launch_blocked_spectrum(Ctx *c, float *P, int64_t cap_px, cudaStream_t s) {
  const ddhf_status st = list_slot0(c, s);
  if (st != DDHF_OK) return st;
  return blocked::launch_blocked_any<false>(c, 1, P, cap_px, s);
}

// Pixels of slot `slot` with at least the plan's threshold of events through
// the hybrid grid path, the others through the blocked kernel; without a plan
// (hybrid_min 0, or a window whose grid does not fit) all through the latter.
ddhf_status spectrum_with_hybrid(Ctx *c, int slot, int hybrid_min, float *P, int64_t cap_px,
                                 cudaStream_t s, int64_t ld) {
  int skip = 0;
  if (hybrid_min > 0 && c->hyb_c) {
    const HybridPlan hp = hybrid_plan(c, c->slots[slot].window_us, hybrid_min);
    if (hp.ok) {
      const ddhf_status st = launch_hybrid(c, slot, hp, P, cap_px, ld, s);
      if (st != DDHF_OK) return st;
      skip = (int)hp.thr;
    }
  }
  return blocked::launch_blocked_any<false>(c, 1, P, cap_px, s, slot, ld, skip);
}

// Spectra of one window slot (its heavy items must be the only ones queued),
// with the tuning's hybrid threshold.
ddhf_status launch_spectrum_slot(Ctx *c, int slot, float *P, int64_t cap_px, cudaStream_t s,
                                 int64_t ld) {
  DDHF_CUDA_TRY(c, cudaMemsetAsync(c->qctl + 5, 0, 3 * sizeof(uint32_t), s));
  return spectrum_with_hybrid(c, slot, c->tuning.hybrid_min, P, cap_px, s, ld);
}

// ddhf_power_spectrum with DDHF_FORM_HYBRID: slot 0, rows of n_bins floats.
ddhf_status launch_hybrid_spectrum(Ctx *c, float *P, int64_t cap_px, cudaStream_t s) {
  ddhf_status st = hybrid_alloc(c);
  if (st == DDHF_OK) st = list_slot0(c, s);
  if (st != DDHF_OK) return st;
  const int hm = c->tuning.hybrid_min > 0 ? c->tuning.hybrid_min : kHybDefaultMin;
  return spectrum_with_hybrid(c, 0, hm, P, cap_px, s, c->grid.n_bins);
}
}  // namespace ddhf
