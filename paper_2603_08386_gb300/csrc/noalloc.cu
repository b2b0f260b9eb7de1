// ddhf_power_spectrum_noalloc: the BLOCKED NDFT power spectra computed from a
// per-pixel event list that the caller built and owns, with no device memory
// allocated by the library.
//
// Who needs it: callers that must not allocate device memory once they are
// running, e.g. a detector on a drone or another embedded real-time system
// that reserves all memory at start-up (cudaMalloc can synchronise the device
// and take milliseconds, which breaks a 33 ms frame budget), or a host program
// whose own memory manager owns the whole device. ddhf_create() allocates a
// workspace, so those callers cannot use the context-based entry points.
//
// The kernel's scratch (work-queue counters, the list of heavy pixels, the
// per-window view the persistent kernel reads, the flags) lives in one
// file-scope __device__ array of fixed size, present on every device that
// loads the library until the process exits. Host code only knows a stand-in
// for that symbol, so its device address is fetched with
// cudaGetSymbolAddress() once per CUDA context (keyed by the context's
// process-unique id), during the first call made with that context current.
// That first call also loads every kernel this entry point can launch (all
// four tile-count instantiations of the spectrum kernels and the helpers),
// so that under lazy module loading no later call, whatever its grid, loads
// code or allocates; it should therefore come before any stream capture and
// outside any frame budget. Every call shares the array: the counters and
// flags are cleared at the start of each call, and two calls whose work
// overlaps on the GPU (different streams, or different host threads) race on
// it and must be serialised by the caller.
#include <cuda.h>

#include <mutex>

#include "ndft_blocked.cuh"

namespace ddhf {
namespace {

constexpr int64_t kNoAllocMaxEvents = (int64_t)1 << 25;  // per call
constexpr int kNoAllocHeavyMin = 1024;                   // same default as a context
constexpr int64_t kNoAllocMaxHeavy = kNoAllocMaxEvents / kNoAllocHeavyMin;  // 32768
constexpr int kNoAllocWarps = 4;
constexpr int kMaxContexts = 64;

struct NoAllocScratch {
  SlotView view;
  uint64_t counters[8];  // [2] = number of active pixels
  uint32_t qctl[8];      // [0] heavy count, [1] big count, [2-4] cursors (heavy, light, big),
                         // [5] places of the list asked for, [6] pixels for k_team_scan
  uint32_t flags;
  uint32_t pad[3];
  uint64_t heavy[kNoAllocMaxHeavy];  // heavy work items (slot 0 << 32 | active index)
};

// 256-byte aligned; 256 KiB of heavy items plus a small header.
static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

__global__ void k_noalloc_prepare(NoAllocScratch *s, const uint32_t *ev, const uint32_t *offsets,
                                  const uint32_t *active, int64_t n_active) {
  if (threadIdx.x == 0) {
    s->view = SlotView{ev, offsets, active, s->counters, nullptr, nullptr, nullptr, nullptr};
    for (int i = 0; i < 8; ++i) s->counters[i] = 0;
    s->counters[2] = (uint64_t)n_active;
    for (int i = 0; i < 8; ++i) s->qctl[i] = 0;
    s->flags = 0;
  }
}

// Heavy pixels (at least list_min events: kNoAllocHeavyMin, or fewer when the list
// holds every active pixel) into the work list, from its front, the big ones from
// its back. With distinct keys and offsets that stay within the n_events <=
// kNoAllocMaxEvents events of the call the list cannot overflow. A pixel that does
// not fit (more than kNoAllocMaxHeavy entries of both classes together: keys listed
// many times, or offsets beyond n_events) gets a row of NaN and raises
// DDHF_FLAG_CAPACITY. A place is asked for before an end is chosen, so that the two
// ends never meet.
__global__ void k_noalloc_heavy(NoAllocScratch *s, const uint32_t *offsets, const uint32_t *active,
                                int64_t n_active, float *P, int n_bins, int list_min) {
  bool for_scan = false;
  for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < n_active;
       a += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t k = active[a];
    const uint32_t cnt = offsets[k + 1] - offsets[k];
    if (cnt >= (uint32_t)list_min) {
      if (atomicAdd(&s->qctl[5], 1u) < (uint32_t)kNoAllocMaxHeavy) {
        const bool big = cnt >= (uint32_t)kBigPixel;
        const uint32_t pos = atomicAdd(&s->qctl[big ? 1 : 0], 1u);
        s->heavy[big ? kNoAllocMaxHeavy - 1 - pos : pos] = (uint32_t)a;
      } else {
        atomicOr(&s->flags, DDHF_FLAG_CAPACITY);
        for (int j = 0; j < n_bins; ++j) P[a * n_bins + j] = __int_as_float(0x7fc00000);
      }
    } else if (cnt >= (uint32_t)kTeamPixel) {
      for_scan = true;
    }
  }
  if (__any_sync(0xffffffffu, for_scan) && (threadIdx.x & 31) == 0) s->qctl[6] = 1u;
}

// The DDHF_FLAG_* bits this call raised, into the caller's word.
__global__ void k_noalloc_finish(const NoAllocScratch *s, uint32_t *flags_out) {
  if (threadIdx.x == 0) *flags_out = s->flags;
}

// Scratch address per CUDA context: (process-unique context id, address).
struct AddrEntry {
  unsigned long long ctx_id;
  NoAllocScratch *addr;
};
std::mutex g_addr_mu;
AddrEntry g_addr[kMaxContexts] = {};
int g_addr_n = 0;

typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long *);

// Id of the current context (0 when none is current or the query fails).
unsigned long long current_ctx_id() {
  static CtxGetIdFn fn = nullptr;
  static bool looked = false;
  if (!looked) {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<CtxGetIdFn>(f);
    looked = true;
  }
  unsigned long long id = 0;
  if (!fn || fn(nullptr, &id) != CUDA_SUCCESS) return 0;
  return id;
}

template <int MT>
cudaError_t load_blocked() {
  cudaFuncAttributes fa;
  const cudaError_t e = cudaFuncGetAttributes(&fa, blocked::k_blocked<MT, 1, false>);
  return e != cudaSuccess ? e : cudaFuncGetAttributes(&fa, blocked::k_team_scan<MT>);
}

// The scratch address for the current context: looked up, and every kernel of
// this entry point loaded, on the context's first call.
ddhf_status scratch_for_current(NoAllocScratch **out) {
  std::lock_guard<std::mutex> lock(g_addr_mu);
  unsigned long long id = current_ctx_id();
  for (int i = 0; id != 0 && i < g_addr_n; ++i)
    if (g_addr[i].ctx_id == id) {
      *out = g_addr[i].addr;
      return DDHF_OK;
    }
  void *p = nullptr;
  if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return DDHF_ERR_CUDA;
  cudaFuncAttributes fa;
  if (load_blocked<1>() != cudaSuccess || load_blocked<2>() != cudaSuccess ||
      load_blocked<3>() != cudaSuccess || load_blocked<4>() != cudaSuccess ||
      cudaFuncGetAttributes(&fa, k_noalloc_prepare) != cudaSuccess ||
      cudaFuncGetAttributes(&fa, k_noalloc_heavy) != cudaSuccess ||
      cudaFuncGetAttributes(&fa, k_noalloc_finish) != cudaSuccess)
    return DDHF_ERR_CUDA;
  if (id == 0) id = current_ctx_id();  // the symbol lookup made the primary context current
  if (id != 0 && g_addr_n < kMaxContexts) g_addr[g_addr_n++] = AddrEntry{id, static_cast<NoAllocScratch *>(p)};
  *out = static_cast<NoAllocScratch *>(p);
  return DDHF_OK;
}

template <int MT>
ddhf_status launch_noalloc(NoAllocScratch *sp, const GridConst &g, float *P, int64_t cap_px,
                           int64_t n_active, int64_t n_events, int list_min, int num_sms,
                           cudaStream_t s) {
  blocked::BlockedArgs A{};
  A.views = &sp->view;
  A.slot0 = 0;
  A.n_slots = 1;
  A.npx = n_active;  // light pixels: virtual index over the active list
  A.heavy = sp->heavy;
  A.n_heavy = &sp->qctl[0];
  A.heavy_cap = (uint32_t)kNoAllocMaxHeavy;
  A.cursors = &sp->qctl[2];
  A.N = g.N;
  A.nbr = g.nbr;
  A.nd = blocked::make_ndft_const(g.a0, g.da, g.denom, g.N, g.nbr, MT);
  A.cc = CombConst{};
  A.P = P;
  A.ld = g.N;
  A.vec_store = (A.ld % 4 == 0) && (reinterpret_cast<uintptr_t>(P) % 16 == 0);
  A.cap_px = cap_px;
  A.heavy_min = list_min;
  A.light_max = kTeamPixel;
  A.warp_bytes = blocked::Stage<MT>::kBytes;
  A.flags = &sp->flags;
  A.ev_cap = n_events;
  const size_t smem = (size_t)A.warp_bytes * kNoAllocWarps;
  auto kern = blocked::k_blocked<MT, 1, false>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return DDHF_ERR_CUDA;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kNoAllocWarps * 32, smem) !=
          cudaSuccess ||
      occ < 1)
    return DDHF_ERR_CUDA;
  if (blocked::launch_clusters(kern, num_sms * occ, blocked::kShares, kNoAllocWarps * 32, smem, s,
                               A) != cudaSuccess)
    return DDHF_ERR_CUDA;
  if (list_min <= kTeamPixel) return DDHF_OK;
  auto scan = blocked::k_team_scan<MT>;
  if (cudaFuncSetAttribute(scan, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return DDHF_ERR_CUDA;
  scan<<<(unsigned)(num_sms * 4), kNoAllocWarps * 32, smem, s>>>(A);
  return cudaGetLastError() == cudaSuccess ? DDHF_OK : DDHF_ERR_CUDA;
}

}  // namespace
}  // namespace ddhf

using namespace ddhf;

extern "C" ddhf_status ddhf_power_spectrum_noalloc(const ddhf_grid *grid, const uint32_t *offsets,
                                                   const uint32_t *ev, int64_t n_events,
                                                   const uint32_t *active, int64_t n_active,
                                                   float *P, int64_t cap_px, uint32_t *flags_dev,
                                                   ddhf_stream stream) {
  if (!grid || !offsets || !active || !P) return DDHF_ERR_INVALID_ARG;
  if (n_events < 0 || n_events > kNoAllocMaxEvents) return DDHF_ERR_INVALID_ARG;
  if (n_events > 0 && !ev) return DDHF_ERR_INVALID_ARG;
  if (n_active < 0 || n_active > ((int64_t)1 << 26) || cap_px < n_active)
    return DDHF_ERR_INVALID_ARG;
  if (!grid_ok(grid)) return DDHF_ERR_INVALID_ARG;
  int dev = 0, num_sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return DDHF_ERR_CUDA;
  if (cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return DDHF_ERR_CUDA;
  NoAllocScratch *sp = nullptr;
  const ddhf_status ss = scratch_for_current(&sp);
  if (ss != DDHF_OK) return ss;
  cudaStream_t s = (cudaStream_t)stream;
  if (n_active == 0) {
    if (flags_dev && cudaMemsetAsync(flags_dev, 0, sizeof(uint32_t), s) != cudaSuccess)
      return DDHF_ERR_CUDA;
    return DDHF_OK;
  }
  const GridConst g = make_grid_const(*grid);
  k_noalloc_prepare<<<1, 32, 0, s>>>(sp, ev, offsets, active, n_active);
  const int blocks = (int)std::min<int64_t>(ceil_div(n_active, 256), (int64_t)num_sms * 8);
  // up to kNoAllocMaxHeavy active pixels the list holds any of them, so those that go
  // to teams are listed too and k_team_scan is not needed (its blocks take them in
  // runs of active pixels: 300 pixels of 500 events 287 us, listed 55; 20,000 of 1000
  // events at 750 bins 1.25 ms, listed 0.97)
  const int list_min = n_active <= kNoAllocMaxHeavy ? kTeamPixel : kNoAllocHeavyMin;
  k_noalloc_heavy<<<blocks, 256, 0, s>>>(sp, offsets, active, n_active, P, g.N, list_min);
  if (cudaGetLastError() != cudaSuccess) return DDHF_ERR_CUDA;
  ddhf_status st;
  switch (blocked::tiles_per_pass(g.nbr, 0)) {
    case 1: st = launch_noalloc<1>(sp, g, P, cap_px, n_active, n_events, list_min, num_sms, s); break;
    case 2: st = launch_noalloc<2>(sp, g, P, cap_px, n_active, n_events, list_min, num_sms, s); break;
    case 3: st = launch_noalloc<3>(sp, g, P, cap_px, n_active, n_events, list_min, num_sms, s); break;
    default: st = launch_noalloc<4>(sp, g, P, cap_px, n_active, n_events, list_min, num_sms, s); break;
  }
  if (st != DDHF_OK) return st;
  if (flags_dev) {
    k_noalloc_finish<<<1, 32, 0, s>>>(sp, flags_dev);
    if (cudaGetLastError() != cudaSuccess) return DDHF_ERR_CUDA;
  }
  return DDHF_OK;
}
