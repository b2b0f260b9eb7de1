// Segmentation-mask processing (Sec. 3.5): 8-connected component labelling,
// per-component bounding boxes, the A_min area filter and centroid merging
// with Eq. 12, repeated to a fixed point.
//
// Labelling is a lock-free union-find over the pixel grid: the foreground runs
// of each 32-pixel segment start as one, and runs that touch are united (see
// k_label_union); a union always hooks the larger root under the smaller one (compare-and-swap on the
// root's parent), so every parent index is smaller than its child and the
// final root of a component is its smallest linear index, whatever order the
// unions ran in. Boxes use the root index as a slot (atomic min/max/add),
// survivors of the area filter are collected, and one thread block merges
// them: all pairs satisfying Eq. 12 are unioned (smallest index as root),
// each group becomes its union box, the survivors are compacted in root
// order, and the round repeats until no pair is close. The result is sorted
// by (y0, x0, y1, x1, n_px) by rank counting.
#include <algorithm>

#include "ddhf_internal.cuh"

namespace ddhf {

namespace {

// Every union-find loop below stops after `limit` iterations (the context's
// loop limit, 2^24 unless a test lowers it), raises DDHF_FLAG_TIMEOUT and
// returns an index that is still in range, so a run-out leaves wrong labels
// but no bad access.
__device__ __forceinline__ int find_root(int32_t *lab, int x, uint32_t *flags, int limit) {
  int it = 0;
  int p = lab[x];
  while (p != x) {
    int gp = lab[p];
    if (gp < p) lab[x] = gp;  // path halving; parents only move to smaller ancestors
    x = p;
    p = gp;
    if (++it > limit) {
      atomicOr(flags, DDHF_FLAG_TIMEOUT);
      break;
    }
  }
  return x;
}

__device__ __forceinline__ void unite(int32_t *lab, int a, int b, uint32_t *flags, int limit) {
  for (int it = 0; it < limit; ++it) {
    a = find_root(lab, a, flags, limit);
    b = find_root(lab, b, flags, limit);
    if (a == b) return;
    if (a < b) {
      int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(&lab[a], a, b) == a) return;
  }
  atomicOr(flags, DDHF_FLAG_TIMEOUT);
}

// Every foreground pixel starts at the first pixel of its run within its 32-pixel
// segment (one warp: 32 consecutive pixels, 32-aligned), so that the unions below
// work on runs: their trees start one level deep instead of a pixel per level
// (unions of a dense 1280x720 mask 38 -> 26 us, of a sparse one 15 -> 10 us).
__global__ void k_label_init(const uint8_t *__restrict__ mask, int32_t *__restrict__ lab, int W,
                             int64_t npx, uint64_t *n_fg) {
  uint32_t cnt = 0;
  const int lane = threadIdx.x & 31;
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; i0 < npx;
       i0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = i0 + lane;
    const bool fg = i < npx && mask[i] != 0;
    const uint32_t b = __ballot_sync(0xffffffffu, fg);
    const uint32_t row = __ballot_sync(0xffffffffu, (uint32_t)i % (uint32_t)W == 0);
    const uint32_t start = b & (~(b << 1) | row);  // lane 0 of a run that came in starts too
    const uint32_t mine = start & (0xffffffffu >> (31 - lane));
    if (i < npx) lab[i] = fg ? (int32_t)(i - lane + (31 - __clz(mine))) : -1;
    cnt += fg;
  }
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  if (lane == 0 && cnt && n_fg) atomicAdd((unsigned long long *)n_fg, cnt);
}

__global__ void k_label_union(const uint8_t *__restrict__ mask, int32_t *lab, int W, int H,
                              uint32_t *flags, int limit) {
  const int64_t npx = (int64_t)W * H;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npx;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (!mask[i]) continue;
    const int y = (int)((uint32_t)i / (uint32_t)W), x = (int)i - y * W;
    // Only the unions that no other pixel's own unions imply. A run that crosses
    // a segment is joined at the segment's first pixel. Two rows' overlapping
    // runs are joined where their overlap begins: a pixel whose left neighbour
    // also has its upper neighbour set leaves the union to that one (both rows
    // are connected between them). Diagonal contacts: the left neighbour, when
    // set, has the upper left above it, the right one the upper right. The
    // components (and so the minimum-index labels) are those of all
    // eight-neighbour unions.
    const bool left = x > 0 && mask[i - 1];
    if (left && (i & 31) == 0) unite(lab, (int)i, (int)(i - 1), flags, limit);
    if (y == 0) continue;
    const bool up_left = x > 0 && mask[i - W - 1];
    if (mask[i - W]) {
      if (!(left && up_left)) unite(lab, (int)i, (int)(i - W), flags, limit);
    } else {
      if (up_left && !left) unite(lab, (int)i, (int)(i - W - 1), flags, limit);
      if (x < W - 1 && mask[i - W + 1] && !mask[i + 1])
        unite(lab, (int)i, (int)(i - W + 1), flags, limit);
    }
  }
}

// Root of x without writing any parent: during the compress pass every thread
// writes only its own pixel, so no stale path-halving write can overwrite a
// root that another thread has already stored.
__device__ __forceinline__ int find_root_ro(const int32_t *lab, int x, uint32_t *flags,
                                            int limit) {
  for (int it = 0; it < limit; ++it) {
    const int p = lab[x];
    if (p == x) return x;
    x = p;
  }
  atomicOr(flags, DDHF_FLAG_TIMEOUT);
  return x;
}

// With bx (the detections, whose boxes follow): each root's box slot as
// k_box_root_init sets it (a root's own label does not change here).
__global__ void k_label_compress(int32_t *lab, int32_t *bx, int W, int64_t npx, uint32_t *flags,
                                 int limit) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npx;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t p = lab[i];
    if (p < 0) continue;
    if (p != (int32_t)i) {
      lab[i] = find_root_ro(lab, p, flags, limit);
    } else if (bx) {
      bx[i] = bx[2 * npx + i] = (int32_t)(i % W);
      bx[npx + i] = bx[3 * npx + i] = (int32_t)(i / W);
      bx[4 * npx + i] = 0;
    }
  }
}

// Box slots indexed by root pixel: x0, y0, x1, y1, n (5 arrays of npx int32).
__global__ void k_box_root_init(const int32_t *__restrict__ lab, int32_t *bx, int W, int64_t npx) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npx;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (lab[i] == (int32_t)i) {
      bx[i] = (int32_t)(i % W);
      bx[npx + i] = (int32_t)(i / W);
      bx[2 * npx + i] = (int32_t)(i % W);
      bx[3 * npx + i] = (int32_t)(i / W);
      bx[4 * npx + i] = 0;
    }
  }
}

// Pixels of one component usually share a warp, so the bounds are first
// reduced among the lanes with the same root and one lane updates the slot.
// A label at or beyond npx (a caller's labels array) is skipped and raises
// DDHF_FLAG_INPUT.
__global__ void k_box_accum(const int32_t *__restrict__ lab, int32_t *bx, int W, int64_t npx,
                            uint32_t *flags) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < npx; base += stride) {
    const int64_t i = base + threadIdx.x;
    int r = i < npx ? lab[i] : -1;
    if ((int64_t)r >= npx) {
      atomicOr(flags, DDHF_FLAG_INPUT);
      r = -1;
    }
    const uint32_t peers = __match_any_sync(0xffffffffu, r);
    if (r < 0) continue;
    const int x = (int)(i % W), y = (int)(i / W);
    const int xmin = __reduce_min_sync(peers, x);
    const int xmax = __reduce_max_sync(peers, x);
    const int ymax = __reduce_max_sync(peers, y);
    const int n = __popc(peers);
    if ((threadIdx.x & 31) == __ffs(peers) - 1) {
      atomicMin(&bx[r], xmin);
      atomicMax(&bx[2 * npx + r], xmax);
      atomicMax(&bx[3 * npx + r], ymax);
      atomicAdd(&bx[4 * npx + r], n);
    }
  }
}

// Survivors of the area filter, appended as quintuples (order fixed later).
__global__ void k_box_collect(const int32_t *__restrict__ lab, const int32_t *__restrict__ bx,
                              int64_t npx, int A_min, int32_t *list, uint32_t *count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npx;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (lab[i] != (int32_t)i) continue;
    const int x0 = bx[i], y0 = bx[npx + i], x1 = bx[2 * npx + i], y1 = bx[3 * npx + i];
    const int64_t area = (int64_t)(x1 - x0 + 1) * (int64_t)(y1 - y0 + 1);
    if (area < A_min) continue;
    const uint32_t pos = atomicAdd(count, 1u);
    int32_t *o = list + 5 * (int64_t)pos;
    o[0] = x0;
    o[1] = y0;
    o[2] = x1;
    o[3] = y1;
    o[4] = bx[4 * npx + i];
  }
}

// Every component (no area filter), shifted to sensor coordinates.
__global__ void k_comp_collect(const int32_t *__restrict__ lab, const int32_t *__restrict__ bx,
                               int64_t npx, int W, int32_t row0, ddhf_component *out, int cap,
                               uint32_t *count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npx;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (lab[i] != (int32_t)i) continue;
    const uint32_t pos = atomicAdd(count, 1u);
    if ((int64_t)pos >= cap) continue;
    ddhf_component c;
    c.label = (int32_t)(i + (int64_t)row0 * W);
    c.x0 = bx[i];
    c.y0 = bx[npx + i] + row0;
    c.x1 = bx[2 * npx + i];
    c.y1 = bx[3 * npx + i] + row0;
    c.n_px = bx[4 * npx + i];
    out[pos] = c;
  }
}

// Eq. 12 in FP64, every product rounded on its own.
__device__ __forceinline__ bool eq12_close(const int32_t *a, const int32_t *b, double alpha) {
  const int64_t dx2 = (int64_t)(a[0] + a[2]) - (int64_t)(b[0] + b[2]);
  const int64_t dy2 = (int64_t)(a[1] + a[3]) - (int64_t)(b[1] + b[3]);
  int64_t m = a[2] - a[0] + 1;
  m = max(m, (int64_t)(a[3] - a[1] + 1));
  m = max(m, (int64_t)(b[2] - b[0] + 1));
  m = max(m, (int64_t)(b[3] - b[1] + 1));
  const double lhs = (double)(dx2 * dx2 + dy2 * dy2);
  const double s = __dmul_rn(__dmul_rn(2.0, alpha), (double)m);
  return lhs < __dmul_rn(s, s);
}

__device__ __forceinline__ int gfind(int32_t *par, int x, uint32_t *flags, int limit) {
  int p = par[x];
  for (int it = 0; p != x; ++it) {
    int gp = par[p];
    par[x] = gp;
    x = p;
    p = gp;
    if (it > limit) {
      atomicOr(flags, DDHF_FLAG_TIMEOUT);
      break;
    }
  }
  return x;
}

__device__ __forceinline__ void gunite(int32_t *par, int a, int b, uint32_t *flags, int limit) {
  for (int it = 0; it < limit; ++it) {
    a = gfind(par, a, flags, limit);
    b = gfind(par, b, flags, limit);
    if (a == b) return;
    if (a < b) {
      int t = a;
      a = b;
      b = t;
    }
    if (atomicCAS(&par[a], a, b) == a) return;
  }
  atomicOr(flags, DDHF_FLAG_TIMEOUT);
}

__device__ __forceinline__ bool box_less(const int32_t *a, const int32_t *b) {
  for (int k = 0; k < 5; ++k) {
    const int ka = k == 0 ? 1 : k == 1 ? 0 : k == 2 ? 3 : k == 3 ? 2 : 4;  // y0, x0, y1, x1, n
    if (a[ka] != b[ka]) return a[ka] < b[ka];
  }
  return false;
}

constexpr int kMergeThreads = 1024;

__global__ void __launch_bounds__(kMergeThreads) k_box_merge(int32_t *list, int32_t *list2,
                                                             int32_t *par, int32_t *root,
                                                             const uint32_t *count,
                                                             double alpha, ddhf_box *out, int cap,
                                                             int32_t *n_out, uint32_t *flags,
                                                             int limit) {
  __shared__ int any;
  __shared__ uint32_t warp_tot[32];
  __shared__ uint32_t s_base;
  int B = (int)*count;
  const int tid = threadIdx.x, bs = blockDim.x;
  for (int round = 0; round <= B + 1; ++round) {
    for (int i = tid; i < B; i += bs) par[i] = i;
    if (tid == 0) any = 0;
    __syncthreads();
    const int64_t pairs = (int64_t)B * B;
    for (int64_t p = tid; p < pairs; p += bs) {
      const int i = (int)(p / B), j = (int)(p % B);
      if (j <= i) continue;
      if (eq12_close(list + 5 * (int64_t)i, list + 5 * (int64_t)j, alpha)) {
        any = 1;
        gunite(par, i, j, flags, limit);
      }
    }
    __syncthreads();
    if (!any) break;
    if (round == B + 1) {
      if (tid == 0) atomicOr(flags, DDHF_FLAG_TIMEOUT);
      break;
    }
    for (int i = tid; i < B; i += bs) root[i] = find_root_ro(par, i, flags, limit);
    __syncthreads();
    for (int i = tid; i < B; i += bs) par[i] = root[i];
    __syncthreads();
    for (int i = tid; i < B; i += bs) {
      if (par[i] == i) {
        int32_t *d = list2 + 5 * (int64_t)i;
        const int32_t *s = list + 5 * (int64_t)i;
        d[0] = s[0];
        d[1] = s[1];
        d[2] = s[2];
        d[3] = s[3];
        d[4] = 0;
      }
    }
    __syncthreads();
    for (int i = tid; i < B; i += bs) {
      const int r = par[i];
      int32_t *d = list2 + 5 * (int64_t)r;
      const int32_t *s = list + 5 * (int64_t)i;
      atomicMin(&d[0], s[0]);
      atomicMin(&d[1], s[1]);
      atomicMax(&d[2], s[2]);
      atomicMax(&d[3], s[3]);
      atomicAdd(&d[4], s[4]);
    }
    __syncthreads();
    // compact roots in index order into list
    if (tid == 0) s_base = 0;
    __syncthreads();
    for (int c0 = 0; c0 < B; c0 += bs) {
      const int i = c0 + tid;
      const bool root = i < B && par[i] == i;
      const uint32_t bal = __ballot_sync(0xffffffffu, root);
      const int lane = tid & 31, warp = tid >> 5;
      if (lane == 0) warp_tot[warp] = __popc(bal);
      __syncthreads();
      uint32_t wpre = 0;
      for (int w2 = 0; w2 < warp; ++w2) wpre += warp_tot[w2];
      const uint32_t pos = s_base + wpre + __popc(bal & ((1u << lane) - 1));
      if (root) {
        int32_t *d = list + 5 * (int64_t)pos;
        const int32_t *s = list2 + 5 * (int64_t)i;
        for (int k = 0; k < 5; ++k) d[k] = s[k];
      }
      __syncthreads();
      if (tid == 0) {
        uint32_t t = 0;
        for (int w2 = 0; w2 < (bs >> 5); ++w2) t += warp_tot[w2];
        s_base += t;
      }
      __syncthreads();
    }
    B = (int)s_base;
    __syncthreads();
  }
  for (int i = tid; i < B; i += bs) {
    const int32_t *bi = list + 5 * (int64_t)i;
    int rank = 0;
    for (int j = 0; j < B; ++j) {
      const int32_t *bj = list + 5 * (int64_t)j;
      if (box_less(bj, bi) || (j < i && !box_less(bi, bj))) ++rank;
    }
    if (rank < cap) {
      ddhf_box o;
      o.x0 = bi[0];
      o.y0 = bi[1];
      o.x1 = bi[2];
      o.y1 = bi[3];
      o.n_px = bi[4];
      out[rank] = o;
    }
  }
  if (tid == 0) {
    *n_out = B;
    if (B > cap) atomicOr(flags, DDHF_FLAG_CAPACITY);
  }
}

}  // namespace

ddhf_status launch_label(Ctx *c, const uint8_t *mask, int32_t *labels, uint64_t *nfg,
                         cudaStream_t s, bool boxes_follow) {
  const int blocks = c->num_sms * 8;
  DDHF_CUDA_TRY(c, cudaMemsetAsync(nfg, 0, sizeof(uint64_t), s));
  k_label_init<<<blocks, 256, 0, s>>>(mask, labels, c->W, c->npx, nfg);
  k_label_union<<<blocks, 256, 0, s>>>(mask, labels, c->W, c->H, c->flags, c->loop_limit);
  k_label_compress<<<blocks, 256, 0, s>>>(labels, boxes_follow ? c->box_tmp : nullptr, c->W,
                                          c->npx, c->flags, c->loop_limit);
  DDHF_CUDA_TRY(c, cudaGetLastError());
  return DDHF_OK;
}

// Dominant frequency of each box, over every block of the grid whatever the
// boxes' sizes (a crowded mask merges into one box that covers the sensor, and
// one block per box took 9.65 ms on a 1280x720 box of 921,348 rotor pixels:
// detection and frequencies of that window 15.06 ms, split as here 5.28 ms,
// of a 347x261 window 0.80 -> 0.57 ms). A box is cut into units of kF0Unit pixels of
// its rows (the work is one pass over the box's rotor pixels, bound by the
// latency of its dependent loads, so a unit is small enough that every warp of
// the grid gets one or two row segments); each unit offers its strongest pixel
// (SNR bits, -active index) to the box's maximum and adds its rotor pixels'
// dominant bins to the box's histogram, one counter per bin, and the box's
// last unit reads the lower median off the histogram. The order of these
// integer atomics does not matter. A box of one unit, as most are, needs no
// record: its block counts in shared memory and reads the median off there, or
// (grids of more than kF0SharedBins bins) selects it by two passes over 7 bits of
// the bin (3,000 boxes of 5x5 pixels at 750 bins: 103 us with a record each, 40 so;
// at 5000 bins 137 and 53).
//
// A record in scratch (the label workspace, free after the boxes are out): the
// maximum (2 words), rotor count, units done and N histogram counters.
// Whole calls on a 347x261, a sparse and a dense 1280x720 window (us): 292 / 305 /
// 3783; units of 1024 pixels 288 / 302 / 3791, of 16,384 305 / 311 / 3824; row segments
// of 128 pixels 292 / 304 / 3784, of 512 291 / 307 / 3797.
constexpr int kF0Unit = 4096;  // pixels of a box per unit
constexpr int kF0Seg = 256;    // pixels of a row per warp step
constexpr int kF0Head = 4;     // words of a box's record before its histogram
constexpr int kF0SharedBins = 4096;  // up to this many bins a unit counts in shared memory

struct BoxF0Args {
  const uint32_t *active;
  const uint64_t *counters;
  const uint8_t *mask;
  const float *snr;
  const int32_t *f0;
  const ddhf_box *boxes;
  const int32_t *n_boxes;
  int32_t cap, W, H, N;
  int32_t room;          // boxes that the scratch has entries for
  uint32_t *first_unit;  // [room + 1] first unit of each box
  uint32_t *rec_of;      // [room] the record of a box of several units
  int32_t rec_words;     // words of a record: kF0Head + N, rounded up to even
  int32_t rec_room;      // records
  uint32_t *rec;         // [rec_room][rec_words]
  int32_t *f0_out;
  float *snr_out, *med_hz;
  int64_t g_a0, g_da, g_denom;
  uint32_t *flags;
};

struct BoxRows {
  int x0, x1, y0, y1, nseg, items;  // clipped bounds, row segments, segments in all
};
__device__ __forceinline__ BoxRows box_rows(const BoxF0Args &A, const ddhf_box &b) {
  BoxRows r;
  r.x0 = max(b.x0, 0);
  r.x1 = min(b.x1, A.W - 1);
  r.y0 = max(b.y0, 0);
  r.y1 = min(b.y1, A.H - 1);
  r.nseg = r.x1 >= r.x0 ? (r.x1 - r.x0) / kF0Seg + 1 : 0;
  r.items = r.y1 >= r.y0 ? (r.y1 - r.y0 + 1) * r.nseg : 0;
  return r;
}
__device__ __forceinline__ uint32_t box_units(const BoxRows &r) {
  const int64_t px = r.items > 0 ? (int64_t)(r.x1 - r.x0 + 1) * (r.y1 - r.y0 + 1) : 0;
  return (uint32_t)max((int64_t)1, (px + kF0Unit - 1) / kF0Unit);
}

// First index i of the ascending active[0..n) with active[i] >= key, by the
// whole warp: each step narrows the range to one of 32 parts.
__device__ __forceinline__ int64_t warp_lower_bound(const uint32_t *active, int64_t n,
                                                    uint32_t key) {
  const int lane = threadIdx.x & 31;
  int64_t l = 0, r = n;  // active[l - 1] < key <= active[r]
  while (r - l > 32) {
    const int64_t step = (r - l) / 32;
    const int64_t m = l + (lane + 1) * step - 1;
    const uint32_t lower = __popc(__ballot_sync(0xffffffffu, active[m] < key));
    // the values ascend, so the lanes below `lower` are the ones under the key
    if (lower < 32) r = l + (lower + 1) * step - 1;
    l += lower * step;
  }
  const bool under = l + lane < r && active[l + lane] < key;
  return l + __popc(__ballot_sync(0xffffffffu, under));
}

// Row segments first, first + step, ... of a box: fn(i) for every rotor pixel
// i (active index) in them, warp by warp.
template <typename F>
__device__ __forceinline__ void box_visit(const BoxF0Args &A, const BoxRows &r, int64_t n_act,
                                          int first, int step, int end, F fn) {
  const int lane = threadIdx.x & 31;
  for (int it = first; it < end; it += step) {
    const int y = r.y0 + it / r.nseg, xs = r.x0 + (it % r.nseg) * kF0Seg;
    const uint32_t lo = (uint32_t)((int64_t)y * A.W + xs);
    const uint32_t hi = (uint32_t)((int64_t)y * A.W + min(r.x1, xs + kF0Seg - 1));
    const int64_t l = warp_lower_bound(A.active, n_act, lo);
    // at most kF0Seg active pixels lie in the segment
    uint32_t key[kF0Seg / 32];
#pragma unroll
    for (int u = 0; u < kF0Seg / 32; ++u) {
      const int64_t i = l + lane + 32 * u;
      key[u] = i < n_act ? A.active[i] : 0xffffffffu;
    }
#pragma unroll
    for (int u = 0; u < kF0Seg / 32; ++u)
      if (key[u] <= hi && A.mask[key[u]]) fn(l + lane + 32 * u);
  }
}

__device__ __forceinline__ void box_f0_best(const BoxF0Args &A, int b, unsigned long long best) {
  if (best == 0ull) {
    A.f0_out[b] = -1;
    if (A.snr_out) A.snr_out[b] = 0.f;
  } else {
    const uint32_t i = 0xffffffffu - (uint32_t)best;
    A.f0_out[b] = A.f0[i];
    if (A.snr_out) A.snr_out[b] = A.snr[i];
  }
}

__device__ __forceinline__ float box_f0_hz(const BoxF0Args &A, uint32_t bin) {
  return (float)((double)(A.g_a0 + (int64_t)bin * A.g_da) * 1e6 / (double)A.g_denom);
}

// Strongest pixel and rotor count of the block's warps.
__device__ __forceinline__ void box_f0_reduce(unsigned long long &best, uint32_t &n,
                                              unsigned long long *red, uint32_t *cnt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long u = __shfl_xor_sync(0xffffffffu, best, o);
    best = u > best ? u : best;
    n += __shfl_xor_sync(0xffffffffu, n, o);
  }
  __syncthreads();
  if (lane == 0) {
    red[warp] = best;
    cnt[warp] = n;
  }
  __syncthreads();
  best = red[0];
  n = cnt[0];
  for (int w = 1; w < 8; ++w) {
    best = red[w] > best ? red[w] : best;
    n += cnt[w];
  }
}

// The lower median (the bin of rank (total - 1) / 2) of a histogram, get(k) being
// counter k, by the whole block; cnt: eight words.
template <typename G>
__device__ __forceinline__ void box_f0_median(const BoxF0Args &A, int b, uint32_t total,
                                              uint32_t *cnt, G get) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t rank = total > 0 ? (total - 1) / 2 : 0;
  const int per = (A.N + 255) / 256, k0 = (int)threadIdx.x * per, k1 = min(A.N, k0 + per);
  uint32_t own = 0;
  for (int k = k0; k < k1; ++k) own += get(k);
  uint32_t inc = own;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  __syncthreads();  // cnt has been read
  if (lane == 31) cnt[warp] = inc;
  __syncthreads();
  uint32_t pre = inc - own;
  for (int w = 0; w < warp; ++w) pre += cnt[w];
  if (total == 0) {
    if (threadIdx.x == 0) A.med_hz[b] = 0.f;
  } else if (rank >= pre && rank < pre + own) {
    uint32_t run = pre;
    for (int k = k0; k < k1; ++k) {
      const uint32_t h = get(k);
      if (rank < run + h) {
        A.med_hz[b] = box_f0_hz(A, (uint32_t)k);
        break;
      }
      run += h;
    }
  }
}

struct BoxF0Shared {
  unsigned long long red[8];
  uint32_t cnt[8];
  uint32_t hist[128];
  uint32_t sel[2];
};

// A whole box by one block. SHARED: sh_hist holds a counter per bin; else the
// lower median by a two-digit radix selection (bins below 2^14, 7 bits per pass).
template <bool SHARED>
__device__ __forceinline__ void box_f0_one(const BoxF0Args &A, int b, int64_t n_act,
                                           BoxF0Shared &sh, uint32_t *sh_hist) {
  const int warp = threadIdx.x >> 5;
  const BoxRows r = box_rows(A, A.boxes[b]);
  const bool want_med = A.med_hz != nullptr;
  if (SHARED && want_med) {
    for (int k = threadIdx.x; k < A.N; k += blockDim.x) sh_hist[k] = 0;
    __syncthreads();
  }
  unsigned long long best = 0ull;
  uint32_t n = 0;
  box_visit(A, r, n_act, warp, 8, r.items, [&](int64_t i) {
    const unsigned long long v =
        ((unsigned long long)__float_as_uint(A.snr[i]) << 32) | (0xffffffffu - (uint32_t)i);
    best = v > best ? v : best;
    ++n;
    if (SHARED && want_med)
      atomicAdd(&sh_hist[min((uint32_t)A.f0[i], (uint32_t)A.N - 1)], 1u);  // always below N
  });
  box_f0_reduce(best, n, sh.red, sh.cnt);  // its barriers also end the shared counting
  if (threadIdx.x == 0) box_f0_best(A, b, best);
  if (!want_med) return;
  if (SHARED) {
    box_f0_median(A, b, n, sh.cnt, [&](int k) { return sh_hist[k]; });
    __syncthreads();
    return;
  }
  uint32_t rank = n > 0 ? (n - 1) / 2 : 0, prefix = 0;
  for (int pass = 0; pass < 2 && n > 0; ++pass) {
    const int shift = pass == 0 ? 7 : 0;
    for (int k = threadIdx.x; k < 128; k += blockDim.x) sh.hist[k] = 0;
    __syncthreads();
    box_visit(A, r, n_act, warp, 8, r.items, [&](int64_t i) {
      const uint32_t v = (uint32_t)A.f0[i];
      if (!ddhf_check(v < (1u << 14), A.flags)) return;
      if (pass == 1 && (v >> 7) != prefix) return;
      atomicAdd(&sh.hist[(v >> shift) & 127u], 1u);
    });
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t run = 0;
      int dsel = 127;
      for (int k = 0; k < 128; ++k) {
        if (rank < run + sh.hist[k]) {
          dsel = k;
          break;
        }
        run += sh.hist[k];
      }
      sh.sel[0] = (uint32_t)dsel;
      sh.sel[1] = rank - run;
    }
    __syncthreads();
    prefix = pass == 0 ? sh.sel[0] : (prefix << 7) | sh.sel[0];
    rank = sh.sel[1];
    __syncthreads();
  }
  if (threadIdx.x == 0) A.med_hz[b] = n > 0 ? box_f0_hz(A, prefix) : 0.f;
}

// Exclusive sum of v over the block's 256 threads, plus base, which then takes the
// total too.
__device__ __forceinline__ uint32_t box_scan(uint32_t v, uint32_t &base, uint32_t *cnt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  __syncthreads();  // cnt has been read
  if (lane == 31) cnt[warp] = inc;
  __syncthreads();
  uint32_t pre = base;
  for (int w = 0; w < 8; ++w) {
    if (w < warp) pre += cnt[w];
    base += cnt[w];
  }
  return pre + inc - v;
}

// Units and records of the boxes, and the records cleared. A box of several units
// takes the next record; without one (boxes of more than kF0Unit pixels beyond
// rec_room) it is one unit. Every block does the sums, to know how many records to
// clear, and block 0 writes them. Boxes beyond the room (a caller's capacity of
// more than 15 npx / 4 boxes) are done here, one block each.
__global__ void __launch_bounds__(256) k_box_f0_plan(BoxF0Args A) {
  __shared__ BoxF0Shared sh;
  const int nb = min(*A.n_boxes, A.cap), nr = min(nb, A.room);
  uint32_t recs = 0, units = 0;
  for (int b0 = 0; b0 < nr; b0 += 256) {
    const int b = b0 + (int)threadIdx.x;
    const uint32_t own = b < nr ? box_units(box_rows(A, A.boxes[b])) : 0u;
    const uint32_t r = box_scan(own > 1 ? 1u : 0u, recs, sh.cnt);
    const bool has_rec = own > 1 && r < (uint32_t)A.rec_room;
    const uint32_t u = box_scan(has_rec ? own : min(own, 1u), units, sh.cnt);
    if (blockIdx.x == 0 && b < nr) {
      A.first_unit[b] = u;
      A.rec_of[b] = r;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) A.first_unit[max(nr, 0)] = units;
  const int64_t words = (int64_t)min(recs, (uint32_t)A.rec_room) * A.rec_words;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < words;
       i += (int64_t)gridDim.x * blockDim.x)
    A.rec[i] = 0;
  const int64_t n_act = (int64_t)A.counters[2];
  for (int b = A.room + (int)blockIdx.x; b < nb; b += (int)gridDim.x)
    box_f0_one<false>(A, b, n_act, sh, nullptr);
}

// The box of unit u: the last b with first[b] <= u (first ascends, first[nb] > u),
// by the whole warp.
__device__ __forceinline__ int unit_box(const uint32_t *first, int nb, uint32_t u) {
  int lo = 0, hi = nb;
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32, i = lo + ((int)(threadIdx.x & 31) + 1) * step;
    const int below = __popc(__ballot_sync(0xffffffffu, i < hi && first[i] <= u));
    lo += below * step;
    hi = min(hi, lo + step);
  }
  return lo;
}

// The units of the boxes, and the results of a box of several by its last unit.
// SHARED: a unit counts its bins in shared memory first.
template <bool SHARED>
__global__ void __launch_bounds__(256) k_box_f0_units(BoxF0Args A) {
  extern __shared__ uint32_t sh_hist[];
  __shared__ BoxF0Shared sh;
  __shared__ uint32_t s_last;
  const int nr = min(min(*A.n_boxes, A.cap), A.room);
  if (nr <= 0) return;
  const int warp = threadIdx.x >> 5;
  const int64_t n_act = (int64_t)A.counters[2];
  const uint32_t n_units = A.first_unit[nr];
  const bool want_med = A.med_hz != nullptr;
  for (uint32_t u = blockIdx.x; u < n_units; u += gridDim.x) {
    const int b = n_units == (uint32_t)nr ? (int)u : unit_box(A.first_unit, nr, u);
    const uint32_t part = u - A.first_unit[b], parts = A.first_unit[b + 1] - A.first_unit[b];
    if (parts == 1) {
      box_f0_one<SHARED>(A, b, n_act, sh, sh_hist);
      continue;
    }
    const BoxRows r = box_rows(A, A.boxes[b]);
    uint32_t *rec = A.rec + (int64_t)A.rec_of[b] * A.rec_words, *hist = rec + kF0Head;
    if (SHARED && want_med) {
      for (int k = threadIdx.x; k < A.N; k += blockDim.x) sh_hist[k] = 0;
      __syncthreads();
    }
    const int i0 = (int)((int64_t)r.items * part / parts);
    const int i1 = (int)((int64_t)r.items * (part + 1) / parts);
    unsigned long long best = 0ull;
    uint32_t n = 0;
    box_visit(A, r, n_act, i0 + warp, 8, i1, [&](int64_t i) {
      const unsigned long long v =
          ((unsigned long long)__float_as_uint(A.snr[i]) << 32) | (0xffffffffu - (uint32_t)i);
      best = v > best ? v : best;
      ++n;
      if (!want_med) return;
      const uint32_t f = min((uint32_t)A.f0[i], (uint32_t)A.N - 1);  // always below N
      atomicAdd(SHARED ? &sh_hist[f] : &hist[f], 1u);
    });
    box_f0_reduce(best, n, sh.red, sh.cnt);  // its barriers also end the shared counting
    if (SHARED && want_med)
      for (int k = threadIdx.x; k < A.N; k += blockDim.x)
        if (sh_hist[k]) atomicAdd(&hist[k], sh_hist[k]);
    if (threadIdx.x == 0) {
      if (best) atomicMax(reinterpret_cast<unsigned long long *>(rec), best);
      if (n) atomicAdd(&rec[2], n);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&rec[3], 1u) == parts - 1;
    __syncthreads();
    if (!s_last) continue;
    __threadfence();
    if (threadIdx.x == 0)
      box_f0_best(A, b, __ldcg(reinterpret_cast<const unsigned long long *>(rec)));
    if (!want_med) continue;
    box_f0_median(A, b, __ldcg(&rec[2]), sh.cnt, [&](int k) { return __ldcg(&hist[k]); });
    __syncthreads();
  }
}

ddhf_status launch_box_f0(Ctx *c, int slot, const ddhf_box *boxes, const int32_t *n_boxes,
                          int32_t cap, int32_t *f0_out, float *snr_out, float *med_hz,
                          cudaStream_t s) {
  const Slot &sl = c->slots[slot];
  if (cap <= 0) return DDHF_OK;
  BoxF0Args A{};
  A.active = sl.active;
  A.counters = sl.counters;
  A.mask = sl.mask;
  A.snr = sl.snr;
  A.f0 = sl.f0;
  A.boxes = boxes;
  A.n_boxes = n_boxes;
  A.cap = cap;
  A.W = c->W;
  A.H = c->H;
  A.N = c->grid.n_bins;
  // in the box workspace of 15 npx words: two words of a box each and one more, in
  // up to half of it, then the records (8-byte aligned, of an even number of words)
  A.rec_words = (kF0Head + A.N + 1) & ~1;
  const int64_t words = 15 * c->npx;
  A.room = (int32_t)std::min<int64_t>(cap, words / 4);
  A.first_unit = reinterpret_cast<uint32_t *>(c->box_tmp);
  A.rec_of = A.first_unit + A.room + 1;
  const int64_t head = (2 * (int64_t)A.room + 2) & ~(int64_t)1;
  A.rec = A.first_unit + head;
  A.rec_room = (int32_t)std::max<int64_t>(0, (words - head) / A.rec_words);
  A.f0_out = f0_out;
  A.snr_out = snr_out;
  A.med_hz = med_hz;
  // bin j at (a0 + j da) / denom cycles per microsecond
  A.g_a0 = c->grid.a0;
  A.g_da = c->grid.da;
  A.g_denom = c->grid.denom;
  A.flags = c->flags;
  k_box_f0_plan<<<c->num_sms, 256, 0, s>>>(A);
  if (A.room > 0) {
    const unsigned units = (unsigned)c->num_sms * 6;
    if (A.N <= kF0SharedBins)
      k_box_f0_units<true><<<units, 256, A.N * sizeof(uint32_t), s>>>(A);
    else
      k_box_f0_units<false><<<units, 256, 0, s>>>(A);
  }
  DDHF_CUDA_TRY(c, cudaGetLastError());
  return DDHF_OK;
}

ddhf_status launch_components(Ctx *c, const int32_t *labels, int32_t row0, ddhf_component *out,
                              int32_t cap, int32_t *n_out, cudaStream_t s) {
  const int blocks = c->num_sms * 8;
  const int64_t npx = c->npx;
  int32_t *bx = c->box_tmp;  // 5 * npx
  uint32_t *count = reinterpret_cast<uint32_t *>(n_out);
  DDHF_CUDA_TRY(c, cudaMemsetAsync(count, 0, sizeof(uint32_t), s));
  k_box_root_init<<<blocks, 256, 0, s>>>(labels, bx, c->W, npx);
  k_box_accum<<<blocks, 256, 0, s>>>(labels, bx, c->W, npx, c->flags);
  k_comp_collect<<<blocks, 256, 0, s>>>(labels, bx, npx, c->W, row0, out, cap, count);
  DDHF_CUDA_TRY(c, cudaGetLastError());
  return DDHF_OK;
}

ddhf_status launch_boxes(Ctx *c, const int32_t *labels, ddhf_box *boxes, int32_t cap,
                         int32_t *n_boxes, cudaStream_t s, bool after_label) {
  const int blocks = c->num_sms * 8;
  const int64_t npx = c->npx;
  int32_t *bx = c->box_tmp;                  // 5 * npx
  int32_t *list = c->box_tmp + 5 * npx;      // 5 * npx
  int32_t *list2 = c->box_tmp + 10 * npx;    // 5 * npx
  int32_t *par = c->box_root;                // npx
  uint32_t *count = c->qctl + 9;
  DDHF_CUDA_TRY(c, cudaMemsetAsync(count, 0, sizeof(uint32_t), s));
  if (!after_label) k_box_root_init<<<blocks, 256, 0, s>>>(labels, bx, c->W, npx);
  k_box_accum<<<blocks, 256, 0, s>>>(labels, bx, c->W, npx, c->flags);
  k_box_collect<<<blocks, 256, 0, s>>>(labels, bx, npx, c->params.A_min, list, count);
  k_box_merge<<<1, kMergeThreads, 0, s>>>(list, list2, par, bx, count, c->params.alpha, boxes,
                                          cap, n_boxes, c->flags, c->loop_limit);
  DDHF_CUDA_TRY(c, cudaGetLastError());
  return DDHF_OK;
}

}  // namespace ddhf
