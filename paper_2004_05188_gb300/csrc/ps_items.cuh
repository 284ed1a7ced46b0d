// Building blocks of the kernels that give every central its lanes (exact query, batched sweep): the
// search of an item's candidates, the direct bins, the k smallest distances.
#pragma once

#include "ps_internal.cuh"
#include "ps_sweep.cuh"

namespace ps {

constexpr int kMaxRuns = 49;         // (2 * stencil + 1)^2 for stencil <= 3
constexpr uint32_t kHalf = 16;       // candidate pairs tested between two insertions
constexpr uint32_t kRing = 128;      // candidates kept for testing (a batch of 64 and 63 more)

// the neighbour records a search walks
struct Search {
  const float4* nrec;
  const uint32_t* nstart;
  const uint32_t* nsub;   // sub-cell starts (where the cells have sub-cells)
  int stencil;
  const int8_t* row_w;    // half-width of each stencil row (see row_widths)
};

template <int K>
__device__ __forceinline__ void topk_insert(float (&top)[K], float x) {
  if (x < top[K - 1]) {
#pragma unroll
    for (int t = K - 1; t > 0; --t) top[t] = fminf(top[t], fmaxf(x, top[t - 1]));
    top[0] = fminf(top[0], x);
  }
}

template <int K>
__device__ __forceinline__ float topk_get(const float (&top)[K], uint32_t idx) {
  float v = INFINITY;
#pragma unroll
  for (int t = 0; t < K; ++t)
    if ((uint32_t)t == idx) v = top[t];
  return v;
}

// Bound on the k-th distance (k <= K) of the central that the lane shares with L - 1 others, each
// holding the K smallest of its part of the candidates: the K-th of any one list, and the largest over
// the lists of their ceil(K / L)-th values, below or at which the lists together hold K.
template <int K>
__device__ __forceinline__ float topk_bound(const float (&top)[K], uint32_t L) {
  float kth = top[K - 1];
  if (L > 1u) {
    float part = top[(K + 15) / 16 - 1];
    if (L == 2u) part = top[(K + 1) / 2 - 1];
    if (L == 4u) part = top[(K + 3) / 4 - 1];
    if (L == 8u) part = top[(K + 7) / 8 - 1];
#pragma unroll 1
    for (uint32_t o = 1; o < L; o <<= 1) {
      kth = fminf(kth, __shfl_xor_sync(0xffffffffu, kth, o));
      part = fmaxf(part, __shfl_xor_sync(0xffffffffu, part, o));
    }
    kth = fminf(kth, part);
  }
  return kth;
}

// bin b in [0, nb) with sE[b] <= d2 < sE[b+1]; caller guarantees sE[0] <= d2 < sE[nb].
// The guess from an approximate square root is checked against the exact edge
// table; the (rare) wrong guess is walked to the right bin.
__device__ __forceinline__ uint32_t bin_index(float d2, const float* sE, uint32_t nb, float r0f, float inv_dr) {
  const float d = d2 > 0.f ? d2 * rsqrtf(d2) : 0.f;
  int b = (int)((d - r0f) * inv_dr);
  b = b < 0 ? 0 : (b >= (int)nb ? (int)nb - 1 : b);
  if (d2 < sE[b] || d2 >= sE[b + 1]) {
    while (b > 0 && d2 < sE[b]) --b;
    while (b + 1 < (int)nb && d2 >= sE[b + 1]) ++b;
  }
  return (uint32_t)b;
}

// The inline assembly below writes shared memory without telling the compiler so (no "memory" clobber, which
// would make it reload what the pair loops hold in registers).  That is sound because C++ code reads or
// writes those words only behind a barrier: volatile statements keep their order among themselves and
// around __syncwarp / __syncthreads / the votes, which the compiler takes as barriers for memory.
//
// Insertion queue of a lane: a column of a [row][32 lanes] array, `at` the shared address of its next
// slot.  Every value is stored and the slot taken only if it is below thr: no branch, and one
// predicated add per value.
__device__ __forceinline__ void queue_push(uint32_t& at, float v, float thr) {
  asm volatile(
      "{\n .reg .pred p;\n st.shared.f32 [%0], %1;\n setp.lt.f32 p, %1, %2;\n @p add.u32 %0, %0, 128;\n}"
      : "+r"(at)
      : "f"(v), "f"(thr));
}
// the same for a candidate of index word j, other than the lane's central (index word own)
__device__ __forceinline__ void queue_push_other(uint32_t& at, float v, float thr, uint32_t j, uint32_t own) {
  asm volatile(
      "{\n .reg .pred p;\n st.shared.f32 [%0], %1;\n setp.ne.u32 p, %3, %4;\n setp.lt.and.f32 p, %1, %2, p;\n"
      " @p add.u32 %0, %0, 128;\n}"
      : "+r"(at)
      : "f"(v), "f"(thr), "r"(j), "r"(own));
}
__device__ __forceinline__ float queue_at(uint32_t first, uint32_t q) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(first + 128u * q));
  return v;
}

// Rows of the stencil, nearest first: (dy, dz) ordered by dy^2 + dz^2 (the first 9 entries are
// the 3 x 3 rows of the 27-cell stencil, the first 25 the 5 x 5 rows).  Walking the central row
// first lets the k-th distance of every central settle early, so later candidates rarely enter
// the top-k lists.
static __constant__ signed char c_row_dy[kMaxRuns] = {0, -1, 1, 0, 0, -1, 1, -1, 1, -2, 2, 0, 0, -2, 2, -2, 2,
                                               -1, 1, -1, 1, -2, 2, -2, 2, 0, 0, -3, 3, -1, 1, -1, 1,
                                               -3, 3, -3, 3, -2, 2, -2, 2, -3, 3, -3, 3, -3, 3, -3, 3};
static __constant__ signed char c_row_dz[kMaxRuns] = {0, 0, 0, -1, 1, -1, -1, 1, 1, 0, 0, -2, 2, -1, -1, 1, 1,
                                               -2, -2, 2, 2, -2, -2, 2, 2, -3, 3, 0, 0, -3, -3, 3, 3,
                                               -1, -1, 1, 1, -3, -3, 3, 3, -2, -2, 2, 2, -3, -3, 3, 3};

__device__ __forceinline__ int row_width(const Search& a, int dy, int dz) {
  const int s = a.stencil;
  return a.row_w[(dz + s) * (2 * s + 1) + dy + s];
}

// x-run of cells cx - w .. cx + w (clipped to the grid) of row (y, z): its records
__device__ __forceinline__ void row_run(const Search& a, const Geo& ng, uint32_t cx, int y, int z, int w,
                                        uint32_t& src, uint32_t& len) {
  src = 0;
  len = 0;
  if (w < 0 || y < 0 || z < 0 || y >= (int)ng.dims[1] || z >= (int)ng.dims[2]) return;
  const uint32_t xlo = cx >= (uint32_t)w ? cx - w : 0;
  const uint32_t xhi = cx + w < ng.dims[0] ? cx + w : ng.dims[0] - 1;
  const uint32_t row = ((uint32_t)z * ng.dims[1] + (uint32_t)y) * ng.dims[0];
  src = a.nstart[row + xlo];
  len = a.nstart[row + xhi + 1] - src;
}

// cell c -> run r of its stencil: the x-contiguous records of cells (cx-w .. cx+w, cy+dy, cz+dz)
__device__ __forceinline__ void cell_run(const Search& a, const Geo& ng, uint32_t c, uint32_t r, uint32_t& src,
                                         uint32_t& len) {
  const int s = a.stencil, w = 2 * s + 1;
  const uint32_t cx = c % ng.dims[0], cy = (c / ng.dims[0]) % ng.dims[1], cz = c / (ng.dims[0] * ng.dims[1]);
  src = 0;
  len = 0;
  if ((int)r >= w * w) return;
  const int dy = c_row_dy[r], dz = c_row_dz[r];
  row_run(a, ng, cx, (int)cy + dy, (int)cz + dz, row_width(a, dy, dz), src, len);
}

// Run r of the candidates of an item whose box, in cell edges, is ulo .. uhi.  Cells without sub-cells:
// the own cell, the own row to its left and to its right, then rows 1 .. of the stencil (nearest
// first).  With them, the x-rods of 2^sub sub-cells, cell by cell from the own row
// outwards, those out of reach left empty: a 2 nm cell's 27 cells hold 216 octants, an octant's
// items reach 105 of them within 2 nm and about 27 within a 10th-neighbour distance.
__device__ __forceinline__ uint32_t item_runs(const Search& a, const Geo& ng) {
  const uint32_t W = 2 * a.stencil + 1;
  return ng.sub ? W * W * W << (2 * ng.sub) : W * W + 2;
}
__device__ __forceinline__ void item_run(const Search& a, const Geo& ng, uint32_t c, uint32_t r, const float (&ulo)[3],
                                         const float (&uhi)[3], float lim_u, uint32_t& src, uint32_t& len) {
  src = 0, len = 0;
  if (r >= item_runs(a, ng)) return;
  if (ng.sub) {
    const uint32_t W = 2 * a.stencil + 1, cell = r >> (2 * ng.sub), yz = r & ((1u << (2 * ng.sub)) - 1u);
    const int row = (int)(cell / W), q = (int)(cell - row * W), dx = q & 1 ? -((q + 1) >> 1) : q >> 1;  // 0 -1 1 -2 2 ..
    const int x = (int)(c % ng.dims[0]) + dx, y = (int)((c / ng.dims[0]) % ng.dims[1]) + c_row_dy[row],
              z = (int)(c / (ng.dims[0] * ng.dims[1])) + c_row_dz[row];
    if (x < 0 || y < 0 || z < 0 || x >= (int)ng.dims[0] || y >= (int)ng.dims[1] || z >= (int)ng.dims[2]) return;
    const float e = 1.0f / (float)(1u << ng.sub);
    const float y0 = (float)y + e * (float)(yz & ((1u << ng.sub) - 1u)), z0 = (float)z + e * (float)(yz >> ng.sub);
    const float gx = fmaxf(0.f, fmaxf((float)x - uhi[0], ulo[0] - (float)(x + 1)));
    const float gy = fmaxf(0.f, fmaxf(y0 - uhi[1], ulo[1] - (y0 + e)));
    const float gz = fmaxf(0.f, fmaxf(z0 - uhi[2], ulo[2] - (z0 + e)));
    if (gx * gx + gy * gy + gz * gz > lim_u) return;  // (a NaN box keeps the rod)
    const uint32_t cc = ((uint32_t)z * ng.dims[1] + (uint32_t)y) * ng.dims[0] + (uint32_t)x;
    const uint32_t f = (cc << (3 * ng.sub)) | (yz << ng.sub), f1 = f + (1u << ng.sub);
    src = a.nsub[f];
    len = (f1 == ng.n_cells << (3 * ng.sub) ? ng.n_sel : a.nsub[f1]) - src;
    return;
  }
  if (r >= 3) {
    cell_run(a, ng, c, r - 2, src, len);
    return;
  }
  const uint32_t row = c - c % ng.dims[0], cx = c - row, w = (uint32_t)row_width(a, 0, 0);
  const uint32_t lo = r == 0 ? cx : (r == 1 ? (cx >= w ? cx - w : 0u) : cx + 1);
  const uint32_t hi = r == 0 ? cx + 1 : (r == 1 ? cx : min(cx + w, ng.dims[0] - 1) + 1);
  if (lo < hi) {
    src = a.nstart[row + lo];
    len = a.nstart[row + hi] - src;
  }
}

// ---------------------------------------------------------------------------
// direct bins (r0 = 0)
// ---------------------------------------------------------------------------
constexpr float kBinBias = 1.0f / 2097152.0f;   // 2^-21

__device__ __forceinline__ void red_shared_inc(uint32_t addr) {
  asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(addr));
}
__device__ __forceinline__ void red_shared(uint32_t addr, uint32_t v) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v));
}

// Bins of the direct form (r0 = 0).  With s = sqrt.approx(d2) and inv = (1 +- 2^-21) / dr, the true
// quotient sqrt(d2) / dr lies between s * inv- and s * inv+ (the root is good to 2^-23, inv to 2^-24,
// the edge table to 2^-25 of the distance).  The bin is floor(s * inv+), or the one below where the two floors
// differ (2 in 10^4 pairs at 200 bins): those compare d2 with that edge.  Pairs out of range are
// clamped into the unused bin n_bins, so that every lane increments and no instruction is
// predicated: the compiler branches around a predicated shared-memory increment.  Measured on the
// pair loop alone (cycles per 32 tests and scheduler): 23 with a predicated increment and the excess over
// the edge computed, 17 in this form, of which 14.5 are the distance, root and floor; no table load per pair, so
// the shared-memory pipe is left to the increments (increments by one merge in a bin).
struct FastBins {
  const float* sE;
  unsigned long long hi2, lo2, magic2;
  float s_far;
  __device__ void init(uint32_t n_bins, double dr, const float* edges) {
    sE = edges;
    const float hi = (float)((1.0 + (double)kBinBias) / dr), lo = (float)((1.0 - (double)kBinBias) / dr);
    hi2 = f2_pack(hi, hi);
    lo2 = f2_pack(lo, lo);
    magic2 = f2_pack(kMagic, kMagic);
    s_far = (float)(((double)n_bins + 0.5) * dr);
  }
  // counts two pairs in the row at shared address `base` (bin b at base + 4 (kMagicBits + b));
  // returns 0 unless one of them may lie under the edge of its bin
  __device__ __forceinline__ uint32_t count2(unsigned long long d2, uint32_t base) const {
    float da, db, ma, mb, la, lb;
    f2_unpack(d2, da, db);
    const unsigned long long s2 = f2_pack(fminf(sqrt_fast(da), s_far), fminf(sqrt_fast(db), s_far));
    f2_unpack(f2_fma_down(s2, hi2, magic2), ma, mb);
    f2_unpack(f2_fma_down(s2, lo2, magic2), la, lb);
    red_shared_inc(__float_as_uint(ma) * 4u + base);
    red_shared_inc(__float_as_uint(mb) * 4u + base);
    return (__float_as_uint(ma) ^ __float_as_uint(la)) | (__float_as_uint(mb) ^ __float_as_uint(lb));
  }
  // counts one pair in range
  __device__ __forceinline__ void count1(float d2, uint32_t base) const {
    float m, l, x;
    const unsigned long long s2 = f2_pack(sqrt_fast(d2), 0.f);
    f2_unpack(f2_fma_down(s2, hi2, magic2), m, x);
    f2_unpack(f2_fma_down(s2, lo2, magic2), l, x);
    uint32_t b = __float_as_uint(m);
    if (b != __float_as_uint(l) && d2 < sE[b - kMagicBits]) --b;
    red_shared_inc(b * 4u + base);
  }
  // a counted pair that may lie under the edge of its bin: moved to the bin below if it does
  __device__ __forceinline__ void settle(float d2, uint32_t base) const {
    float m, x;
    f2_unpack(f2_fma_down(f2_pack(fminf(sqrt_fast(d2), s_far), 0.f), hi2, magic2), m, x);
    const uint32_t addr = __float_as_uint(m) * 4u + base;
    if (d2 < sE[__float_as_uint(m) - kMagicBits]) {
      red_shared(addr, ~0u);
      red_shared_inc(addr - 4u);
    }
  }
  __device__ __forceinline__ void settle2(unsigned long long d2, uint32_t base) const {
    float da, db;
    f2_unpack(d2, da, db);
    settle(da, base);
    settle(db, base);
  }
};

// ---------------------------------------------------------------------------
// candidates of an item
// ---------------------------------------------------------------------------
// Bounding box of an item's centrals: mid +- half (half rounded up), and ulo .. uhi in cell edges
// widened by `slack`, the rounding of (x - origin) inv_h.
struct ItemBox {
  float mid[3], half[3], ulo[3], uhi[3];
  __device__ __forceinline__ void set(const float4& p, bool valid, const Geo& ng, float slack) {
    const float pc[3] = {p.x, p.y, p.z};
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const float lo = key2f(__reduce_min_sync(0xffffffffu, f2key(valid ? pc[ax] : INFINITY)));
      const float hi = key2f(__reduce_max_sync(0xffffffffu, f2key(valid ? pc[ax] : -INFINITY)));
      mid[ax] = 0.5f * (lo + hi);
      half[ax] = fmaxf(hi - mid[ax], mid[ax] - lo) * 1.000001f + fabsf(mid[ax]) * 2.4e-7f;
      ulo[ax] = (lo - ng.origin[ax]) * ng.inv_h - slack, uhi[ax] = (hi - ng.origin[ax]) * ng.inv_h + slack;
    }
  }
};
__device__ __forceinline__ float item_slack(const Geo& ng) {
  return (float)max(ng.dims[0], max(ng.dims[1], ng.dims[2])) * 5.0e-7f + 1.0e-6f;
}

// Ring of kRing kept candidates as interleaved pairs (xa xb ya yb za zb wa wb): slots [head, tail);
// those from near_to on are beyond every current k-th distance.
struct ItemRing {
  float* bf;
  uint32_t head, tail, near_to;
};

// Walks the candidates of an item in cell c: the records within range of its box (emax with `all`, else
// near_max, which the batches lower as the k-th distances settle) and wanted(w) go through the
// ring, nb at a time to batch(n), n <= nb of the slots from head on (the last batch padded with far
// records).
template <class Batch, class Wanted>
__device__ __forceinline__ void item_scan(const Search& S, const Geo& ng, uint32_t c, const ItemBox& box, ItemRing& R,
                                          uint32_t nb, bool all, float emax, const float& near_max, Batch&& batch,
                                          Wanted&& wanted) {
  const uint32_t lane = threadIdx.x & 31;
  const int n_runs = (int)item_runs(S, ng);
  R.head = R.tail = R.near_to = 0;
  for (int r0 = 0; r0 < n_runs; r0 += 32) {
    // lane r: run r0 + r
    uint32_t rs = 0, rl = 0;
    item_run(S, ng, c, (uint32_t)r0 + lane, box.ulo, box.uhi, (all ? emax : near_max) * 1.0001f * ng.inv_h * ng.inv_h, rs, rl);
    // the runs as one list: lane r holds the position at which run r starts and, less that, its first
    // record; a position's run is found by bisection over the lanes (runs of sparse sets hold a few
    // records each, and a round of 32 loads per run would be mostly idle)
    uint32_t pre = rl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, pre, o);
      if (lane >= (uint32_t)o) pre += y;
    }
    const uint32_t n_list = __shfl_sync(0xffffffffu, pre, 31);
    pre -= rl;
    const uint32_t first = rs - pre;
    auto fetch = [&](uint32_t pos) -> float4 {
      uint32_t r = 0;
#pragma unroll
      for (uint32_t st = 16; st > 0; st >>= 1)
        if (__shfl_sync(0xffffffffu, pre, r + st) <= pos) r += st;
      const uint32_t j = __shfl_sync(0xffffffffu, first, r) + pos;
      return pos < n_list ? __ldg(S.nrec + j) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    // one candidate per lane: into the ring if it is within reach
    auto offer = [&](const float4& q, bool ok) {
      const float ex = fmaxf(fabsf(q.x - box.mid[0]) - box.half[0], 0.f);
      const float ey = fmaxf(fabsf(q.y - box.mid[1]) - box.half[1], 0.f);
      const float ez = fmaxf(fabsf(q.z - box.mid[2]) - box.half[2], 0.f);
      // (the factor covers the rounding of both distances)
      const float e2 = __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, ex * ex)) * 0.99999f;
      const bool in = ok && wanted(q.w), close = in && e2 < near_max;
      const bool keep = all ? in && e2 < emax : close;
      const uint32_t bal = __ballot_sync(0xffffffffu, keep);
      if (keep) {
        const uint32_t slot = (R.tail + __popc(bal & ((1u << lane) - 1u))) & (kRing - 1u);
        float* d = R.bf + (slot >> 1) * 8 + (slot & 1u);
        d[0] = q.x, d[2] = q.y, d[4] = q.z, d[6] = q.w;
      }
      R.tail += __popc(bal);
      if (__any_sync(0xffffffffu, close)) R.near_to = R.tail;
    };
    float4 n0 = fetch(lane), n1 = fetch(32 + lane);
    const bool last = r0 + 32 >= n_runs;
    for (uint32_t o = 0; o < n_list || (last && o == 0u); o += 64) {
      const float4 c0 = n0, c1 = n1;
      n0 = fetch(o + 64 + lane);
      if (o + 96 < n_list) n1 = fetch(o + 96 + lane);
      offer(c0, o + lane < n_list);
      if (o + 32 < n_list) offer(c1, o + 32 + lane < n_list);
      // full batches, and at the very end the rest (one call of batch: the kernels' speed depends on
      // their code size)
      const bool end = last && o + 64 >= n_list;
      while (R.tail - R.head >= nb || (end && R.tail != R.head)) {
        const uint32_t n = min(R.tail - R.head, nb);
        for (uint32_t h = n + lane; h < nb; h += 32) {  // far records to the end of the last batch
          const uint32_t slot = (R.head + h) & (kRing - 1u);
          float* d = R.bf + (slot >> 1) * 8 + (slot & 1u);
          d[0] = INFINITY, d[2] = INFINITY, d[4] = INFINITY, d[6] = __uint_as_float(~0u);
        }
        __syncwarp();
        batch(n);
        R.head += nb;
        __syncwarp();
        if (n < nb) R.tail = R.head;
      }
    }
  }
}

}  // namespace ps
