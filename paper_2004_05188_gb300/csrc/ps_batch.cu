// Batched sweeps: many ROIs and a parameter sweep per ROI in one persistent launch.
//
// The paper's batch queue takes an a-priori list of (statistic, ion-type
// combination, dataset) tasks and evaluates all of them per ROI from one
// neighbour search (Suppl. "Customized user defined batch processing queues"),
// to support parameter-sensitivity studies over many specimens (Results,
// application to experimental datasets).  Here one enumeration per (ROI, cell
// batch) at the largest r_max serves every sweep point exactly:
//   - every k = 1..k_max comes from the per-lane sorted top-k lists (one list per
//     distinct neighbour type set);
//   - every smaller r_max is a prefix of the histograms (the bin edges coincide),
//     and a k-th distance beyond a smaller r_max is "not found" there;
//   - every d_srf threshold t_q is a suffix sum over d_srf classes
//     [t_c, t_{c+1}) accumulated separately;
//   - every type pair comes from the same enumeration (the record carries the
//     ion type; a hit counts for the pairs whose central and neighbour sets hold
//     both ends).
// Work: one queue over all ROIs, items (cell, <= 32 centrals) in ROI order,
// padded per ROI to whole chunks of 16 so a CTA (8 warps, which share out a chunk)
// always works on one ROI and can keep that ROI's RDF counts in shared memory.  Pairs
// of the same neighbour set whose central sets are disjoint are searched together (a
// pass: every lane has one pair); kNN counts go to global memory (one update per
// central, k and pair).
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "ps_internal.cuh"
#include "ps_items.cuh"

namespace ps {

constexpr int kChunk = 16;       // items per CTA fetch

struct BRoi {
  const float4* nrec;
  const uint32_t* nstart;
  const uint32_t* nsub;
  const Geo* ngeo;
  const float4* crec;
  const uint32_t* cstart;
  const uint2* witem;
  const Geo* cgeo;
  const float* dsrf;
  uint32_t cap;  // capacity of witem
};

struct BatchArgs {
  const BRoi* roi;
  const uint32_t* item_off;  // [n_roi + 1] padded exclusive prefix of the ROIs' item counts
  uint32_t n_roi;
  uint32_t* next;            // work counter (chunks of kChunk items)
  int stencil;
  double r0, dr;
  uint32_t n_bins;           // bins at the largest r_max
  uint32_t n_pairs, n_cls, k_max;
  uint32_t n_pass;
  uint32_t pass_pairs[4];    // bit p: pair p is searched in this pass
  uint64_t ctr_mask[4][4];
  Mask nbr[4];               // neighbour set of each pass
  float one;                 // 1.0f, opaque to the compiler (see dist2_x2_fma)
  int8_t row_w[kMaxRuns];
  float cls_min[4];          // d_srf class lower bounds (ascending)
  unsigned long long* acc;   // per ROI accumulators, acc_len each
  uint32_t acc_len;
};

// accumulator layout of one ROI: for each (pair p, class c) a block of
//   rdf[n_bins] | rdf_below | n_central | knn[k_max][n_bins] | knn_below[k_max]
__host__ __device__ inline uint32_t acc_block(uint32_t nb, uint32_t kmax) { return nb + 2 + kmax * nb + kmax; }

__device__ __forceinline__ bool mask_has(const uint64_t* m, uint32_t t) { return (m[t >> 6] >> (t & 63)) & 1ull; }

// One item per warp, its passes one after the other: the candidates of the pass's neighbour set near
// the item's box (item_scan), every in-range pair into the bin row of its central's pair and class,
// those that can still enter a k list into the lane's queue.  DIRECT (r0 = 0): direct bins, an
// increment per test by every lane; otherwise a branch per hit, and the pairs below r0 in bin
// n_bins.  Rows are 32-bit and shared by the CTA: a warp drains them before it has added 2^28 since
// its last drain.  Bound by instruction issue (~34 per 32 tests, k = 20).  24 ROIs (2e6 ions, k = 1 .. 20,
// r_max = 3 nm, 3 pairs, 3 thresholds), kernel: 78 -> 17.4 ms (before: every record of the 125 cells, a
// sorted insertion under a branch per candidate, 64-bit counters; 17.9 with a loop for the bins and
// one for the queue, which computes the near candidates' distances twice).  The queue's stores stand
// after the increments: ahead of them the same loop takes 30 ms.
template <int KMAX, bool DIRECT>
__global__ void __launch_bounds__(256, KMAX <= 20 ? 3 : 2) k_batch_query(const __grid_constant__ BatchArgs a) {
  griddep_wait();
  griddep_launch();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float4 s_buf[8][kRing];
  constexpr uint32_t kRows = (KMAX > (int)kHalf ? KMAX : (int)kHalf) + 1;  // of the insertion queue, and of the lists' merge
  __shared__ uint32_t s_chunk, s_roi, s_next;

  const uint32_t nb = a.n_bins, P = a.n_pairs, C = a.n_cls;
  float* sE = reinterpret_cast<float*>(smem);
  uint32_t* s_rdf = reinterpret_cast<uint32_t*>(sE + nb + 1);  // [P][C][nb + 1]
  uint32_t* s_nc = s_rdf + P * C * (nb + 1);                   // [P][C]
  const uint32_t n_rdf = P * C * (nb + 1);
  for (uint32_t b = threadIdx.x; b <= nb; b += blockDim.x) {
    const double e = __dadd_rn(a.r0, __dmul_rn((double)b, a.dr));
    sE[b] = __double2float_rn(__dmul_rn(e, e));
  }
  for (uint32_t i = threadIdx.x; i < n_rdf + P * C; i += blockDim.x) s_rdf[i] = 0;
  __syncthreads();
  const float Emax = sE[nb], E0 = sE[0], r0f = (float)a.r0, inv_dr = (float)(1.0 / a.dr);
  FastBins fb;
  if (DIRECT) fb.init(nb, a.dr, sE);
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t total = a.item_off[a.n_roi];
  const uint32_t blk = acc_block(nb, a.k_max);
  const unsigned long long one2 = f2_pack(a.one, a.one);
  float* bf = reinterpret_cast<float*>(s_buf[w]);
  float* kq = reinterpret_cast<float*>(s_nc + P * C) + w * kRows * 32;
  const uint32_t q0 = smem_u32(kq + lane), rows = smem_u32(s_rdf) - 4u * kMagicBits;
  uint32_t added = 0;  // bound on this warp's increments since it last drained the rows (uniform)
  int cur = -1;

  // the rows' entries i, i + step, ... to ROI roi's accumulators: bin b (or the count below r0, bin nb)
  // of block pc.  A bin 0 may stand below zero while centrals that met themselves are still to be
  // taken out; the direct bins' bin nb holds the pairs out of range.
  auto drain = [&](int roi, uint32_t i, uint32_t step) {
    unsigned long long* A = a.acc + (size_t)roi * a.acc_len;
    for (; i < n_rdf; i += step) {
      const int32_t v = (int32_t)atomicExch(&s_rdf[i], 0u);
      const uint32_t b = i % (nb + 1);
      if (v && !(DIRECT && b == nb)) atomicAdd(&A[(i / (nb + 1)) * blk + b], (unsigned long long)(long long)v);
    }
  };
  auto flush = [&](int roi) {
    __syncthreads();
    drain(roi, threadIdx.x, blockDim.x);
    unsigned long long* A = a.acc + (size_t)roi * a.acc_len;
    for (uint32_t i = threadIdx.x; i < P * C; i += blockDim.x) {
      if (s_nc[i]) atomicAdd(&A[i * blk + nb + 1], (unsigned long long)s_nc[i]);
      s_nc[i] = 0;
    }
    __syncthreads();
  };

  for (;;) {
    if (threadIdx.x == 0) {
      const uint32_t ch = atomicAdd(a.next, (uint32_t)kChunk);
      s_chunk = ch;
      s_next = 0;
      uint32_t lo = 0, hi = a.n_roi;  // item_off[lo] <= ch < item_off[hi]
      if (ch < total)
        while (hi - lo > 1) {
          const uint32_t mid = (lo + hi) >> 1;
          if (a.item_off[mid] <= ch)
            lo = mid;
          else
            hi = mid;
        }
      s_roi = lo;
    }
    __syncthreads();
    const uint32_t chunk = s_chunk, roi = s_roi;
    if (chunk >= total) break;
    if ((int)roi != cur) {
      if (cur >= 0) flush(cur);
      cur = (int)roi;
    }
    const BRoi R = a.roi[roi];
    const Geo ng = *R.ngeo;
    const Search S{R.nrec, R.nstart, R.nsub, a.stencil, a.row_w};
    const float slack = item_slack(ng);
    const uint32_t n_front = R.cgeo->work_n2, n_items = n_front + R.cgeo->work_n3;
    unsigned long long* A = a.acc + (size_t)roi * a.acc_len;
    for (;;) {
      uint32_t l_item = 0;
      if (lane == 0) l_item = atomicAdd(&s_next, 1u);
      l_item = __shfl_sync(0xffffffffu, l_item, 0);
      if (l_item >= (uint32_t)kChunk) break;
      l_item += chunk - a.item_off[roi];
      if (l_item >= n_items) break;
      const uint2 it = work_item(R.witem, R.cap, n_front, l_item);
      const uint32_t c = it.x, cnt = it.y & 63u, c0 = R.cstart[c] + (it.y >> 6);
      const uint32_t L = item_lanes(cnt), lg = 31u - __clz(L), sub = lane & (L - 1u), ci = lane >> lg;
      const uint32_t nbat = L > 1u ? 64u : 32u;
      float4 rec = make_float4(INFINITY, INFINITY, INFINITY, __uint_as_float(~0u));
      uint32_t cls = 0;
      if (ci < cnt) {
        rec = R.crec[c0 + ci];
        const float di = R.dsrf ? R.dsrf[__float_as_uint(rec.w) >> 8] : INFINITY;
        for (uint32_t q = 1; q < C; ++q)
          if (di >= a.cls_min[q]) cls = q;
      }
      const uint32_t pw = __float_as_uint(rec.w);
#pragma unroll 1
      for (uint32_t ps = 0; ps < a.n_pass; ++ps) {
        // the lane's pair in this pass (the central sets of a pass are disjoint)
        uint32_t pair = ~0u;
        if (ci < cnt)
          for (uint32_t pp = 0; pp < P; ++pp)
            if (((a.pass_pairs[ps] >> pp) & 1u) && mask_has(a.ctr_mask[pp], pw & 0xFFu)) pair = pp;
        const bool valid = pair != ~0u;
        if (__ballot_sync(0xffffffffu, valid) == 0u) continue;
        const uint32_t pc = valid ? pair * C + cls : 0u, row = rows + 4u * pc * (nb + 1);
        // lanes without a central never hit (their distances are infinite or NaN)
        const float4 p = valid ? rec : make_float4(INFINITY, INFINITY, INFINITY, 0.f);
        const unsigned long long px = f2_pack(p.x, p.x), py = f2_pack(p.y, p.y), pz = f2_pack(p.z, p.z);
        ItemBox box;
        box.set(p, valid, ng, slack);
        float top[KMAX];
#pragma unroll
        for (int t = 0; t < KMAX; ++t) top[t] = INFINITY;
        float thr = Emax, near_max = Emax;
        ItemRing ring{bf, 0, 0, 0};
        auto batch = [&](uint32_t n) __attribute__((always_inline)) {
          const ulonglong2* rp = reinterpret_cast<const ulonglong2*>(bf) + (ring.head & (kRing - 1u));
          const uint32_t n_pr = (n + 1) >> 1;
          const bool near = (int32_t)(ring.near_to - ring.head) > 0;
          const ulonglong2 *pa = rp + 2 * sub, *pb = pa + 2 * L;
#pragma unroll 1
          for (uint32_t t0 = 0; t0 < n_pr; t0 += 8 * L) {
            uint32_t qa = q0;
            const uint32_t t1 = min(n_pr, t0 + 8 * L);
#pragma unroll 1
            for (uint32_t t = t0; t < t1; t += 2 * L, pa += 4 * L, pb += 4 * L) {
              const ulonglong2 xy0 = pa[0], xy1 = pb[0], zw0 = pa[1], zw1 = pb[1];
              const unsigned long long d20 = dist2_x2_fma(px, py, pz, xy0.x, xy0.y, zw0.x, one2);
              const unsigned long long d21 = dist2_x2_fma(px, py, pz, xy1.x, xy1.y, zw1.x, one2);
              float d[4], wv[4];
              f2_unpack(d20, d[0], d[1]), f2_unpack(d21, d[2], d[3]);
              f2_unpack(zw0.y, wv[0], wv[1]), f2_unpack(zw1.y, wv[2], wv[3]);
              if (DIRECT) {
                const uint32_t x = fb.count2(d20, row) | fb.count2(d21, row);
                if (__any_sync(0xffffffffu, x != 0u)) {
                  fb.settle2(d20, row);
                  fb.settle2(d21, row);
                }
              } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  if (d[e] < Emax && __float_as_uint(wv[e]) != pw) {
                    const uint32_t bn = d[e] < E0 ? nb : bin_index(d[e], sE, nb, r0f, inv_dr);
                    red_shared_inc(row + 4u * (kMagicBits + bn));
                  }
              }
              if (near) {
#pragma unroll
                for (int e = 0; e < 4; ++e) queue_push_other(qa, d[e], thr, __float_as_uint(wv[e]), pw);
              }
            }
            __syncwarp();
            if (near) {
              const uint32_t qn = (qa - q0) >> 7, m = __reduce_max_sync(0xffffffffu, qn);
#pragma unroll 1
              for (uint32_t q = 0; q < m; ++q)
                if (q < qn) topk_insert(top, queue_at(q0, q));
              float kth = top[KMAX - 1];  // an upper bound of the central's k-th distance in each of its lanes
              for (uint32_t o = 1; o < L; o <<= 1) kth = fminf(kth, __shfl_xor_sync(0xffffffffu, kth, o));
              thr = fminf(kth, Emax);
            }
          }
          if (near) near_max = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(valid ? thr : 0.f)));
          added += 32u * 64u;
          if (added >= (1u << 28) - 4096u) {
            __syncwarp();
            drain(cur, lane, 32);
            added = 0;
          }
        };
        const Mask nm = a.nbr[ps];
        item_scan(S, ng, c, box, ring, nbat, true, Emax, near_max, batch,
                  [&](float qw) { return in_mask(nm, __float_as_uint(qw) & 0xFFu); });
        // the centrals whose type is in the neighbour set met themselves once each, at d2 = 0
        if (DIRECT && valid && sub == 0 && in_mask(nm, pw & 0xFFu) && dist2(p.x, p.y, p.z, p.x, p.y, p.z) == 0.f)
          red_shared(row + 4u * kMagicBits, ~0u);
        // merge the partial lists of the L lanes of each central (disjoint candidate subsets)
        for (uint32_t o = 1; o < L; o <<= 1) {
          __syncwarp();
#pragma unroll
          for (int t = 0; t < KMAX; ++t) kq[t * 32 + lane] = top[t];
          __syncwarp();
          const float* ot = kq + (lane ^ o);
#pragma unroll 1
          for (int t = 0; t < KMAX; ++t) {
            const float v = ot[t * 32];
            if (!(v < top[KMAX - 1])) break;  // the partner's list is sorted
            topk_insert(top, v);
          }
        }
        __syncwarp();
        if (valid && sub == 0) {
          atomicAdd(&s_nc[pc], 1u);
#pragma unroll
          for (int t = 0; t < KMAX; ++t) {
            const float D = top[t];
            if ((uint32_t)t >= a.k_max || !(D < Emax)) break;  // not found: derived from the counts
            if (D < E0)
              atomicAdd(&A[pc * blk + nb + 2 + a.k_max * nb + t], 1ull);
            else
              atomicAdd(&A[pc * blk + nb + 2 + t * nb + bin_index(D, sE, nb, r0f, inv_dr)], 1ull);
          }
        }
      }
    }
    __syncthreads();
  }
  if (cur >= 0) flush(cur);
}

// Padded item offsets: item_off[r] = sum over ROIs before r of ceil(items / kChunk) * kChunk.
__global__ void k_batch_offsets(const BRoi* __restrict__ roi, uint32_t n_roi, uint32_t* __restrict__ item_off,
                                uint32_t* __restrict__ next) {
  griddep_wait();
  griddep_launch();
  if (threadIdx.x == 0) {
    uint32_t acc = 0;
    for (uint32_t r = 0; r < n_roi; ++r) {
      item_off[r] = acc;
      const uint32_t n = roi[r].cgeo->work_n2 + roi[r].cgeo->work_n3;
      acc += (n + kChunk - 1) / kChunk * kChunk;
    }
    item_off[n_roi] = acc;
    *next = 0;
  }
}

// Expands the class accumulators into one result per (ROI, pair, r_max, d_srf threshold),
// in the layout of ps_spatstat: rdf[n_bins] | knn[k_max][n_bins] | meta[PS_META_LEN(k_max)].
__global__ void __launch_bounds__(256) k_batch_expand(const unsigned long long* __restrict__ acc, uint32_t acc_len,
                                                      uint32_t nb, uint32_t P, uint32_t C, uint32_t kmax, uint32_t R,
                                                      const uint32_t* __restrict__ rbins, unsigned long long* out) {
  griddep_wait();
  griddep_launch();
  const uint32_t rec = nb + kmax * nb + PS_META_LEN(kmax);
  const uint32_t blk = acc_block(nb, kmax);
  const uint32_t id = blockIdx.x;  // ((roi * P + p) * R + r) * C + q
  const uint32_t q = id % C, r = (id / C) % R, pp = (id / (C * R)) % P, roi = id / (C * R * P);
  const unsigned long long* A = acc + (size_t)roi * acc_len + (size_t)pp * C * blk;
  unsigned long long* O = out + (size_t)id * rec;
  const uint32_t nbr_ = rbins[r];
  __shared__ unsigned long long s_red[8];
  // rdf
  unsigned long long binned = 0;
  for (uint32_t b = threadIdx.x; b < nb; b += blockDim.x) {
    unsigned long long v = 0;
    if (b < nbr_)
      for (uint32_t c = q; c < C; ++c) v += A[c * blk + b];
    O[b] = v;
    binned += v;
  }
  // knn
  for (uint32_t i = threadIdx.x; i < kmax * nb; i += blockDim.x) {
    const uint32_t k = i / nb, b = i % nb;
    unsigned long long v = 0;
    if (b < nbr_)
      for (uint32_t c = q; c < C; ++c) v += A[c * blk + nb + 2 + k * nb + b];
    O[nb + i] = v;
  }
  for (int o = 16; o > 0; o >>= 1) binned += __shfl_xor_sync(0xffffffffu, binned, o);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = binned;
  __syncthreads();
  unsigned long long* M = O + nb + kmax * nb;
  if (threadIdx.x == 0) {
    unsigned long long tb = 0, nc = 0, below = 0;
    for (uint32_t i = 0; i < (blockDim.x >> 5); ++i) tb += s_red[i];
    for (uint32_t c = q; c < C; ++c) nc += A[c * blk + nb + 1], below += A[c * blk + nb];
    M[PS_META_N_CENTRAL] = nc;
    M[PS_META_N_PAIRS] = tb;
    M[PS_META_N_BELOW] = below;
    M[PS_META_STATUS] = 0;
  }
  // per k: not found = centrals - found in range - below range
  for (uint32_t k = threadIdx.x; k < kmax; k += blockDim.x) {
    unsigned long long nc = 0, found = 0, kb = 0;
    for (uint32_t c = q; c < C; ++c) {
      nc += A[c * blk + nb + 1];
      kb += A[c * blk + nb + 2 + kmax * nb + k];
      for (uint32_t b = 0; b < nbr_; ++b) found += A[c * blk + nb + 2 + k * nb + b];
    }
    M[PS_META_HEAD + 2 * k] = nc - found - kb;
    M[PS_META_HEAD + 2 * k + 1] = kb;
  }
}

}  // namespace ps

struct ps_batch {
  ps_sweep sw;
  std::vector<ps_dataset> ds;
  std::vector<ps_grid*> grids;
  ps::BRoi* d_roi = nullptr;
  uint32_t* d_item_off = nullptr;
  uint32_t* d_next = nullptr;
  uint32_t* d_rbins = nullptr;
  unsigned long long* d_acc = nullptr;
  uint32_t acc_len = 0, n_pass = 0, pass_pairs[4] = {0, 0, 0, 0};
  uint64_t pass_nbr[4][4];
  uint64_t nbr_union[4], ctr_union[4];
  float r_cut = 0.f;
};

using namespace ps;

template <int KMAX, bool DIRECT>
static int launch_batch(const BatchArgs& a, int sms, cudaStream_t st) {
  auto kern = k_batch_query<KMAX, DIRECT>;
  // edges, bin rows, central counts, insertion queues
  const uint32_t smem = (a.n_bins + 1) * 4 + a.n_pairs * a.n_cls * ((a.n_bins + 1) * 4 + 4) +
                        8u * ((KMAX > (int)kHalf ? KMAX : (int)kHalf) + 1) * 32u * 4u;
  PS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  PS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, smem));
  if (per_sm < 1) return fail(PS_ERR_UNSUPPORTED, "batched query kernel does not fit on an SM");
  PS_LAUNCH(PS_KID_BATCH, st, PS_CUDA(launch_pdl(kern, sms * per_sm, 256, smem, st, a)));
  PS_CUDA(cudaGetLastError());
  return PS_OK;
}

template <bool DIRECT>
static int dispatch_batch(const BatchArgs& a, int sms, cudaStream_t st) {
  return a.k_max <= 8    ? launch_batch<8, DIRECT>(a, sms, st)
         : a.k_max <= 16 ? launch_batch<16, DIRECT>(a, sms, st)
         : a.k_max <= 20 ? launch_batch<20, DIRECT>(a, sms, st)
                         : launch_batch<32, DIRECT>(a, sms, st);
}

extern "C" {

int ps_batch_create(const ps_dataset* ds, int n_ds, const ps_sweep* sw, ps_batch** out) {
  if (!out || !ds || !sw || n_ds < 1) return fail(PS_ERR_INVALID_ARG, "ps_batch_create: NULL argument or n_ds < 1");
  *out = nullptr;
  if (sw->struct_size < sizeof(ps_sweep)) return fail(PS_ERR_INVALID_ARG, "ps_batch_create: sweep struct_size");
  const ps_sweep& s = *sw;
  if (!(s.bins.dr > 0.0) || !(s.bins.r0 >= 0.0) || s.bins.n_bins < 1 || s.bins.n_bins > 512)
    return fail(PS_ERR_UNSUPPORTED, "ps_batch_create: need dr > 0, r0 >= 0 and 1..512 bins");
  if (s.n_rmax < 1 || s.n_rmax > 4 || s.n_dsrf < 1 || s.n_dsrf > 4 || s.n_pairs < 1 || s.n_pairs > 4)
    return fail(PS_ERR_UNSUPPORTED, "ps_batch_create: 1..4 r_max values, d_srf thresholds and type pairs");
  if (s.k_max < 1 || s.k_max > PS_K_MAX) return fail(PS_ERR_UNSUPPORTED, "ps_batch_create: k_max in 1..32");
  for (uint32_t r = 0; r < s.n_rmax; ++r)
    if (s.rmax_bins[r] < 1 || s.rmax_bins[r] > s.bins.n_bins || (r && s.rmax_bins[r] <= s.rmax_bins[r - 1]))
      return fail(PS_ERR_INVALID_ARG, "ps_batch_create: rmax_bins must ascend within 1..n_bins");
  if (s.rmax_bins[s.n_rmax - 1] != s.bins.n_bins)
    return fail(PS_ERR_INVALID_ARG, "ps_batch_create: the last r_max must be bins.n_bins");
  for (uint32_t q = 0; q < s.n_dsrf; ++q)
    if (std::isnan(s.dsrf_min[q]) || (q && !(s.dsrf_min[q] > s.dsrf_min[q - 1])))
      return fail(PS_ERR_INVALID_ARG, "ps_batch_create: dsrf_min must ascend");
  if (s.cell_scale != 0.0f && !(s.cell_scale >= 0.5f))
    return fail(PS_ERR_UNSUPPORTED, "ps_batch_create: cell_scale must be 0 (default) or >= 0.5");
  const uint32_t smem_rdf = s.n_pairs * s.n_dsrf * s.bins.n_bins;
  if (smem_rdf > 8192) return fail(PS_ERR_UNSUPPORTED, "ps_batch_create: pairs x thresholds x bins > 8192");
  ps_batch* b = new (std::nothrow) ps_batch();
  if (!b) return fail(PS_ERR_OOM, "host allocation failed");
  b->sw = s;
  // at most two distinct neighbour sets; passes: pairs of one neighbour set with disjoint central sets
  uint32_t n_sets = 0;
  for (uint32_t p = 0; p < s.n_pairs; ++p) {
    bool known = false;
    for (uint32_t q = 0; q < p; ++q) known = known || !memcmp(s.nbr_mask[q], s.nbr_mask[p], sizeof(uint64_t) * 4);
    n_sets += known ? 0u : 1u;
    if (n_sets > 2) {
      delete b;
      return fail(PS_ERR_UNSUPPORTED, "ps_batch_create: at most 2 distinct neighbour type sets");
    }
    uint32_t ps = 0;
    for (; ps < b->n_pass; ++ps) {
      bool fits = !memcmp(b->pass_nbr[ps], s.nbr_mask[p], sizeof(uint64_t) * 4);
      for (uint32_t q = 0; q < p; ++q)
        if ((b->pass_pairs[ps] >> q) & 1u)
          for (int w = 0; w < 4; ++w) fits = fits && (s.ctr_mask[q][w] & s.ctr_mask[p][w]) == 0;
      if (fits) break;
    }
    if (ps == b->n_pass) memcpy(b->pass_nbr[b->n_pass++], s.nbr_mask[p], sizeof(uint64_t) * 4);
    b->pass_pairs[ps] |= 1u << p;
  }
  for (int w = 0; w < 4; ++w) {
    b->nbr_union[w] = b->ctr_union[w] = 0;
    for (uint32_t p = 0; p < s.n_pairs; ++p) b->nbr_union[w] |= s.nbr_mask[p][w], b->ctr_union[w] |= s.ctr_mask[p][w];
  }
  const double stop = s.bins.r0 + (double)s.bins.n_bins * s.bins.dr;
  b->r_cut = (float)(stop * (1.0 + 1e-6));
  b->acc_len = s.n_pairs * s.n_dsrf * acc_block(s.bins.n_bins, s.k_max);
  ps_grid_opts go;
  memset(&go, 0, sizeof(go));
  go.struct_size = sizeof(go);
  go.cell_scale = s.cell_scale;
  int rc = PS_OK;
  for (int i = 0; i < n_ds && rc == PS_OK; ++i) {
    if (ds[i].n < 0 || ds[i].n >= (1 << 24)) rc = fail(PS_ERR_UNSUPPORTED, "ps_batch_create: ROIs hold < 2^24 ions");
    if (rc == PS_OK && ds[i].n > 0 && (!ds[i].xyz || !ds[i].type))
      rc = fail(PS_ERR_INVALID_ARG, "ps_batch_create: dataset xyz/type is NULL");
    if (rc) break;
    b->ds.push_back(ds[i]);
    ps_grid* g = nullptr;
    rc = ps_grid_create(ds[i].n, &go, &g);
    if (rc == PS_OK) {
      g->pack_type = true;
      b->grids.push_back(g);
    }
  }
  auto cleanup = [&](int code) {
    for (ps_grid* g : b->grids) ps_grid_destroy(g);
    dev_free(b->d_roi);
    dev_free(b->d_item_off);
    dev_free(b->d_next);
    dev_free(b->d_rbins);
    dev_free(b->d_acc);
    delete b;
    return code;
  };
  if (rc) return cleanup(rc);
  cudaError_t e = dev_malloc((void**)&b->d_roi, sizeof(BRoi) * n_ds);
  if (e == cudaSuccess) e = dev_malloc((void**)&b->d_item_off, sizeof(uint32_t) * (n_ds + 1));
  if (e == cudaSuccess) e = dev_malloc((void**)&b->d_next, sizeof(uint32_t));
  if (e == cudaSuccess) e = dev_malloc((void**)&b->d_rbins, sizeof(uint32_t) * 4);
  if (e == cudaSuccess) e = dev_malloc((void**)&b->d_acc, sizeof(unsigned long long) * (size_t)b->acc_len * n_ds);
  if (e != cudaSuccess) return cleanup(cuda_fail(e, "cudaMalloc(batch)"));
  std::vector<BRoi> h(n_ds);
  for (int i = 0; i < n_ds; ++i) {
    ps_grid* g = b->grids[i];
    h[i] = BRoi{g->nbr.rec, g->nbr.start, g->nbr.count, g->nbr.geo, g->ctr.rec, g->ctr.start,
                g->ctr.witem, g->ctr.geo,  ds[i].dsrf, g->item_cap};
  }
  e = cudaMemcpy(b->d_roi, h.data(), sizeof(BRoi) * n_ds, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(b->d_rbins, s.rmax_bins, sizeof(uint32_t) * 4, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cleanup(cuda_fail(e, "cudaMemcpy(batch)"));
  *out = b;
  return PS_OK;
}

int ps_batch_destroy(ps_batch* b) {
  if (!b) return PS_OK;
  cudaDeviceSynchronize();
  for (ps_grid* g : b->grids) ps_grid_destroy(g);
  dev_free(b->d_roi);
  dev_free(b->d_item_off);
  dev_free(b->d_next);
  dev_free(b->d_rbins);
  dev_free(b->d_acc);
  delete b;
  return PS_OK;
}

int64_t ps_batch_out_len(const ps_batch* b) {
  if (!b) return -1;
  const ps_sweep& s = b->sw;
  const int64_t rec = s.bins.n_bins + (int64_t)s.k_max * s.bins.n_bins + PS_META_LEN(s.k_max);
  return (int64_t)b->ds.size() * s.n_pairs * s.n_rmax * s.n_dsrf * rec;
}

int ps_batch_run(ps_batch* b, uint64_t* d_out, void* stream) {
  if (!b || !d_out) return fail(PS_ERR_INVALID_ARG, "ps_batch_run: NULL argument");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const ps_sweep& s = b->sw;
  const uint32_t n_roi = (uint32_t)b->ds.size();
  // grids and central lists of every ROI (records carry the ion type)
  for (uint32_t i = 0; i < n_roi; ++i) {
    int rc = ps_grid_build(b->grids[i], b->ds[i].xyz, b->ds[i].type, b->ds[i].n, b->nbr_union, b->r_cut, stream);
    if (rc) return rc;
    rc = build_central_list(b->grids[i], b->ds[i].dsrf, b->ctr_union, s.dsrf_min[0], st);
    if (rc) return rc;
  }
  PS_CUDA(cudaMemsetAsync(b->d_acc, 0, sizeof(unsigned long long) * (size_t)b->acc_len * n_roi, st));
  PS_LAUNCH(PS_KID_BATCH, st, PS_CUDA(launch_pdl(k_batch_offsets, 1, 32, 0, st, b->d_roi, n_roi, b->d_item_off, b->d_next)));
  BatchArgs a;
  memset(&a, 0, sizeof(a));
  a.roi = b->d_roi;
  a.item_off = b->d_item_off;
  a.n_roi = n_roi;
  a.next = b->d_next;
  a.stencil = b->grids[0]->stencil;
  a.r0 = s.bins.r0;
  a.dr = s.bins.dr;
  a.n_bins = s.bins.n_bins;
  a.n_pairs = s.n_pairs;
  a.n_cls = s.n_dsrf;
  a.k_max = s.k_max;
  a.n_pass = b->n_pass;
  a.one = 1.0f;
  row_widths(b->grids[0]->stencil, b->grids[0]->cell_scale, a.row_w);
  for (uint32_t p = 0; p < s.n_pairs; ++p)
    for (int w = 0; w < 4; ++w) a.ctr_mask[p][w] = s.ctr_mask[p][w];
  for (uint32_t ps = 0; ps < b->n_pass; ++ps) {
    a.pass_pairs[ps] = b->pass_pairs[ps];
    for (int w = 0; w < 4; ++w) a.nbr[ps].w[w] = b->pass_nbr[ps][w];
  }
  for (uint32_t q = 0; q < s.n_dsrf; ++q) a.cls_min[q] = s.dsrf_min[q];
  a.acc = b->d_acc;
  a.acc_len = b->acc_len;
  const int sms = b->grids[0]->num_sms;
  // direct bins: r0 = 0 and edges far from the limits of float32 (as the exact query; at most 512 bins)
  const double stop = (double)s.bins.n_bins * s.bins.dr;
  const bool direct = s.bins.r0 == 0.0 && s.bins.dr > 1e-15 && stop < 1e15;
  const int rc = direct ? dispatch_batch<true>(a, sms, st) : dispatch_batch<false>(a, sms, st);
  if (rc) return rc;
  const uint32_t n_out = n_roi * s.n_pairs * s.n_rmax * s.n_dsrf;
  PS_LAUNCH(PS_KID_BATCH, st,
            PS_CUDA(launch_pdl(k_batch_expand, n_out, 256, 0, st, b->d_acc, b->acc_len, s.bins.n_bins, s.n_pairs, s.n_dsrf, s.k_max,
                                                  s.n_rmax, b->d_rbins, reinterpret_cast<unsigned long long*>(d_out))));
  PS_CUDA(cudaGetLastError());
  return PS_OK;
}

}  // extern "C"
