// Gaussian-smoothed RDF and its adjoint (the differentiable form).
//
// The paper bins pair distances with rectangular transfer functions (Methods,
// "Descriptive, two-point spatial statistics, and clustering").  Here every
// pair spreads a Gaussian of width sigma that is integrated over each bin:
//   u_ij = s * |x_j - x_i|,  K_b(u) = Phi((e_{b+1} - u)/sigma) - Phi((e_b - u)/sigma)
//   h[b] = sum over central i, neighbour j != i with u_ij < stop + 6 sigma of K_b(u_ij)
// and, for an upstream gradient G[b] = dL/dh[b],
//   W(u) = dL/du = sum_b G[b] K_b'(u),
//   dL/dx_i += W s (x_i - x_j)/d,  dL/dx_j -= W s (x_i - x_j)/d,  dL/ds += W d.
//
// Forward: each pair deposits u on a fine grid of width w (<= sigma/40) as three
// moments about the fine-bin centre c_m (count, sum of delta, sum of delta^2);
// a finalize kernel evaluates h[b] = sum_m M0 K_b(c_m) + M1 K_b'(c_m) + M2/2 K_b''(c_m)
// in FP64 over all bins.  The remainder is third order in delta (|delta| <= w/2)
// and odd about c_m, i.e. a relative error ~1e-7 that averages out.
// Adjoint: W, W', W'' are tabulated on the same fine grid (FP64, stored as
// float) and evaluated per pair by the same second-order expansion.  Pairs are
// recomputed, never stored.  Where the centrals are neighbour records, forward and
// adjoint meet every unordered pair once (sweep_pairs), weighted by the central
// flags of both ends, and the adjoint adds a pair's force at both of them.
// Otherwise the forward has one lane per central, and the adjoint's pass A (one
// lane per central) writes and pass B (one lane per neighbour, candidates =
// centrals) adds: each gradient then has one owner.  dL/ds sums W d over the
// pairs, once per central end.
#include <cmath>
#include <cstring>

#include "ps_internal.cuh"
#include "ps_sweep.cuh"

namespace ps {

constexpr int kSoftRuns = 49;  // (2 * stencil + 1)^2 for stencil <= 3

struct SoftArgs {
  // owners (one lane per record) and their work items
  const float4* orec;
  const uint32_t* ostart;
  const uint2* oitem;
  uint32_t ocap;    // capacity of oitem
  Geo* ogeo;        // owner list counters (work_n2 + work_n3 items, work_next2)
  // candidates and their cell starts (same geometry as the owners)
  const float4* nrec;
  const uint32_t* nstart;
  const Geo* ngeo;  // geometry
  int stencil;
  float scale, sigma, rc;  // rc = stop + 6 sigma (scaled units)
  float rc2u;              // (rc / scale)^2 * (1 + 1e-6): cheap prefilter on d2
  float w, inv_w;          // fine grid
  uint32_t n_fine;
  // forward outputs
  unsigned long long* M0;
  double* M1;
  double* M2;
  // adjoint
  const float4* T;         // [n_fine]: W, W', W'' / 2 at the fine-bin centres, times the scale
  float* grad;             // [n][3]
  double* grad_s;
  int pass_b;              // 0: owners are centrals (write), 1: owners are neighbours (add, sign flipped)
};

__device__ __forceinline__ void soft_run(const SoftArgs& a, const Geo& ng, uint32_t c, uint32_t r, uint32_t& src,
                                         uint32_t& len) {
  const int s = a.stencil, wd = 2 * s + 1;
  const uint32_t cx = c % ng.dims[0], cy = (c / ng.dims[0]) % ng.dims[1], cz = c / (ng.dims[0] * ng.dims[1]);
  const int y = (int)cy + (int)(r % wd) - s, z = (int)cz + (int)(r / wd) - s;
  src = 0;
  len = 0;
  if ((int)r < wd * wd && y >= 0 && z >= 0 && y < (int)ng.dims[1] && z < (int)ng.dims[2]) {
    const uint32_t xlo = cx >= (uint32_t)s ? cx - s : 0;
    const uint32_t xhi = cx + s < ng.dims[0] ? cx + s : ng.dims[0] - 1;
    const uint32_t row = ((uint32_t)z * ng.dims[1] + (uint32_t)y) * ng.dims[0];
    src = a.nstart[row + xlo];
    len = a.nstart[row + xhi + 1] - src;
  }
}

// Iterates the items of the owner list (the centrals; candidates: their full stencil of
// neighbours, whose staged .w is the ion index so that the owner itself is skipped) with the
// candidates staged 32 at a time as interleaved pairs (xa xb ya yb za zb wa wb) and tested two at
// a time with packed float32 math; the in-range pairs of every half-batch of 16 candidates go to
// a warp list that all lanes then process: hit(d2) for each.  item_hook(cnt, n_cand) runs once
// per item.
template <class H, class I>
__device__ __forceinline__ void soft_items_listed(const SoftArgs& a, float* bf, uint32_t* rsrc, uint32_t* rpre,
                                                  float* wlist, H&& hit, I&& item_hook) {
  const uint32_t lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
  const Geo ng = *a.ngeo;
  const uint32_t n_front = a.ogeo->work_n2, n_items = n_front + a.ogeo->work_n3;
  const int s = a.stencil, wd = 2 * s + 1;
  const int n_runs = wd * wd;
  for (;;) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(&a.ogeo->work_next2, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_items) break;
    const uint2 it = work_item(a.oitem, a.ocap, n_front, item);
    const uint32_t c = it.x, first = it.y >> 6, cnt = it.y & 63u;
    const uint32_t c0 = a.ostart[c] + first;
    const uint32_t n_cand = run_table(lane, n_runs, rsrc, rpre, [&](uint32_t r, uint32_t& src, uint32_t& len) {
      soft_run(a, ng, c, r, src, len);
    });
    item_hook(cnt, n_cand);
    const bool valid = lane < cnt;
    float4 p = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    float emax = -INFINITY;
    uint32_t pidx = ~0u;
    if (valid) {
      p = a.orec[c0 + lane];
      pidx = __float_as_uint(p.w);
      emax = a.rc2u;
    }
    const unsigned long long px = f2_pack(p.x, p.x), py = f2_pack(p.y, p.y), pz = f2_pack(p.z, p.z);
    int rr = 0;
    auto fetch = [&](uint32_t pos) -> float4 {
      if (pos >= n_cand) return make_float4(INFINITY, INFINITY, INFINITY, __uint_as_float(~0u));
      while (pos >= rpre[rr + 1]) ++rr;
      return __ldg(a.nrec + rsrc[rr] + (pos - rpre[rr]));
    };
    float4 nxt = fetch(lane);
    for (uint32_t b = 0; b < n_cand; b += 32) {
      __syncwarp();
      {
        float* d = bf + (lane >> 1) * 8 + (lane & 1);
        d[0] = nxt.x, d[2] = nxt.y, d[4] = nxt.z, d[6] = nxt.w;
      }
      __syncwarp();
      nxt = fetch(b + 32 + lane);
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        uint32_t nh = 0;
#pragma unroll 2
        for (uint32_t u = 0; u < 8; ++u) {
          const uint32_t t = 8 * half + u;
          const ulonglong2 xy = reinterpret_cast<const ulonglong2*>(bf)[2 * t];
          const ulonglong2 zw = reinterpret_cast<const ulonglong2*>(bf)[2 * t + 1];
          float d2a, d2b, wa, wb;
          dist2_x2(px, py, pz, xy.x, xy.y, zw.x, d2a, d2b);
          f2_unpack(zw.y, wa, wb);
          const bool ha = d2a < emax && __float_as_uint(wa) != pidx;
          const bool hb = d2b < emax && __float_as_uint(wb) != pidx;
          const uint32_t ba = __ballot_sync(0xffffffffu, ha);
          wlist[ha ? nh + __popc(ba & lt) : 512 + lane] = d2a;
          nh += __popc(ba);
          const uint32_t bb = __ballot_sync(0xffffffffu, hb);
          wlist[hb ? nh + __popc(bb & lt) : 512 + lane] = d2b;
          nh += __popc(bb);
        }
        __syncwarp();
        for (uint32_t h = lane; h < nh; h += 32) hit(wlist[h]);
        __syncwarp();
      }
    }
  }
}

// Same iteration for the adjoint, where every in-range pair updates its owner lane's
// accumulators: f(p, qx, qy, qz, d2) under a branch per candidate (queueing the pairs first
// measured slower).  begin_owner() / end_owner(valid, p) bracket each owner.
template <class F, class B, class E>
__device__ __forceinline__ void soft_items_owned(const SoftArgs& a, float* bf, uint32_t* rsrc, uint32_t* rpre,
                                                 F&& f, B&& begin_owner, E&& end_owner) {
  const uint32_t lane = threadIdx.x & 31;
  const Geo ng = *a.ngeo;
  const uint32_t n_front = a.ogeo->work_n2, n_items = n_front + a.ogeo->work_n3;
  const int n_runs = (2 * a.stencil + 1) * (2 * a.stencil + 1);
  for (;;) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(&a.ogeo->work_next2, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_items) break;
    const uint2 it = work_item(a.oitem, a.ocap, n_front, item);
    const uint32_t c = it.x, first = it.y >> 6, cnt = it.y & 63u;
    const uint32_t c0 = a.ostart[c] + first;
    const uint32_t n_cand = run_table(lane, n_runs, rsrc, rpre, [&](uint32_t r, uint32_t& src, uint32_t& len) {
      soft_run(a, ng, c, r, src, len);
    });
    const bool valid = lane < cnt;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) p = a.orec[c0 + lane];
    const uint32_t pidx = valid ? __float_as_uint(p.w) : ~0u;
    const float emax = valid ? a.rc2u : -INFINITY;
    const unsigned long long px = f2_pack(p.x, p.x), py = f2_pack(p.y, p.y), pz = f2_pack(p.z, p.z);
    begin_owner();
    int rr = 0;
    auto fetch = [&](uint32_t pos) -> float4 {
      if (pos >= n_cand) return make_float4(INFINITY, INFINITY, INFINITY, __uint_as_float(~0u));
      while (pos >= rpre[rr + 1]) ++rr;
      return __ldg(a.nrec + rsrc[rr] + (pos - rpre[rr]));
    };
    auto hit = [&](float d2, float w) -> bool { return d2 < emax && __float_as_uint(w) != pidx; };
    float4 nxt = fetch(lane);
    for (uint32_t b = 0; b < n_cand; b += 32) {
      __syncwarp();
      {
        float* d = bf + (lane >> 1) * 8 + (lane & 1);
        d[0] = nxt.x, d[2] = nxt.y, d[4] = nxt.z, d[6] = nxt.w;
      }
      __syncwarp();
      nxt = fetch(b + 32 + lane);
#pragma unroll 2
      for (uint32_t t = 0; t < 16; ++t) {
        const ulonglong2 xy = reinterpret_cast<const ulonglong2*>(bf)[2 * t];
        const ulonglong2 zw = reinterpret_cast<const ulonglong2*>(bf)[2 * t + 1];
        float d2a, d2b, xa, xb, ya, yb, za, zb, wa, wb;
        dist2_x2(px, py, pz, xy.x, xy.y, zw.x, d2a, d2b);
        f2_unpack(zw.y, wa, wb);
        if (hit(d2a, wa)) {
          f2_unpack(xy.x, xa, xb), f2_unpack(xy.y, ya, yb), f2_unpack(zw.x, za, zb);
          f(p, xa, ya, za, d2a);
        }
        if (hit(d2b, wb)) {
          f2_unpack(xy.x, xa, xb), f2_unpack(xy.y, ya, yb), f2_unpack(zw.x, za, zb);
          f(p, xb, yb, zb, d2b);
        }
      }
    }
    end_owner(valid, p);
  }
}

// ---------------------------------------------------------------------------
// forward: fine-grid moments
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_soft_fwd(const SoftArgs a) {
  griddep_wait();
  griddep_launch();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float4 s_grp[8][64];        // per warp: staged records (the cell's, or a batch of candidates)
  __shared__ float s_hits[8][512 + 32];  // per warp: one half-batch's in-range d2 + a trash row
  __shared__ uint32_t s_rsrc[8][kSoftRuns], s_rpre[8][kSoftRuns + 1];
  // 32-bit counts per CTA; a warp whose item could push the CTA past 2^31 pairs writes to global
  // instead
  uint32_t* sM0 = reinterpret_cast<uint32_t*>(smem);
  float* sM1 = reinterpret_cast<float*>(smem + a.n_fine * 4);
  float* sM2 = reinterpret_cast<float*>(smem + a.n_fine * 8);
  __shared__ unsigned long long s_pairs;
  for (uint32_t m = threadIdx.x; m < a.n_fine; m += blockDim.x) sM0[m] = 0, sM1[m] = 0.f, sM2[m] = 0.f;
  if (threadIdx.x == 0) s_pairs = 0;
  __syncthreads();
  bool glob = false;
  const uint32_t w = threadIdx.x >> 5;
  const float s = a.scale, inv_w = a.inv_w, wf = a.w, rc = a.rc;
  const uint32_t nf = a.n_fine;
  // one pair at distance sqrt(d2) into the fine-grid moments
  auto pair = [&](float d2) {
    const float u = s * (d2 > 0.f ? d2 * rsqrtf(d2) : 0.f);
    if (!(u < rc)) return;
    uint32_t m = (uint32_t)(u * inv_w);
    m = m < nf ? m : nf - 1;
    const float delta = u - ((float)m + 0.5f) * wf;
    if (glob) {
      atomicAdd(&a.M0[m], 1ull);
      atomicAdd(&a.M1[m], (double)delta);
      atomicAdd(&a.M2[m], (double)delta * (double)delta);
    } else {
      atomicAdd(&sM0[m], 1u);
      atomicAdd(&sM1[m], delta);
      atomicAdd(&sM2[m], delta * delta);
    }
  };
  auto bound = [&](uint32_t cnt, uint32_t n_cand) {
    unsigned long long old = 0;
    const unsigned long long inc = (unsigned long long)cnt * n_cand;
    if ((threadIdx.x & 31) == 0) old = atomicAdd(&s_pairs, inc);
    old = __shfl_sync(0xffffffffu, old, 0);
    glob = old + inc >= (1ull << 31);
  };
  soft_items_listed(a, reinterpret_cast<float*>(s_grp[w]), s_rsrc[w], s_rpre[w], s_hits[w], pair, bound);
  __syncthreads();
  for (uint32_t m = threadIdx.x; m < nf; m += blockDim.x) {
    if (sM0[m]) {
      atomicAdd(&a.M0[m], (unsigned long long)sM0[m]);
      atomicAdd(&a.M1[m], (double)sM1[m]);
      atomicAdd(&a.M2[m], (double)sM2[m]);
    }
  }
}

// Pairs of the sweep as packed distances: the range test is u < rc (u = scale * distance), the fine
// bin floor(u / w).  The bin centres (m + 1/2) w are exact in float32 (see soft_width), so that the remainder
// u - (m + 1/2) w carries only the rounding of u.
struct SoftFine {
  unsigned long long scale2, inv_w2, w2, half_w2, magic2;
  __device__ explicit SoftFine(const SoftArgs& a) {
    scale2 = f2_pack(a.scale, a.scale);
    inv_w2 = f2_pack(a.inv_w, a.inv_w);
    w2 = f2_pack(a.w, a.w);
    half_w2 = f2_pack(0.5f * a.w, 0.5f * a.w);
    magic2 = f2_pack(kMagic, kMagic);
  }
  // u -> floor(u / w) in the low bits of m, and the remainder about the bin centre
  __device__ __forceinline__ void split(unsigned long long u2, unsigned long long& m2, unsigned long long& delta2) const {
    m2 = f2_fma_down(u2, inv_w2, magic2);
    delta2 = f2_sub(u2, f2_fma(f2_sub(m2, magic2), w2, half_w2));
  }
};

// (subnormal squared distances count as 0, i.e. as coincident ions)
__device__ __forceinline__ float rsqrt_fast(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ unsigned long long soft_d2(unsigned long long dx, unsigned long long dy,
                                                      unsigned long long dz) {
  return f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
}

// The forward's moments of a fine bin in integers: the weights, the remainders in units of w / 2^18 and their
// squares in units of w^2 / 2^18.  The sums do not round, and a unit of the remainders is at most float32's step
// of u from the 32nd bin on (u = 0.8 sigma), so that they hold what the distance does; where nearer pairs
// are not rare (LOW, fewer than 512 fine bins: sigma above a sixth of the range) the remainders take units of
// w / 2^22 in two words, the low kSoftLow bits apart.  (Units of w / 2^13 showed wherever the sums have few or
// equal pairs: a lattice of 343 ions, a = 0.286 and sigma = 0.2 nm, 1.6e-7 of h against FP64, float32 sums 1.0e-7,
// now 4e-8; 50 ions, sigma = 0.5 nm, 3.7e-8, 2.0e-8 and 7e-9.)
// Integer shared-memory atomics run at the rate of the plain count (measured, 2 of 5 lanes active at random
// places, cycles per warp and SM: one count 4.5, three integers 5.4, a count and two floats 12.1).  A bin's sums
// stay inside 32 bits while its weight is below 2^14: the addition of the weight returns the bin's weight
// before it, and a warp that meets one of 2^12 in its turn of 4 records drains all bins to the global
// moments.  A turn adds at most 512 to a bin, and a warp that has not met the limit in one turn meets it in the
// next: below 2^12 + 8 * 2 * 512.
constexpr float kSoftQ = 262144.0f, kSoftQLow = 4194304.0f;
constexpr uint32_t kSoftLow = 11, kSoftLowFine = 512;
constexpr uint32_t kSoftDrain = 1u << 12;

// Forward where the centrals are neighbour records: every unordered pair once (sweep_pairs), its
// moments straight from the testing lane into the CTA's shared fine grid.  Bound by the shared-
// memory pipe (three scattered atomics per in-range pair) and issue.  Measured, 1e7-ion needle on
// half-size cells / 2e5 cylinder on full-size cells (ms): 36.8 -> 17.7 / 14.5 -> 0.79 (before: a warp
// list of the hits of every candidate of the half stencil, a float sum per moment, cells not split;
// 27.4 / 1.25 with the sweep and float sums; 19.4 / 0.92 with a row of bins per moment, which takes
// two more additions per pair than the three moments of a bin side by side); 17.7 -> 18.6 / 0.79 -> 0.82 with
// the finer units (the returned weights; with every turn of 2 records checked 20.2, with the low bits in a
// fourth word 22.6).
template <bool LOW>
__global__ void __launch_bounds__(256, 4) k_soft_fwd_sym(const SoftArgs a, const __grid_constant__ SweepArgs sw,
                                                         double unit1, double unit2) {
  griddep_wait();
  griddep_launch();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SweepBuf s_sweep[8];
  const uint32_t nf = a.n_fine, nf4 = (nf + 3u) & ~3u, lane = threadIdx.x & 31;
  uint32_t* sM = reinterpret_cast<uint32_t*>(smem);  // [nf4][3]: the three moments of a bin side by side
  uint32_t* sL = sM + 3 * nf4;                       // LOW [nf4]: the remainders' low bits
  for (uint32_t m = threadIdx.x; m < (LOW ? 4 : 3) * nf4; m += blockDim.x) sM[m] = 0;
  __syncthreads();
  SweepBuf& buf = s_sweep[threadIdx.x >> 5];
  const SoftFine fine(a);
  const float rc = a.rc, q1 = (LOW ? kSoftQLow : kSoftQ) * a.inv_w, q2 = kSoftQ * a.inv_w * a.inv_w;
  const unsigned long long q1_2 = f2_pack(q1, q1), q2_2 = f2_pack(q2, q2);
  const uint32_t base = smem_u32(sM) - 12u * kMagicBits, base_l = smem_u32(sL) - 4u * kMagicBits;
  // the rows' bins i, i + step, ... to the global moments
  auto drain = [&](uint32_t i, uint32_t step) {
    for (; i < nf; i += step) {
      const int32_t v0 = (int32_t)atomicExch(&sM[3 * i], 0u), vh = (int32_t)atomicExch(&sM[3 * i + 1], 0u),
                    v2 = (int32_t)atomicExch(&sM[3 * i + 2], 0u);
      const int64_t v1 = LOW ? (int64_t)vh * (1 << kSoftLow) + (int32_t)atomicExch(&sL[i], 0u) : (int64_t)vh;
      // (a count may stand below zero when its self pairs were drained before they were taken out)
      if (v0) atomicAdd(&a.M0[i], (unsigned long long)(long long)v0);
      if (v1) atomicAdd(&a.M1[i], (double)v1 * unit1);
      if (v2) atomicAdd(&a.M2[i], (double)v2 * unit2);
    }
  };
  sweep_pairs<false>(sw, buf, [&](uint32_t n_pr, uint32_t m, uint32_t nc, bool) __attribute__((always_inline)) {
    const float4 far = make_float4(INFINITY, INFINITY, INFINITY, __uint_as_float(kCandSingle));
    const float4 c0 = lane < nc ? buf.cand[lane] : far, c1 = lane + 32 < nc ? buf.cand[lane + 32] : far;
    const uint32_t k0 = __float_as_uint(c0.w), k1 = __float_as_uint(c1.w);
    const uint32_t w0 = k0 == kCandBoth ? 2u : 1u, w1 = k1 == kCandBoth ? 2u : 1u;
    const unsigned long long x0 = f2_pack(c0.x, c0.x), y0 = f2_pack(c0.y, c0.y), z0 = f2_pack(c0.z, c0.z);
    const unsigned long long x1 = f2_pack(c1.x, c1.x), y1 = f2_pack(c1.y, c1.y), z1 = f2_pack(c1.z, c1.z);
    auto deposit = [&](unsigned long long d2, uint32_t wt, uint32_t& hot) __attribute__((always_inline)) {
      const uint32_t off = 0u - kMagicBits * wt;
      const uint32_t off_h = 0u - (kMagicBits >> kSoftLow) * wt;  // (kMagicBits is a multiple of 2^kSoftLow)
      float da, db, u[2], mm[2], r1[2], r2[2];
      f2_unpack(d2, da, db);
      const unsigned long long u2 = f2_mul(f2_pack(sqrt_fast(da), sqrt_fast(db)), fine.scale2);
      unsigned long long m2, dl2;
      fine.split(u2, m2, dl2);
      f2_unpack(u2, u[0], u[1]), f2_unpack(m2, mm[0], mm[1]);
      f2_unpack(f2_fma(dl2, q1_2, fine.magic2), r1[0], r1[1]);  // rounded to the nearest unit
      f2_unpack(f2_fma(f2_mul(dl2, dl2), q2_2, fine.magic2), r2[0], r2[1]);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (u[e] < rc) {
          const uint32_t at = __float_as_uint(mm[e]) * 12u + base;
          // (without "memory" clobbers: C++ code touches these words only behind barriers and votes, see ps_items.cuh)
          uint32_t old;
          asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(at), "r"(wt));
          hot |= old;
          const uint32_t q = __float_as_uint(r1[e]);
          if (LOW) {
            const uint32_t at_l = __float_as_uint(mm[e]) * 4u + base_l;
            asm volatile("red.shared.add.u32 [%0+4], %1;" ::"r"(at), "r"((q >> kSoftLow) * wt + off_h));
            asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(at_l), "r"((q & ((1u << kSoftLow) - 1u)) * wt));
          } else {
            asm volatile("red.shared.add.u32 [%0+4], %1;" ::"r"(at), "r"(q * wt + off));
          }
          asm volatile("red.shared.add.u32 [%0+8], %1;" ::"r"(at), "r"(__float_as_uint(r2[e]) * wt + off));
        }
      }
    };
    const ulonglong2* rxy = reinterpret_cast<const ulonglong2*>(buf.rxy);
    const unsigned long long* rz = reinterpret_cast<const unsigned long long*>(buf.rz);
#pragma unroll 1
    for (uint32_t k = 0; k < n_pr; k += 2) {
      uint32_t hot = 0;
#pragma unroll
      for (uint32_t i = 0; i < 2; ++i) {
        const ulonglong2 xy = rxy[k + i];
        const unsigned long long zz = rz[k + i];
        deposit(soft_d2(f2_sub(x0, xy.x), f2_sub(y0, xy.y), f2_sub(z0, zz)), w0, hot);
        deposit(soft_d2(f2_sub(x1, xy.x), f2_sub(y1, xy.y), f2_sub(z1, zz)), w1, hot);
      }
      if (__any_sync(0xffffffffu, hot >= kSoftDrain)) drain(lane, 32);
    }
    // the staged records met themselves once each, at u = 0: taken out of bin 0 (remainder -w / 2)
    const uint32_t self = __popc(__ballot_sync(0xffffffffu, k0 == kCandSelf)) +
                          __popc(__ballot_sync(0xffffffffu, k1 == kCandSelf));
    if (self && lane == 0) {
      atomicAdd(&sM[0], 0u - self);
      atomicAdd(&sM[1], self * (LOW ? (uint32_t)(kSoftQLow / 2) >> kSoftLow : (uint32_t)(kSoftQ / 2)));
      atomicAdd(&sM[2], 0u - self * (uint32_t)(kSoftQ / 4));
    }
  });
  __syncthreads();
  drain(threadIdx.x, blockDim.x);
}

// d^n/du^n of Phi((e - u)/sigma), n = 0..3, in FP64
__device__ __forceinline__ void phi_derivs(double e, double u, double sigma, double out[4]) {
  const double t = (e - u) / sigma;
  const double ph = exp(-0.5 * t * t) * 0.39894228040143267794;  // 1/sqrt(2 pi)
  out[0] = 0.5 * erfc(-t * 0.70710678118654752440);
  out[1] = -ph / sigma;
  out[2] = -t * ph / (sigma * sigma);
  out[3] = (1.0 - t * t) * ph / (sigma * sigma * sigma);
}

// h[b] = sum_m M0 K_b + M1 K_b' + M2/2 K_b'' (one block per bin)
__global__ void __launch_bounds__(256) k_soft_finalize(const unsigned long long* __restrict__ M0,
                                                       const double* __restrict__ M1, const double* __restrict__ M2,
                                                       uint32_t n_fine, double w, double r0, double dr, double sigma,
                                                       float* __restrict__ h) {
  griddep_wait();
  griddep_launch();
  __shared__ double s_part[8];
  const uint32_t b = blockIdx.x;
  const double e0 = r0 + (double)b * dr, e1 = r0 + (double)(b + 1) * dr;
  double acc = 0.0;
  for (uint32_t m = threadIdx.x; m < n_fine; m += blockDim.x) {
    const unsigned long long n0 = M0[m];
    if (!n0) continue;
    const double c = ((double)m + 0.5) * w;
    double p1[4], p0[4];
    phi_derivs(e1, c, sigma, p1);
    phi_derivs(e0, c, sigma, p0);
    acc += (double)n0 * (p1[0] - p0[0]) + M1[m] * (p1[1] - p0[1]) + 0.5 * M2[m] * (p1[2] - p0[2]);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += s_part[i];
    h[b] = (float)t;
  }
}

// T[m] = W(c_m), W'(c_m), W''(c_m) / 2, all times `scale`, for W(u) = sum_b G[b] K_b'(u)
__global__ void __launch_bounds__(256) k_soft_table(const float* __restrict__ G, uint32_t n_bins, uint32_t n_fine,
                                                    double w, double r0, double dr, double sigma,
                                                    double scale, float4* __restrict__ T) {
  griddep_wait();
  griddep_launch();
  const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n_fine) return;
  const double c = ((double)m + 0.5) * w;
  double a1 = 0.0, a2 = 0.0, a3 = 0.0;
  double pl[4];
  phi_derivs(r0, c, sigma, pl);
  for (uint32_t b = 0; b < n_bins; ++b) {
    double ph[4];
    phi_derivs(r0 + (double)(b + 1) * dr, c, sigma, ph);
    const double g = (double)G[b];
    a1 += g * (ph[1] - pl[1]);
    a2 += g * (ph[2] - pl[2]);
    a3 += g * (ph[3] - pl[3]);
    for (int k = 0; k < 4; ++k) pl[k] = ph[k];
  }
  T[m] = make_float4((float)(scale * a1), (float)(scale * a2), (float)(0.5 * scale * a3), 0.f);
}

// ---------------------------------------------------------------------------
// adjoint passes
// ---------------------------------------------------------------------------
// Pass A (owners = centrals, write) and pass B (owners = neighbours, add), for central types that are
// not all neighbour types.
__global__ void __launch_bounds__(256) k_soft_bwd(const SoftArgs a) {
  griddep_wait();
  griddep_launch();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float4 s_buf[8][32];
  __shared__ uint32_t s_rsrc[8][kSoftRuns], s_rpre[8][kSoftRuns + 1];
  __shared__ double s_gs[8];
  float4* sT = reinterpret_cast<float4*>(smem);
  for (uint32_t m = threadIdx.x; m < a.n_fine; m += blockDim.x) sT[m] = a.T[m];
  __syncthreads();
  const uint32_t w = threadIdx.x >> 5;
  const float s = a.scale, inv_w = a.inv_w, wf = a.w, rc = a.rc;
  const uint32_t nf = a.n_fine;
  float gx = 0.f, gy = 0.f, gz = 0.f;
  double gs_lane = 0.0;
  float gs_item = 0.f;
  auto begin = [&]() { gx = gy = gz = 0.f, gs_item = 0.f; };
  auto pair = [&](const float4& p, float qx, float qy, float qz, float d2) {
    const float rs = d2 > 0.f ? rsqrtf(d2) : 0.f;
    const float d = d2 * rs;
    const float u = s * d;
    if (!(u < rc)) return;
    uint32_t m = (uint32_t)(u * inv_w);
    m = m < nf ? m : nf - 1;
    const float delta = u - ((float)m + 0.5f) * wf;
    const float4 t = sT[m];
    const float W = t.x + delta * (t.y + delta * t.z);  // times s
    const float f = W * rs;                             // W s / d (0 for coincident ions)
    gx += f * (p.x - qx);
    gy += f * (p.y - qy);
    gz += f * (p.z - qz);
    gs_item += W * d;
  };
  auto end = [&](bool valid, const float4& p) {
    if (!valid) return;
    const uint32_t idx = __float_as_uint(p.w);
    float* g = a.grad + 3 * (int64_t)idx;
    if (a.pass_b) {
      // owners are neighbours j: dL/dx_j = -sum W s (x_i - x_j)/d, here p = x_j, q = x_i
      g[0] += gx, g[1] += gy, g[2] += gz;
    } else {
      g[0] = gx, g[1] = gy, g[2] = gz;
      gs_lane += (double)gs_item;
    }
  };
  soft_items_owned(a, reinterpret_cast<float*>(s_buf[w]), s_rsrc[w], s_rpre[w], pair, begin, end);
  if (!a.pass_b) {
    for (int o = 16; o > 0; o >>= 1) gs_lane += __shfl_xor_sync(0xffffffffu, gs_lane, o);
    if ((threadIdx.x & 31) == 0) s_gs[w] = gs_lane;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += s_gs[i];
      atomicAdd(a.grad_s, t / (double)a.scale);
    }
  }
}

// Sums v[0..11] over the warp: afterwards lane l holds, in v[0], the sum of value
// sum_slot(l) (lanes that differ in bit 0 alone hold the same one).  13 exchanges instead of 60:
// each step sends away the half of the values that the partner keeps.
template <int N>
__device__ __forceinline__ void warp_sum_step(float (&v)[12], uint32_t lane, uint32_t o) {
  const bool up = (lane & o) != 0u;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float keep = up ? v[i + N] : v[i], send = up ? v[i] : v[i + N];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
}
__device__ __forceinline__ void warp_sum12(float (&v)[12], uint32_t lane) {
  warp_sum_step<6>(v, lane, 16);
  warp_sum_step<3>(v, lane, 8);
  v[3] = 0.f;  // the fourth value of each lane is empty
  warp_sum_step<2>(v, lane, 4);
  warp_sum_step<1>(v, lane, 2);
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
}
// the value that lane l ends up with, or 12 (none)
__device__ __forceinline__ uint32_t sum_slot(uint32_t lane) {
  const uint32_t k = ((lane >> 2) & 1u) * 2u + ((lane >> 1) & 1u);  // of the three left after two steps
  return k == 3u ? 12u : ((lane >> 4) & 1u) * 6u + ((lane >> 3) & 1u) * 3u + k;
}

__device__ __forceinline__ void red_global_v4(float4* p, float x, float y, float z) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(0.f)
               : "memory");
}

// Adjoint where the centrals are neighbour records: every unordered pair once (sweep_pairs), its
// force f (x_j - x_i) added at both ends.  The candidate end sums over the staged records in
// its lane's registers; the record end is summed over the lanes (warp_sum12, four records at a
// time) into shared memory; both go to the record-ordered gradient `acc` with one 16-byte
// reduction per record and tile (neighbouring candidates are neighbouring records), which
// k_soft_grad_out scatters to the ions.  Bound by issue (~30 instructions per 32 tests) and by
// the table's shared-memory reads.  Measured, 1e7-ion needle on half-size cells / 2e5 cylinder on
// full-size cells (ms): 75.4 -> 23.3 / 3.56 -> 1.32 (before: every record a lane of its own, each
// pair tested and evaluated from both ends); 128 or 64 registers a thread: 29.1 and 23.7 ms; the
// table as a pair and a single value per bin instead of one 16-byte entry: 23.8 ms.
__global__ void __launch_bounds__(256, 3) k_soft_bwd_sym(const SoftArgs a, const __grid_constant__ SweepArgs sw,
                                                         float4* __restrict__ acc) {
  griddep_wait();
  griddep_launch();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SweepBuf s_sweep[8];
  __shared__ float s_rec[8][kSweepRec * 3];  // per warp: gradients of the staged records
  __shared__ double s_gs[8];
  float4* sT = reinterpret_cast<float4*>(smem);
  const uint32_t nf = a.n_fine, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (uint32_t m = threadIdx.x; m < nf; m += blockDim.x) sT[m] = a.T[m];
  for (uint32_t i = lane; i < kSweepRec * 3; i += 32) s_rec[w][i] = 0.f;
  __syncthreads();
  SweepBuf& buf = s_sweep[w];
  float* grec = s_rec[w];
  const SoftFine fine(a);
  const float rc = a.rc;
  const uint32_t table = smem_u32(sT) - 16u * kMagicBits;
  const uint32_t slot = sum_slot(lane);
  double gs_lane = 0.0;
  sweep_pairs<true>(
      sw, buf,
      [&](uint32_t n_pr, uint32_t, uint32_t nc, bool) __attribute__((always_inline)) {
        const float4 far = make_float4(INFINITY, INFINITY, INFINITY, __uint_as_float(kCandSingle));
        float4 c[2] = {lane < nc ? buf.cand[lane] : far, lane + 32 < nc ? buf.cand[lane + 32] : far};
        float ws[2], g[2][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}}, gs = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) ws[h] = __float_as_uint(c[h].w) == kCandBoth ? 2.f : 1.f;
        const ulonglong2* rxy = reinterpret_cast<const ulonglong2*>(buf.rxy);
        const unsigned long long* rz = reinterpret_cast<const unsigned long long*>(buf.rz);
#pragma unroll 1
        for (uint32_t k = 0; k < n_pr; k += 2) {  // four records
          float r[12];
#pragma unroll
          for (int i = 0; i < 12; ++i) r[i] = 0.f;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const ulonglong2 xy = rxy[k + q];
            const unsigned long long zz = rz[k + q];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const unsigned long long dx2 = f2_sub(f2_pack(c[h].x, c[h].x), xy.x),
                                       dy2 = f2_sub(f2_pack(c[h].y, c[h].y), xy.y),
                                       dz2 = f2_sub(f2_pack(c[h].z, c[h].z), zz);
              float da, db;
              const unsigned long long d2 = soft_d2(dx2, dy2, dz2);
              f2_unpack(d2, da, db);
              const unsigned long long rs2 = f2_pack(rsqrt_fast(da), rsqrt_fast(db)), dd2 = f2_mul(d2, rs2),
                                       u2 = f2_mul(dd2, fine.scale2);  // NaN at d = 0: no pair
              unsigned long long m2, dl2;
              fine.split(u2, m2, dl2);
              float u[2], mm[2], dl[2], rs[2], dd[2], dx[2], dy[2], dz[2];
              f2_unpack(u2, u[0], u[1]), f2_unpack(m2, mm[0], mm[1]), f2_unpack(dl2, dl[0], dl[1]);
              f2_unpack(rs2, rs[0], rs[1]), f2_unpack(dd2, dd[0], dd[1]);
              f2_unpack(dx2, dx[0], dx[1]), f2_unpack(dy2, dy[0], dy[1]), f2_unpack(dz2, dz[0], dz[1]);
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                if (u[e] < rc) {
                  float t0, t1, t2;  // (the fourth value pads the entry to one 16-byte load)
                  asm("{.reg .f32 pad; ld.shared.v4.f32 {%0, %1, %2, pad}, [%3];}"
                      : "=f"(t0), "=f"(t1), "=f"(t2)
                      : "r"(__float_as_uint(mm[e]) * 16u + table));
                  const float W = (t0 + dl[e] * (t1 + dl[e] * t2)) * ws[h];
                  const float f = W * rs[e];
                  gs += W * dd[e];
                  g[h][0] = __fmaf_rn(f, dx[e], g[h][0]), g[h][1] = __fmaf_rn(f, dy[e], g[h][1]),
                  g[h][2] = __fmaf_rn(f, dz[e], g[h][2]);
                  r[6 * q + 3 * e] = __fmaf_rn(-f, dx[e], r[6 * q + 3 * e]);
                  r[6 * q + 3 * e + 1] = __fmaf_rn(-f, dy[e], r[6 * q + 3 * e + 1]);
                  r[6 * q + 3 * e + 2] = __fmaf_rn(-f, dz[e], r[6 * q + 3 * e + 2]);
                }
              }
            }
          }
          warp_sum12(r, lane);
          // value 6 q + 3 e + axis: record 2 (k + q) + e
          if (slot < 12u && !(lane & 1u)) grec[6 * k + slot] += r[0];
        }
        gs_lane += (double)gs;
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (lane + 32 * h < nc) red_global_v4(acc + buf.cidx[lane + 32 * h], g[h][0], g[h][1], g[h][2]);
      },
      [&](uint32_t m, bool) __attribute__((always_inline)) {
        __syncwarp();
        for (uint32_t r = lane; r < m; r += 32) {
          red_global_v4(acc + buf.ridx[r], grec[3 * r], grec[3 * r + 1], grec[3 * r + 2]);
          grec[3 * r] = grec[3 * r + 1] = grec[3 * r + 2] = 0.f;
        }
        __syncwarp();
      });
  for (int o = 16; o > 0; o >>= 1) gs_lane += __shfl_xor_sync(0xffffffffu, gs_lane, o);
  if (lane == 0) s_gs[w] = gs_lane;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += s_gs[i];
    atomicAdd(a.grad_s, t / (double)a.scale);
  }
}

// the record-ordered gradient to the ions
__global__ void __launch_bounds__(256) k_soft_grad_out(const float4* __restrict__ nrec, const float4* __restrict__ acc,
                                                       const Geo* __restrict__ geo, float* __restrict__ grad) {
  griddep_wait();
  griddep_launch();
  const uint32_t n = geo->n_sel;
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    const float4 v = acc[j];
    float* g = grad + 3 * (int64_t)__float_as_uint(__ldg(nrec + j).w);
    g[0] = v.x, g[1] = v.y, g[2] = v.z;
  }
}

// warp items (cell, first << 6 | count) over every non-empty cell of a list
__global__ void __launch_bounds__(256) k_make_items(const uint32_t* __restrict__ start, Geo* geo,
                                                    uint2* __restrict__ item) {
  griddep_wait();
  griddep_launch();
  const uint32_t nc = geo->n_cells;
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t base = blockIdx.x * blockDim.x; base < nc; base += gridDim.x * blockDim.x) {
    const uint32_t c = base + threadIdx.x;
    const uint32_t v = c < nc ? start[c + 1] - start[c] : 0u;
    const uint32_t m = v == 0 ? 0u : (v + 31u) / 32u;
    uint32_t x = m;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, x, 31);
    uint32_t b0 = 0;
    if (lane == 31 && total) b0 = atomicAdd(&geo->work_n2, total);
    b0 = __shfl_sync(0xffffffffu, b0, 31);
    uint32_t slot = b0 + x - m;
    if (m) {
      const uint32_t bs = v / m, rem = v % m;
      uint32_t first = 0;
      for (uint32_t q = 0; q < m; ++q) {
        const uint32_t cnt = bs + (q < rem ? 1u : 0u);
        item[slot++] = make_uint2(c, (first << 6) | cnt);
        first += cnt;
      }
    }
  }
}

__global__ void k_reset_items(Geo* geo) {
  griddep_wait();
  griddep_launch();
  if (threadIdx.x == 0) geo->work_n2 = 0, geo->work_n3 = 0, geo->work_next2 = 0;
}

__global__ void k_soft_gs_out(const double* __restrict__ gs, float* __restrict__ out) {
  griddep_wait();
  griddep_launch();
  if (threadIdx.x == 0) *out = (float)*gs;
}

static int soft_setup(ps_grid* g, float sigma, float scale, ps_bins bins, SoftArgs& sa, double& w_out) {
  if (!(sigma > 0.0f) || !std::isfinite(sigma)) return fail(PS_ERR_INVALID_ARG, "smoothed RDF: sigma must be > 0");
  if (!(scale > 0.0f) || !std::isfinite(scale)) return fail(PS_ERR_INVALID_ARG, "smoothed RDF: scale must be > 0");
  const double stop = bins.r0 + (double)bins.n_bins * bins.dr;
  const double rc = stop + 6.0 * (double)sigma;
  if ((double)g->r_cut * (double)scale < rc * (1.0 + 1e-6))
    return fail(PS_ERR_INVALID_ARG, "smoothed RDF: grid r_cut * scale must cover stop + 6 sigma");
  const double w = soft_width(sigma, rc);
  sa.n_fine = soft_bins(w, rc);
  sa.w = (float)w;
  sa.inv_w = (float)(1.0 / w);
  sa.scale = scale;
  sa.sigma = sigma;
  sa.rc = (float)rc;
  const double rcu = rc / (double)scale;
  sa.rc2u = (float)(rcu * rcu * (1.0 + 1e-6));
  sa.stencil = g->stencil;
  w_out = w;
  return PS_OK;
}

static int launch_grid_for(const ps_grid* g, const void* kern, uint32_t smem, int* blocks) {
  int per_sm = 0;
  PS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  PS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, smem));
  if (per_sm < 1) return fail(PS_ERR_UNSUPPORTED, "smoothed RDF kernel does not fit on an SM");
  *blocks = g->num_sms * per_sm;
  return PS_OK;
}

// Owners = the neighbour records: warp items over the non-empty neighbour cells.
static int nbr_items(ps_grid* g, SoftArgs& sa, cudaStream_t s, uint32_t kid) {
  PS_LAUNCH(kid, s, PS_CUDA(launch_pdl(k_reset_items, 1, 32, 0, s, g->nbr.geo)));
  PS_LAUNCH(kid, s, PS_CUDA(launch_pdl(k_make_items, g->num_sms * 4, 256, 0, s, g->nbr.start, g->nbr.geo, g->nbr_witem)));
  sa.orec = g->nbr.rec;
  sa.ostart = g->nbr.start;
  sa.oitem = g->nbr_witem;
  sa.ocap = g->item_cap;
  sa.ogeo = g->nbr.geo;
  return PS_OK;
}

int soft_forward(ps_grid* g, const float* dsrf, const uint64_t ctr_mask[4], float dsrf_min, float sigma, float scale,
                 ps_bins bins, float* d_h, cudaStream_t s) {
  SoftArgs sa;
  memset(&sa, 0, sizeof(sa));
  double w = 0.0;
  int rc = soft_setup(g, sigma, scale, bins, sa, w);
  if (rc) return rc;
  ZeroOut z;  // the moment accumulators are zeroed by the central-list reset kernel
  z.p[0] = reinterpret_cast<uint64_t*>(g->soft_m0);
  z.p[1] = reinterpret_cast<uint64_t*>(g->soft_m1);
  z.p[2] = reinterpret_cast<uint64_t*>(g->soft_m2);
  z.n[0] = z.n[1] = z.n[2] = sa.n_fine;
  const bool sym = centrals_in_neighbours(g, ctr_mask);
  rc = build_central_list(g, dsrf, ctr_mask, dsrf_min, s, z, false, false, !sym, sym ? kSweep : kNoSweep);
  if (rc) return rc;
  sa.nrec = g->nbr.rec;
  sa.nstart = g->nbr.start;
  sa.ngeo = g->nbr.geo;
  sa.M0 = g->soft_m0;
  sa.M1 = g->soft_m1;
  sa.M2 = g->soft_m2;
  int blocks = 0;
  if (sym) {
    const bool low = sa.n_fine < kSoftLowFine;
    const uint32_t smem = ((sa.n_fine + 3u) & ~3u) * (low ? 16 : 12);
    auto kern = low ? k_soft_fwd_sym<true> : k_soft_fwd_sym<false>;
    rc = launch_grid_for(g, (const void*)kern, smem, &blocks);
    if (rc) return rc;
    SweepArgs sw = sweep_args(g, &g->ctr.geo->sym_next);
    sw.range = sa.rc2u;
    PS_LAUNCH(PS_KID_SOFT_FWD, s,
              PS_CUDA(launch_pdl(kern, blocks, 256, smem, s, sa, sw, w / (double)(low ? kSoftQLow : kSoftQ),
                                 w * w / (double)kSoftQ)));
  } else {
    const uint32_t smem = sa.n_fine * 12;
    rc = launch_grid_for(g, (const void*)k_soft_fwd, smem, &blocks);
    if (rc) return rc;
    sa.orec = g->ctr.rec;
    sa.ostart = g->ctr.start;
    sa.oitem = g->ctr.witem;
    sa.ocap = g->item_cap;
    sa.ogeo = g->ctr.geo;
    PS_LAUNCH(PS_KID_SOFT_FWD, s, PS_CUDA(launch_pdl(k_soft_fwd, blocks, 256, smem, s, sa)));
  }
  PS_LAUNCH(PS_KID_SOFT_FWD, s,
            PS_CUDA(launch_pdl(k_soft_finalize, bins.n_bins, 256, 0, s, g->soft_m0, g->soft_m1, g->soft_m2, sa.n_fine, w, bins.r0,
                                                        bins.dr, (double)sigma, d_h)));
  PS_CUDA(cudaGetLastError());
  return PS_OK;
}

int soft_backward(ps_grid* g, const float* dsrf, const uint64_t ctr_mask[4], float dsrf_min, float sigma, float scale,
                  ps_bins bins, const float* d_G, float* d_grad, float* d_grad_s, cudaStream_t s) {
  SoftArgs sa;
  memset(&sa, 0, sizeof(sa));
  double w = 0.0;
  int rc = soft_setup(g, sigma, scale, bins, sa, w);
  if (rc) return rc;
  const bool sym = centrals_in_neighbours(g, ctr_mask);
  rc = build_central_list(g, dsrf, ctr_mask, dsrf_min, s, ZeroOut(), false, false, !sym, sym ? kSweep : kNoSweep);
  if (rc) return rc;
  PS_CUDA(cudaMemsetAsync(d_grad, 0, (size_t)g->n * 3 * sizeof(float), s));
  PS_CUDA(cudaMemsetAsync(g->soft_gs, 0, sizeof(double), s));
  PS_LAUNCH(PS_KID_SOFT_BWD, s,
            PS_CUDA(launch_pdl(k_soft_table, (sa.n_fine + 255) / 256, 256, 0, s, d_G, bins.n_bins, sa.n_fine, w, bins.r0, bins.dr,
                                                                 (double)sigma, (double)scale, reinterpret_cast<float4*>(g->soft_T))));
  sa.T = reinterpret_cast<const float4*>(g->soft_T);
  sa.grad = d_grad;
  sa.grad_s = g->soft_gs;
  const uint32_t smem = sa.n_fine * 16;
  int blocks = 0;
  if (sym) {
    // the record-ordered gradient takes the place of the central records, which the sweep does not use
    rc = launch_grid_for(g, (const void*)k_soft_bwd_sym, smem, &blocks);
    if (rc) return rc;
    float4* acc = g->ctr.rec;
    PS_CUDA(cudaMemsetAsync(acc, 0, (size_t)g->n * sizeof(float4), s));
    SweepArgs sw = sweep_args(g, &g->ctr.geo->sym_next);
    sw.range = sa.rc2u;
    PS_LAUNCH(PS_KID_SOFT_BWD, s, PS_CUDA(launch_pdl(k_soft_bwd_sym, blocks, 256, smem, s, sa, sw, acc)));
    PS_LAUNCH(PS_KID_SOFT_BWD, s,
              PS_CUDA(launch_pdl(k_soft_grad_out, g->num_sms * 8, 256, 0, s, g->nbr.rec, acc, g->nbr.geo, d_grad)));
  } else {
    rc = launch_grid_for(g, (const void*)k_soft_bwd, smem, &blocks);
    if (rc) return rc;
    // pass A: owners = centrals, candidates = neighbours
    sa.orec = g->ctr.rec;
    sa.ostart = g->ctr.start;
    sa.oitem = g->ctr.witem;
    sa.ocap = g->item_cap;
    sa.ogeo = g->ctr.geo;
    sa.nrec = g->nbr.rec;
    sa.nstart = g->nbr.start;
    sa.ngeo = g->nbr.geo;
    sa.pass_b = 0;
    PS_LAUNCH(PS_KID_SOFT_BWD, s, PS_CUDA(launch_pdl(k_soft_bwd, blocks, 256, smem, s, sa)));
    // pass B: owners = neighbours, candidates = centrals
    rc = nbr_items(g, sa, s, PS_KID_SOFT_BWD);
    if (rc) return rc;
    sa.nrec = g->ctr.rec;
    sa.nstart = g->ctr.start;
    sa.ngeo = g->nbr.geo;
    sa.pass_b = 1;
    PS_LAUNCH(PS_KID_SOFT_BWD, s, PS_CUDA(launch_pdl(k_soft_bwd, blocks, 256, smem, s, sa)));
  }
  PS_LAUNCH(PS_KID_SOFT_BWD, s, PS_CUDA(launch_pdl(k_soft_gs_out, 1, 32, 0, s, g->soft_gs, d_grad_s)));
  PS_CUDA(cudaGetLastError());
  return PS_OK;
}

}  // namespace ps
