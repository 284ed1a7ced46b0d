// Spatial distribution map: the three-dimensional two-point statistic of which
// the RDF and the kNN distributions are annular integrals (Methods,
// "Descriptive, two-point spatial statistics, and clustering").  For every
// central ion and every neighbour within the ROI radius R (d2 < (float)(R*R)),
// the float32 displacement x_j - x_i is binned into cubic voxels of edge w;
// the paper's setting is w = 0.025 nm with R = 2 nm (Results, strong scaling).
//
// Where the centrals are neighbour records and not few every unordered pair is met once
// (sweep_pairs) and the pairs with two central ends are mirrored afterwards; where they
// are few each gets a warp.
// Otherwise the enumeration is over the exact query's cell grid and central list:
// each central gets one thread; the centrals of a dense cell's item share the
// candidate walk, so their loads of a record broadcast from L1 (cells with at
// most 3 centrals let the lanes split each central's candidates instead);
// sparse cells' items are taken 32 at a time.  Voxel edges V[m] = (float)((m - n_vox/2) * w)
// (double arithmetic) sit in shared memory; a voxel index is guessed from
// (d - V[0]) / w and checked against the table, so the half-open rule
// V[m] <= d < V[m+1] holds exactly.  The map (n_vox^3 uint64 counters, 33 MB
// for the paper's 160^3 voxels) stays L2-resident and takes global atomics.
#include <cstring>

#include "ps_internal.cuh"
#include "ps_sweep.cuh"

namespace ps {

struct SdmArgs {
  const float4* nrec;
  const uint32_t* nstart;
  const Geo* ngeo;
  const float4* crec;
  const uint32_t* cstart;
  const uint32_t* cwork;
  const uint2* witem;
  uint32_t work_cap;
  Geo* cgeo;
  int stencil;
  float ER;  // (float)(R * R)
  double w;
  uint32_t n_vox;
  unsigned long long* H;
  uint64_t* meta;
  int covers;  // the voxel cube holds every displacement below the ROI radius
};

constexpr uint32_t kSdmMaxVox = 1024;
constexpr uint32_t kSdmLightCap = 32 * (kHeavy - 1);

// voxel index along one axis: m with V[m] <= d < V[m+1], or -1 outside [V[0], V[n])
__device__ __forceinline__ int sdm_vox(float d, const float* sV, uint32_t n, float inv_w) {
  if (!(d >= sV[0]) || !(d < sV[n])) return -1;
  int m = (int)((d - sV[0]) * inv_w);
  m = m < 0 ? 0 : (m >= (int)n ? (int)n - 1 : m);
  while (m > 0 && d < sV[m]) --m;
  while (m + 1 < (int)n && d >= sV[m + 1]) ++m;
  return m;
}

// one candidate q of central p (index word pidx)
__device__ __forceinline__ void sdm_pair(const SdmArgs& a, const float* sV, float inv_w, const float4& p, const float4& q,
                                         uint64_t& in_map, uint64_t& outside) {
  // the same float32 operations as the squared distance: dx = x_j - x_i
  const float dx = __fsub_rn(q.x, p.x), dy = __fsub_rn(q.y, p.y), dz = __fsub_rn(q.z, p.z);
  const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
  if (d2 < a.ER && __float_as_uint(q.w) != __float_as_uint(p.w)) {
    const uint32_t nv = a.n_vox;
    const int mx = sdm_vox(dx, sV, nv, inv_w), my = sdm_vox(dy, sV, nv, inv_w), mz = sdm_vox(dz, sV, nv, inv_w);
    if ((mx | my | mz) < 0) {
      ++outside;
    } else {
      atomicAdd(&a.H[((uint64_t)mz * nv + (uint64_t)my) * nv + (uint64_t)mx], 1ull);
      ++in_map;
    }
  }
}

// The pairs of one central (record index rec, cell ce of the neighbour grid) with the
// candidates j0 + off, j0 + off + step, ... of every stencil row.
__device__ __forceinline__ void sdm_central(const SdmArgs& a, const Geo& ng, const float* sV, float inv_w,
                                            uint32_t rec, uint32_t ce, uint32_t off, uint32_t step, uint64_t& in_map,
                                            uint64_t& outside) {
  const float4 p = __ldg(a.crec + rec);
  const int st = a.stencil;
  const uint32_t cx = ce % ng.dims[0], cy = (ce / ng.dims[0]) % ng.dims[1], cz = ce / (ng.dims[0] * ng.dims[1]);
  const uint32_t xlo = cx >= (uint32_t)st ? cx - st : 0;
  const uint32_t xhi = cx + st < ng.dims[0] ? cx + st : ng.dims[0] - 1;
  const int ylo = max((int)cy - st, 0), yhi = min((int)cy + st, (int)ng.dims[1] - 1);
  const int zlo = max((int)cz - st, 0), zhi = min((int)cz + st, (int)ng.dims[2] - 1);
  for (int z = zlo; z <= zhi; ++z)
    for (int y = ylo; y <= yhi; ++y) {
      const uint32_t row = ((uint32_t)z * ng.dims[1] + (uint32_t)y) * ng.dims[0];
      const uint32_t j1 = a.nstart[row + xhi + 1];
      for (uint32_t j = a.nstart[row + xlo] + off; j < j1; j += step)
        sdm_pair(a, sV, inv_w, p, __ldg(a.nrec + j), in_map, outside);
    }
}

// The pairs of one central by a warp: lane r holds stencil row r (32 rows at a time), and the rows' records are
// walked as one list (rows of thin clouds hold a few records each), a position's row found by
// bisection over the lanes.
__device__ __forceinline__ void sdm_central_list(const SdmArgs& a, const Geo& ng, const float* sV, float inv_w,
                                                 const float4& p, uint64_t& in_map, uint64_t& outside) {
  const uint32_t lane = threadIdx.x & 31, ce = cell_of(ng, p.x, p.y, p.z);
  const int st = a.stencil, W = 2 * st + 1, n_rows = W * W;
  const uint32_t cx = ce % ng.dims[0], cy = (ce / ng.dims[0]) % ng.dims[1], cz = ce / (ng.dims[0] * ng.dims[1]);
  const uint32_t xlo = cx >= (uint32_t)st ? cx - st : 0, xhi = min(cx + st, ng.dims[0] - 1);
  for (int r0 = 0; r0 < n_rows; r0 += 32) {
    const int r = r0 + (int)lane, y = (int)cy + r % W - st, z = (int)cz + r / W - st;
    uint32_t src = 0, pre = 0;
    if (r < n_rows && y >= 0 && z >= 0 && y < (int)ng.dims[1] && z < (int)ng.dims[2]) {
      const uint32_t row = ((uint32_t)z * ng.dims[1] + (uint32_t)y) * ng.dims[0];
      src = a.nstart[row + xlo];
      pre = a.nstart[row + xhi + 1] - src;
    }
    const uint32_t len = pre;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, pre, o);
      if (lane >= (uint32_t)o) pre += v;
    }
    const uint32_t n_list = __shfl_sync(0xffffffffu, pre, 31);
    pre -= len;
    const uint32_t first = src - pre;
    for (uint32_t b = 0; b < n_list; b += 32) {
      const uint32_t pos = b + lane;
      uint32_t k = 0;
#pragma unroll
      for (uint32_t h = 16; h > 0; h >>= 1)
        if (__shfl_sync(0xffffffffu, pre, k + h) <= pos) k += h;
      const uint32_t j = __shfl_sync(0xffffffffu, first, k) + pos;
      if (pos < n_list) sdm_pair(a, sV, inv_w, p, __ldg(a.nrec + j), in_map, outside);
    }
  }
}

__global__ void __launch_bounds__(256) k_sdm(const SdmArgs a) {
  griddep_wait();
  griddep_launch();
  __shared__ float sV[kSdmMaxVox + 1];
  __shared__ uint32_t s_rec[8][kSdmLightCap], s_cell[8][kSdmLightCap];
  for (uint32_t m = threadIdx.x; m <= a.n_vox; m += blockDim.x)
    sV[m] = __double2float_rn(__dmul_rn(__dsub_rn((double)m, (double)a.n_vox * 0.5), a.w));
  __syncthreads();
  const float inv_w = (float)(1.0 / a.w);
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const Geo ng = *a.ngeo;
  uint64_t in_map = 0, outside = 0;

  // cells listed for the CTA-staged kernel (when the grid has that option): 32 centrals at a time
  const uint32_t n_dense = a.cgeo->work_n;
  for (;;) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(&a.cgeo->work_next, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_dense) break;
    const uint32_t c = a.cwork[item];
    const uint32_t c0 = a.cstart[c], n_c = a.cstart[c + 1] - c0;
    for (uint32_t b = lane; b < n_c; b += 32) sdm_central(a, ng, sV, inv_w, c0 + b, c, 0, 1, in_map, outside);
  }
  // items from the front (dense cells): the lanes take the item's centrals (one cell, so they walk
  // the same records in step); with <= 3 centrals they split each central's candidates instead
  const uint32_t n_front = a.cgeo->work_n2, n_light = a.cgeo->work_n3;
  for (;;) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(&a.cgeo->work_next2, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_front) break;
    const uint2 it = a.witem[item];
    const uint32_t c = it.x, cnt = it.y & 63u, r0 = a.cstart[c] + (it.y >> 6);
    if (cnt > 3) {
      if (lane < cnt) sdm_central(a, ng, sV, inv_w, r0 + lane, c, 0, 1, in_map, outside);
    } else {
      for (uint32_t ci = 0; ci < cnt; ++ci) sdm_central(a, ng, sV, inv_w, r0 + ci, c, lane, 32, in_map, outside);
    }
  }
  // items from the back (sparse cells), 32 at a time: their centrals are spread over the lanes
  uint32_t* rl = s_rec[w];
  uint32_t* cl = s_cell[w];
  for (;;) {
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(&a.cgeo->work_next3, 32u);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base >= n_light) break;
    uint32_t c = 0, f = 0, cnt = 0;
    if (base + lane < n_light) {
      const uint2 it = a.witem[a.work_cap - 1 - (base + lane)];
      c = it.x;
      f = a.cstart[c] + (it.y >> 6);
      cnt = it.y & 63u;
    }
    uint32_t inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= (uint32_t)o) inc += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
    __syncwarp();
    for (uint32_t q = 0; q < cnt; ++q) rl[inc - cnt + q] = f + q, cl[inc - cnt + q] = c;
    __syncwarp();
    for (uint32_t r = lane; r < total; r += 32) sdm_central(a, ng, sV, inv_w, rl[r], cl[r], 0, 1, in_map, outside);
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    in_map += __shfl_xor_sync(0xffffffffu, in_map, o);
    outside += __shfl_xor_sync(0xffffffffu, outside, o);
  }
  if (lane == 0) {
    if (in_map) atomicAdd((unsigned long long*)&a.meta[1], (unsigned long long)in_map);
    if (outside) atomicAdd((unsigned long long*)&a.meta[2], (unsigned long long)outside);
  }
}

// ---------------------------------------------------------------------------
// centrals among the neighbours: every unordered pair once (sweep_pairs)
//
// The displacements of the two orders of a pair are opposite, and the voxel edges are symmetric
// (V[n - m] == -V[m]), so off the edges the voxel of -d is the mirror image N - 1 - lin of that of d.
// A pair with two central ends is counted once, in the upper of its two voxels, and k_sdm_mirror
// adds the upper half of the map to the lower one at the end.  A displacement that counts alone (one central
// end, or on an edge of its voxel) is counted where it lies; if that is the upper half, one is
// taken from its mirror image (modulo 2^64), which the mirroring puts back.  Bound by the global
// atomics: half as many as one per ordered pair.
//
// The voxel index is floor(d / w + n / 2), taken twice with n / 2 -+ n 2^-21 (the quotient, its
// product with the rounded 1 / w and the rounded edges are each good to n 2^-24): where the
// two floors differ on any axis the pair goes through the edge table.
// Measured on the 8e6-ion needle (all-all, 160^3 voxels, full-size cells): 131 -> 26.8 ms (31.7 with cells
// whose records are not ordered by sub-cells).
// ---------------------------------------------------------------------------
// Few centrals among the records: the sweep stages and culls every record, a warp per central reads the central's
// stencil only, row by row, or in thin clouds (rows of fewer than 24 records) the rows as one list.  Measured, whole
// call, a share of the ions at random (central by central / sweep, ms; before the sweep):
//   8e6-ion needle, 2 nm, half-size cells (13 per cell)  0.05 6.7 / 6.4 (10.9), 0.02 2.9 / 4.4 (4.1), 0.002 0.65 / 1.8 (0.78)
//   the same, full-size cells (104)                      0.05 7.9 / 7.0 (19.6), 0.02 3.4 / 5.0 (13.0)
//   1 nm, half-size cells (1.7), as one list             0.2 5.3 / 5.3 (7.0), 0.1 2.9 / 4.0 (3.8; row by row 4.0)
//   1 nm, full-size cells (13)                           0.1 3.4 / 2.8 (7.0), 0.05 1.9 / 2.4 (2.6)
__host__ __device__ __forceinline__ bool sdm_sweep_pays(uint64_t n_nbr, uint64_t n_cells, uint64_t n_ctr) {
  return 32 * n_ctr >= n_nbr + 8 * n_cells;
}
__host__ __device__ __forceinline__ bool sdm_thin(uint64_t n_nbr, uint64_t n_cells, int stencil) {
  return (2 * stencil + 1) * n_nbr < 24 * n_cells;
}

__device__ __forceinline__ unsigned long long f2_add_down(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__global__ void __launch_bounds__(256, 4) k_sdm_sym(const __grid_constant__ SdmArgs a, const __grid_constant__ SweepArgs sw) {
  griddep_wait();
  griddep_launch();
  __shared__ float sV[kSdmMaxVox + 1];
  __shared__ SweepBuf s_sweep[8];
  const uint32_t nv = a.n_vox, N = nv * nv * nv;
  for (uint32_t m = threadIdx.x; m <= nv; m += blockDim.x)
    sV[m] = __double2float_rn(__dmul_rn(__dsub_rn((double)m, (double)nv * 0.5), a.w));
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31;
  SweepBuf& buf = s_sweep[threadIdx.x >> 5];
  const float inv_w = (float)(1.0 / a.w), eps = (float)nv * (1.0f / 2097152.0f), mid = 0.5f * (float)nv;
  const unsigned long long inv2 = f2_pack(inv_w, inv_w), hi2 = f2_pack(mid + eps, mid + eps),
                           lo2 = f2_pack(mid - eps, mid - eps), magic2 = f2_pack(kMagic, kMagic),
                           one2 = f2_pack(sw.one, sw.one);
  uint64_t in_map = 0, outside = 0;
  auto totals = [&]() __attribute__((always_inline)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      in_map += __shfl_xor_sync(0xffffffffu, in_map, o);
      outside += __shfl_xor_sync(0xffffffffu, outside, o);
    }
    if (lane == 0) {
      if (in_map) atomicAdd((unsigned long long*)&a.meta[1], (unsigned long long)in_map);
      if (outside) atomicAdd((unsigned long long*)&a.meta[2], (unsigned long long)outside);
    }
  };
  const uint32_t n_ctr = a.cgeo->n_sel;
  if (!sdm_sweep_pays(a.ngeo->n_sel, a.ngeo->n_cells, n_ctr)) {
    const Geo ng = *a.ngeo;
    const bool thin = sdm_thin(ng.n_sel, ng.n_cells, a.stencil);
    for (;;) {
      uint32_t i = 0;
      if (lane == 0) i = atomicAdd(sw.next, 1u);
      i = __shfl_sync(0xffffffffu, i, 0);
      if (i >= n_ctr) break;
      const float4 p = __ldg(a.crec + i);
      if (thin)
        sdm_central_list(a, ng, sV, inv_w, p, in_map, outside);
      else
        sdm_central(a, ng, sV, inv_w, i, cell_of(ng, p.x, p.y, p.z), lane, 32, in_map, outside);
    }
    totals();
    return;
  }
  // one displacement of weight v (1, or -1 modulo 2^64) in voxel lin
  auto alone = [&](uint32_t lin, unsigned long long v) {
    atomicAdd(&a.H[lin], v);
    const uint32_t mir = N - 1 - lin;
    if (lin > mir) atomicAdd(&a.H[mir], 0ull - v);
  };
  auto exact = [&](float dx, float dy, float dz) {
    const int mx = sdm_vox(dx, sV, nv, inv_w), my = sdm_vox(dy, sV, nv, inv_w), mz = sdm_vox(dz, sV, nv, inv_w);
    if ((mx | my | mz) < 0) {
      ++outside;
    } else {
      alone(((uint32_t)mz * nv + (uint32_t)my) * nv + (uint32_t)mx, 1ull);
      ++in_map;
    }
  };
  sweep_pairs<false>(sw, buf, [&](uint32_t n_pr, uint32_t, uint32_t nc, bool central) __attribute__((always_inline)) {
    const ulonglong2* rxy = reinterpret_cast<const ulonglong2*>(buf.rxy);
    const unsigned long long* rz = reinterpret_cast<const unsigned long long*>(buf.rz);
    uint32_t self = 0;
    for (uint32_t h = lane; h < kSweepTile; h += 32) {
      const float4 q = h < nc ? buf.cand[h] : make_float4(INFINITY, INFINITY, INFINITY, 0.f);
      const uint32_t kind = __float_as_uint(q.w);
      const bool both = kind == kCandBoth, flip = !central;  // flip: the candidate is the central end
      self += __popc(__ballot_sync(0xffffffffu, h < nc && kind == kCandSelf));
      const unsigned long long qx = f2_pack(q.x, q.x), qy = f2_pack(q.y, q.y), qz = f2_pack(q.z, q.z);
#pragma unroll 2
      for (uint32_t k = 0; k < n_pr; ++k) {
        const ulonglong2 xy = rxy[k];
        const unsigned long long dx = f2_sub(qx, xy.x), dy = f2_sub(qy, xy.y), dz = f2_sub(qz, rz[k]);
        const unsigned long long d2 =
            f2_fma(f2_fma(f2_mul(dx, dx), one2, f2_mul(dy, dy)), one2, f2_mul(dz, dz));
        const unsigned long long hx = f2_add_down(f2_fma(dx, inv2, hi2), magic2), lx = f2_add_down(f2_fma(dx, inv2, lo2), magic2);
        const unsigned long long hy = f2_add_down(f2_fma(dy, inv2, hi2), magic2), ly = f2_add_down(f2_fma(dy, inv2, lo2), magic2);
        const unsigned long long hz = f2_add_down(f2_fma(dz, inv2, hi2), magic2), lz = f2_add_down(f2_fma(dz, inv2, lo2), magic2);
        const unsigned long long amb = (hx ^ lx) | (hy ^ ly) | (hz ^ lz);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float da, db;
          f2_unpack(d2, da, db);
          if (!((e ? db : da) < sw.range)) continue;
          const int sh = 32 * e;
          const uint32_t mx = (uint32_t)(hx >> sh) - kMagicBits, my = (uint32_t)(hy >> sh) - kMagicBits,
                         mz = (uint32_t)(hz >> sh) - kMagicBits;
          if ((uint32_t)(amb >> sh) == 0u && (a.covers || max(mx, max(my, mz)) < nv)) {
            const uint32_t lin = (mz * nv + my) * nv + mx, mir = N - 1 - lin;
            if (both) {
              atomicAdd(&a.H[max(lin, mir)], lin == mir ? 2ull : 1ull);
              in_map += 2;
            } else {
              alone(flip ? mir : lin, 1ull);
              ++in_map;
            }
          } else {
            float xa, xb, ya, yb, za, zb;
            f2_unpack(dx, xa, xb), f2_unpack(dy, ya, yb), f2_unpack(dz, za, zb);
            const float x = e ? xb : xa, y = e ? yb : ya, z = e ? zb : za;
            if (both || !flip) exact(x, y, z);
            if (both || flip) exact(-x, -y, -z);
          }
        }
      }
    }
    // the staged records met themselves once each, at displacement 0 (inside the map: V[0] < 0 < V[n])
    if (self && lane == 0) {
      const uint32_t c = nv / 2;  // V[c] <= 0 < V[c + 1]
      alone((c * nv + c) * nv + c, 0ull - (unsigned long long)self);
      in_map -= self;
    }
  });
  totals();
}

// lower half of the map: its own counts and those of the mirrored upper half
__global__ void __launch_bounds__(256) k_sdm_mirror(unsigned long long* __restrict__ H, uint32_t N,
                                                    const Geo* __restrict__ ngeo, const Geo* __restrict__ cgeo) {
  griddep_wait();
  griddep_launch();
  if (!sdm_sweep_pays(ngeo->n_sel, ngeo->n_cells, cgeo->n_sel)) return;  // (every displacement was counted where it lies)
  const uint32_t half = N / 2;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < half; i += gridDim.x * blockDim.x) H[i] += H[N - 1 - i];
}

// n_central and the device status into the meta array
__global__ void k_sdm_epilogue(const Geo* __restrict__ ngeo, const Geo* __restrict__ cgeo, uint64_t* meta) {
  griddep_wait();
  griddep_launch();
  if (threadIdx.x == 0) {
    meta[0] = cgeo->n_sel;
    int st = cgeo->status;
    if (st == 0) st = ngeo->status;
    meta[3] = (uint64_t)(uint32_t)st;
  }
}

int run_sdm(ps_grid* g, const float* dsrf, const uint64_t ctr_mask[4], float dsrf_min, ps_sdm_spec spec,
            uint64_t* d_hist, uint64_t* d_meta, cudaStream_t s) {
  const uint64_t nh = (uint64_t)spec.n_vox * spec.n_vox * spec.n_vox;
  ZeroOut z;  // the outputs are zeroed by the central-list reset kernel
  z.p[0] = d_meta;
  z.n[0] = PS_SDM_META_LEN;
  z.p[1] = d_hist;
  z.n[1] = (uint32_t)nh;
  // (a radius or voxel near the limits of float32 keeps the general kernel)
  const bool sym = centrals_in_neighbours(g, ctr_mask) && spec.r_max > 1e-15 && spec.r_max < 1e15 && spec.w > 1e-15 &&
                   spec.w < 1e15;
  int rc = build_central_list(g, dsrf, ctr_mask, dsrf_min, s, z, false, false, !sym, sym ? kSweep : kNoSweep, true);
  if (rc) return rc;
  const float ER = (float)(spec.r_max * spec.r_max);
  SdmArgs a;
  memset(&a, 0, sizeof(a));
  a.nrec = g->nbr.rec;
  a.nstart = g->nbr.start;
  a.ngeo = g->nbr.geo;
  a.crec = g->ctr.rec;
  a.cstart = g->ctr.start;
  a.cwork = g->ctr.work;
  a.witem = g->ctr.witem;
  a.work_cap = g->item_cap;
  a.cgeo = g->ctr.geo;
  a.stencil = g->stencil;
  a.ER = ER;
  a.w = spec.w;
  a.n_vox = spec.n_vox;
  a.H = reinterpret_cast<unsigned long long*>(d_hist);
  a.meta = d_meta;
  if (sym) {
    // |dx| >= V[n] would give dx^2 >= ER
    const double top = (double)(float)((double)spec.n_vox * 0.5 * spec.w);
    a.covers = top * top >= (double)ER;
    SweepArgs sw = sweep_args(g, &g->ctr.geo->sym_next);
    sw.range = ER;
    int per_sm = 0;
    PS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sdm_sym, 256, 0));
    if (per_sm < 1) return fail(PS_ERR_UNSUPPORTED, "SDM kernel does not fit on an SM");
    PS_LAUNCH(PS_KID_SDM, s, PS_CUDA(launch_pdl(k_sdm_sym, g->num_sms * per_sm, 256, 0, s, a, sw)));
    PS_LAUNCH(PS_KID_SDM, s, PS_CUDA(launch_pdl(k_sdm_mirror, g->num_sms * 8, 256, 0, s, a.H, (uint32_t)nh, g->nbr.geo, g->ctr.geo)));
    PS_LAUNCH(PS_KID_EPILOGUE, s, PS_CUDA(launch_pdl(k_sdm_epilogue, 1, 32, 0, s, g->nbr.geo, g->ctr.geo, d_meta)));
    PS_CUDA(cudaGetLastError());
    return PS_OK;
  }
  int per_sm = 0;
  PS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sdm, 256, 0));
  if (per_sm < 1) return fail(PS_ERR_UNSUPPORTED, "SDM kernel does not fit on an SM");
  PS_LAUNCH(PS_KID_SDM, s, PS_CUDA(launch_pdl(k_sdm, g->num_sms * per_sm, 256, 0, s, a)));
  PS_LAUNCH(PS_KID_EPILOGUE, s, PS_CUDA(launch_pdl(k_sdm_epilogue, 1, 32, 0, s, g->nbr.geo, g->ctr.geo, d_meta)));
  PS_CUDA(cudaGetLastError());
  return PS_OK;
}

}  // namespace ps
