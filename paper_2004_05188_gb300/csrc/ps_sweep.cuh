// Sweep over the unordered pairs of neighbour records within a range, shared by the statistics
// whose centrals are neighbour records (RDF, smoothed RDF, spatial distribution map).
//
// An unordered pair {i, j} contributes once per central end (c_i + c_j), and d2_ij == d2_ji bit
// for bit, so each pair is met once, from the lower of its two owner blocks.  An owner block is
// B x-consecutive cells of one row of the grid (B > 1 only where cells hold few records); its
// candidates are its own records and the rows of the half stencil (dz > 0, or dz == 0 and dy > 0,
// or the own row to the right).  A warp works on one block at a time:
//
//   * up to 64 of the block's records (whole sub-cells) are staged in shared memory, centrals and others apart
//     (a block with both is swept twice), so that the weight of a pair depends on the candidate
//     alone and the others' sweep drops the candidates that are not central;
//   * the candidates are read 32 at a time (coalesced) and kept only if they lie within range of
//     the staged records' bounding box.  A half-size cell of edge a = r/2 and its stencil of 125
//     cells span 125 a^3, the points within r of the cell only 84 a^3: a third of the pair tests
//     is never made, at ~45 instructions per 32 candidates (against ~14 per test of 32 pairs);
//   * the kept ones are compacted into tiles of 64, two per lane in registers, and tested against
//     the records (read two at a time by every lane at once).
//
// Blocks that hold more than a warp's share of the work (heavy_block) are listed beforehand in groups of at most
// 64 records, which are units of their own.
// The pairs inside the block are met in both orders, with weight 1 for each central end.
#pragma once

#include "ps_internal.cuh"

namespace ps {

constexpr float kMagic = 12582912.0f;           // 1.5 * 2^23: x + kMagic holds floor(x) in its low bits
constexpr uint32_t kMagicBits = 0x4B400000u;

constexpr uint32_t kSweepRec = kHeavyGroup;  // records staged at a time
constexpr uint32_t kSweepGroup = 64;     // of whole sub-cells
constexpr uint32_t kSweepTile = 64;       // candidates per tile, two per lane
constexpr uint32_t kCandSingle = 0u, kCandBoth = 1u, kCandOwn = 2u, kCandSelf = 3u;

__device__ __forceinline__ float sqrt_fast(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b,
                                                     unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// rounded down: with c = kMagic the floor of a * b in the low bits
__device__ __forceinline__ unsigned long long f2_fma_down(unsigned long long a, unsigned long long b,
                                                          unsigned long long c) {
  unsigned long long r;
  asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

struct SweepArgs {
  const float4* nrec;
  const uint32_t* nstart;
  const uint32_t* nsub; // sub-cell starts (where the cells have sub-cells)
  const uint32_t* pfx;  // central prefix over the neighbour records
  const Geo* ngeo;
  const uint2* heavy;         // groups of the heavy blocks: first record, block (ngeo->n_heavy)
  const uint32_t* heavy_map;  // bit per block: its groups are listed
  uint32_t* next;       // work counter (units taken)
  int stencil;
  float range;          // pairs with d2 < range are in range
  float one;            // 1.0f, opaque to the compiler (see dist2_x2_fma)
  int8_t row_w[49];     // half-width of each stencil row (dy, dz), at [(dz + s)(2s + 1) + dy + s]; -1: none
};

// Row widths of a stencil of s cells for cells of edge h >= r_cut * cs * (1 + 2^-10) (plus the
// grid's rounding margin extent * 2^-20, which covers the float32 rounding of the cell index).
// Two points whose cells are |d| >= 2 apart along an axis are more than (|d| - 1) r_cut cs apart
// along it, so cell offset (dx, dy, dz) can hold a pair within r_cut only if
// sum_i max(0, |d_i| - 1)^2 (cs (1 + 2^-10))^2 < 1; the test keeps a further 2^-20 margin.
// Stencils of three cells (cs < 1/2) lose the 4 far corner cells of each octant; two-cell stencils
// lose corners or rows only for cs above ~0.58.
inline void row_widths(int s, double cs, int8_t* w) {
  const int W = 2 * s + 1;
  const double f = cs * (1.0 + 1.0 / 1024.0), lim = (1.0 + 1.0 / 1048576.0) * (1.0 + 1.0 / 1048576.0);
  auto m2 = [](int d) { const int m = d < 0 ? -d - 1 : d - 1; return m > 0 ? (double)(m * m) : 0.0; };
  for (int dz = -s; dz <= s; ++dz)
    for (int dy = -s; dy <= s; ++dy) {
      int width = -1;
      for (int dx = 0; dx <= s; ++dx)
        if ((m2(dx) + m2(dy) + m2(dz)) * f * f < lim) width = dx;
      w[(dz + s) * W + dy + s] = (int8_t)width;
    }
}

// The arguments over the last build's neighbour records and the central list's prefix over them;
// the caller fills in range.
inline SweepArgs sweep_args(const ps_grid* g, uint32_t* next) {
  SweepArgs a = {};
  a.nrec = g->nbr.rec;
  a.nstart = g->nbr.start;
  a.nsub = g->nbr.count;
  a.pfx = reinterpret_cast<const uint32_t*>(g->cr);  // written by the central-list compaction
  a.ngeo = g->nbr.geo;
  a.heavy = g->heavy;
  a.heavy_map = g->heavy_map;
  a.next = next;
  a.stencil = g->stencil;
  a.one = 1.0f;
  row_widths(g->stencil, g->cell_scale, a.row_w);
  return a;
}

// Per-warp shared memory of the sweep.
struct SweepBuf {
  float4 rxy[kSweepRec / 2];               // staged records as pairs: xa xb ya yb
  float2 rz[kSweepRec / 2];                // za zb
  float4 cand[kSweepTile + 32];            // kept candidates: x, y, z, kind (kCand*) in the low bits of w
  uint32_t cidx[kSweepTile + 32];          // their record numbers (kept when the statistic asks for them)
  uint32_t ridx[kSweepRec];                // record numbers of the staged records (likewise)
};

// Two squared distances as dist2(): packed throughout.  The sums are x * one + y with one = 1.0f
// passed at run time: x * 1 + y rounds once, exactly as x + y does, and the compiler cannot fuse
// the squares into it (a packed add it does fuse).
__device__ __forceinline__ unsigned long long dist2_x2_fma(unsigned long long px, unsigned long long py,
                                                           unsigned long long pz, unsigned long long qx,
                                                           unsigned long long qy, unsigned long long qz,
                                                           unsigned long long one) {
  const unsigned long long dx = f2_sub(qx, px), dy = f2_sub(qy, py), dz = f2_sub(qz, pz);
  return f2_fma(f2_fma(f2_mul(dx, dx), one, f2_mul(dy, dy)), one, f2_mul(dz, dz));
}

// Runs every unit.  tile(n_pr, m, nc, central): the staged records (m of them, n_pr pairs, n_pr even,
// padded with far records), all central or all not, against nc <= 64 candidates in buf.cand.
// INDEX: fill buf.cidx / buf.ridx.  done(m, central) follows the last tile of the staged records.
template <bool INDEX, class Tile, class Done>
__device__ __forceinline__ void sweep_pairs(const SweepArgs& a, SweepBuf& buf, Tile&& tile, Done&& done) {
  const uint32_t lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
  const Geo g = *a.ngeo;
  const int s = a.stencil, W = 2 * s + 1, inv_w = 65536 / W + 1;
  const uint32_t n_warps = gridDim.x * (blockDim.x >> 5);
  // units: S parts of the candidates each for the groups of the heavy blocks and for the blocks
  const uint32_t B = sweep_block(g.n_cells, g.n_sel), nbx = (g.dims[0] + B - 1) / B;
  const uint32_t n_blocks = nbx * g.dims[1] * g.dims[2], S = sweep_parts(n_blocks, n_warps);
  const uint32_t n_heavy = g.n_heavy, n_units = (n_heavy + n_blocks) * S;
  // a record further than this from the box of the staged ones is out of range of each of them
  // (the slack covers the rounding of both float32 distances)
  const float lim = a.range * 1.00001f;
  for (;;) {
    // units per take: a share of those left, so that the warps finish together
    uint32_t base = 0, take = 0;
    if (lane == 0) {
      const uint32_t cur = *reinterpret_cast<volatile uint32_t*>(a.next);
      const uint32_t left = cur < n_units ? n_units - cur : 0u;
      take = cur < n_heavy * S ? 1u : min(32u, max(1u, left / (8 * n_warps)));
      base = atomicAdd(a.next, take);
    }
    base = __shfl_sync(0xffffffffu, base, 0);
    take = __shfl_sync(0xffffffffu, take, 0);
    if (base >= n_units) break;
    // lane i: block (first cell, row) and records of unit base + i
    uint32_t s0 = 0, s1 = 0, ux = 0, uy = 0, uz = 0, upart = 0;
    if (lane < take && base + lane < n_units) {
      const uint32_t u = (base + lane) / S;
      upart = (base + lane) % S;
      uint32_t blk = u - n_heavy;
      if (u < n_heavy) {
        const uint2 e = a.heavy[u];
        s0 = e.x, blk = e.y;
      }
      const uint32_t row = blk / nbx;
      ux = (blk % nbx) * B, uy = row % g.dims[1], uz = row / g.dims[1];
      s1 = a.nstart[row * g.dims[0] + min(ux + B, g.dims[0])];
      if (u < n_heavy)
        s1 = min(s1, s0 + kHeavyGroup);
      else
        s0 = n_heavy && ((a.heavy_map[blk >> 5] >> (blk & 31u)) & 1u) ? s1 : a.nstart[row * g.dims[0] + ux];
    }
    uint32_t todo = __ballot_sync(0xffffffffu, s1 > s0);
    while (todo) {
      const int src_lane = __ffs(todo) - 1;
      todo &= todo - 1u;
      const uint32_t part = __shfl_sync(0xffffffffu, upart, src_lane);
      const uint32_t a0 = __shfl_sync(0xffffffffu, s0, src_lane), a1 = __shfl_sync(0xffffffffu, s1, src_lane);
      // lane r: candidate run r of the block (at most 1 + 3 * 7 + 3 + 1 = 26): the block itself, the
      // rows above (dz > 0, every dy), the rows ahead (dz = 0, dy > 0), the own row to the right:
      // row (ry, rz), cells rx0 .. rx1 (none: rx0 > rx1)
      int ry = (int)__shfl_sync(0xffffffffu, uy, src_lane), rz = (int)__shfl_sync(0xffffffffu, uz, src_lane);
      int rx0 = (int)__shfl_sync(0xffffffffu, ux, src_lane), rx1 = min(rx0 + (int)B, (int)g.dims[0]) - 1;
      {
        const int r = (int)lane - 1, n_up = W * s;
        if (lane > 0) {
          const int q = (r * inv_w) >> 16;  // r / W
          const int dz = r < n_up ? 1 + q : 0, dy = r < n_up ? r - q * W - s : (r < n_up + s ? 1 + r - n_up : 0);
          if (r < n_up + s) {
            const int wd = a.row_w[(dz + s) * W + dy + s];
            rx0 -= wd, rx1 += wd;
            if (wd < 0) rx1 = -1;
          } else {
            rx0 = rx1 + 1, rx1 = r == n_up + s ? rx1 + s : -1;
          }
          ry += dy, rz += dz;
          rx0 = max(rx0, 0), rx1 = min(rx1, (int)g.dims[0] - 1);
          if (ry < 0 || ry >= (int)g.dims[1] || rz >= (int)g.dims[2]) rx1 = -1;
        }
      }
      uint32_t rs = 0, rl = 0, rc = 0;  // first record, length, centrals among them
      if (rx0 <= rx1) {
        const uint32_t rw = ((uint32_t)rz * g.dims[1] + (uint32_t)ry) * g.dims[0];
        rs = a.nstart[rw + rx0];
        rl = a.nstart[rw + rx1 + 1] - rs;
      }
      if (rl) rc = __ldg(a.pfx + rs + rl) - __ldg(a.pfx + rs);
      // Staged together: up to 64 records; with sub-cells (one cell per block then) an aligned power of two of
      // them, so that the records' box is a small one (64 records from where the last ones ended spread over
      // twice as many octants).  RDF with in-range counts, 1e5 cylinder on 2 nm cells 0.308 -> 0.267 ms;
      // smoothed forward, 2e5 cylinder 0.87 -> 0.79 ms; at most 32 or 48 records: 0.271 and 0.269, but
      // 9e5 ions on 1.5 nm cells 1.36 and 1.15 against 1.12 ms.
      const uint32_t f0 = ((__shfl_sync(0xffffffffu, uz, src_lane) * g.dims[1] + __shfl_sync(0xffffffffu, uy, src_lane)) *
                               g.dims[0] + __shfl_sync(0xffffffffu, ux, src_lane)) << (3 * g.sub);
      // (a group of a heavy block is staged as it is)
      uint32_t q = 0, qe = g.sub && a1 - a0 > kSweepGroup ? a0 : a1, g1;
      for (uint32_t g0 = a0; g0 < a1; g0 = g1) {
        while (qe == g0) {  // the next sub-cells: lane l proposes 2^l of them
          const uint32_t w = 1u << min(lane, 6u), q1 = q + w, nq = 1u << (3 * g.sub);
          const bool ok = lane <= 3 * g.sub && (q & (w - 1u)) == 0u;
          const uint32_t e = ok && q1 < nq ? __ldg(a.nsub + f0 + q1) : a1;
          const uint32_t pick = 31 - __clz(__ballot_sync(0xffffffffu, ok && (e - g0 <= kSweepGroup || lane == 0)));
          qe = __shfl_sync(0xffffffffu, e, pick);
          q += 1u << pick;
        }
        g1 = min(g0 + kSweepRec, qe);
        const uint32_t n_ctr = __ldg(a.pfx + g1) - __ldg(a.pfx + g0);
        for (uint32_t central = 0; central < 2; ++central) {
          const uint32_t m = central ? n_ctr : (g1 - g0) - n_ctr;
          if (m == 0) continue;
          // stage the records of this kind as pairs, and their box
          float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
          float* sxy = reinterpret_cast<float*>(buf.rxy);
          float* sz = reinterpret_cast<float*>(buf.rz);
          const uint32_t n_pr = (m + 3) >> 2 << 1;
          __syncwarp();
          uint32_t at = 0;
#pragma unroll
          for (uint32_t h = 0; h < kSweepRec; h += 32) {
            const uint32_t j = g0 + h + lane;
            bool in = false;
            float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j < g1) {
              q = __ldg(a.nrec + j);
              in = (__ldg(a.pfx + j + 1) - __ldg(a.pfx + j)) == central;
            }
            const uint32_t bal = __ballot_sync(0xffffffffu, in);
            if (in) {
              const uint32_t r = at + __popc(bal & lt);
              float* d = sxy + (r >> 1) * 4 + (r & 1u);
              d[0] = q.x, d[2] = q.y, sz[r] = q.z;
              if (INDEX) buf.ridx[r] = j;
              lo[0] = fminf(lo[0], q.x), hi[0] = fmaxf(hi[0], q.x);
              lo[1] = fminf(lo[1], q.y), hi[1] = fmaxf(hi[1], q.y);
              lo[2] = fminf(lo[2], q.z), hi[2] = fmaxf(hi[2], q.z);
            }
            at += __popc(bal);
          }
          if (m + lane < 2 * n_pr) {  // the pad records (at most 3) never hit
            const uint32_t r = m + lane;
            float* d = sxy + (r >> 1) * 4 + (r & 1u);
            d[0] = INFINITY, d[2] = INFINITY, sz[r] = INFINITY;
          }
          float mid[3], half[3];
#pragma unroll
          for (int ax = 0; ax < 3; ++ax) {
            const float l = key2f(__reduce_min_sync(0xffffffffu, f2key(lo[ax])));
            const float h = key2f(__reduce_max_sync(0xffffffffu, f2key(hi[ax])));
            mid[ax] = 0.5f * (l + h);  // the box as mid +- half, half rounded up
            half[ax] = fmaxf(h - mid[ax], mid[ax] - l) * 1.000001f + fabsf(mid[ax]) * 2.4e-7f;
          }
          // records that are not central pair with the central candidates of the other blocks only
          uint32_t mask = __ballot_sync(0xffffffffu, rl != 0u && (central || (rc != 0u && lane != 0u)));
          __syncwarp();

          // the chunks of 32 records of the runs; part p of S takes every S-th chunk
          uint32_t o = 32u * part, src = 0, len = 0, cen = 0, run = 0;
          auto advance = [&]() -> bool {  // to the run of the next chunk (uniform)
            while (o >= ((len + 31u) & ~31u)) {
              if (!mask) return false;
              o -= (len + 31u) & ~31u;
              run = __ffs(mask) - 1;
              mask &= mask - 1u;
              src = __shfl_sync(0xffffffffu, rs, run);
              len = __shfl_sync(0xffffffffu, rl, run);
              cen = __shfl_sync(0xffffffffu, rc, run);
            }
            return true;
          };
          // kind of a candidate of the chunk, and whether it can count at all: kCandBoth when both
          // ends are central; the block's own records with weight 1 in each order
          float4 nq = make_float4(0.f, 0.f, 0.f, 0.f);
          uint32_t nj = 0, nkind = 0;
          bool nok = false;
          auto load = [&]() {
            nj = src + o + lane;
            nok = o + lane < len;
            uint32_t c = cen == len;
            if (nok) {
              nq = __ldg(a.nrec + nj);
              if (cen != len && cen != 0u) c = __ldg(a.pfx + nj + 1) - __ldg(a.pfx + nj);
            }
            nok = nok && (central | c) != 0u;
            nkind = (central & c) ? kCandBoth : kCandSingle;
            if (run == 0) nkind = (c && nj >= g0 && nj < g1) ? kCandSelf : kCandOwn;
          };
          uint32_t nc = 0;
          bool more = advance();
          if (more) load();
          while (more || nc) {
            if (more) {
              const float4 q = nq;
              const uint32_t j = nj;
              uint32_t kind = nkind;
              const bool ok = nok;
              o += 32u * S;
              more = advance();
              if (more) load();
              const float ex = fmaxf(fabsf(q.x - mid[0]) - half[0], 0.f);
              const float ey = fmaxf(fabsf(q.y - mid[1]) - half[1], 0.f);
              const float ez = fmaxf(fabsf(q.z - mid[2]) - half[2], 0.f);
              const bool keep = ok && __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, ex * ex)) < lim;
              const uint32_t bal = __ballot_sync(0xffffffffu, keep);
              if (keep) {
                const uint32_t slot = nc + __popc(bal & lt);
                // (a record with an infinite or NaN coordinate does not meet itself at distance 0)
                if (kind == kCandSelf && !(dist2(q.x, q.y, q.z, q.x, q.y, q.z) == 0.f)) kind = kCandOwn;
                buf.cand[slot] = make_float4(q.x, q.y, q.z, __uint_as_float(kind));
                if (INDEX) buf.cidx[slot] = j;
              }
              nc += __popc(bal);
            }
            if (nc >= kSweepTile || !more) {
              if (nc == 0) break;
              const uint32_t nt = min(nc, kSweepTile);
              __syncwarp();
              tile(n_pr, m, nt, central != 0u);
              __syncwarp();
              nc -= nt;  // at most 31 candidates move to the front
              if (lane < nc) {
                buf.cand[lane] = buf.cand[kSweepTile + lane];
                if (INDEX) buf.cidx[lane] = buf.cidx[kSweepTile + lane];
              }
              __syncwarp();
            }
          }
          done(m, central != 0u);
        }
      }
    }
  }
}

template <bool INDEX, class Tile>
__device__ __forceinline__ void sweep_pairs(const SweepArgs& a, SweepBuf& buf, Tile&& tile) {
  sweep_pairs<INDEX>(a, buf, tile, [](uint32_t, bool) {});
}

}  // namespace ps
