// Exact kNN + RDF query over the cell grid.
//
// The paper evaluates one spherical ROI per central ion and machines the ROIs
// off with a dynamic schedule, each thread keeping its own result buffers that
// are merged afterwards (Suppl. "Customized user defined batch processing
// queues").  Here the ROIs of one cell of the grid share their candidates: the
// cells within `stencil` cells of it (27 cells for cells of edge >= r_cut, 125
// for cells of edge >= r_cut/2, up to 343 for r_cut/3, less the cells that
// cannot hold a pair within r_cut), read as x-contiguous runs of sorted records.
// Dense grids keep a cell's records ordered by sub-cells, whose x-rods are then the
// runs.  Persistent kernels take work from device counters (the dynamic schedule):
//
//   k_query_warp   heavy items = (cell with >= 16 centrals, batch of <= 32 of
//                  them): the candidates within reach of the box around the
//                  item's centrals go through a per-warp shared ring
//                  (item_scan), each lane holds one central (or shares one) and
//                  walks the ring (shared-memory broadcast).  Light items
//                  (sparser cells) are taken 32 at a time and each of their
//                  centrals gets one thread that walks its own stencil.
//   k_rdf_sym      the RDF, and the in-range counts, over unordered pairs of
//                  neighbour records: where every central is one, the cloud is
//                  dense and the centrals are many (sweep_pays), or in passes.
//   k_query_cta    for cells with >= dense_min centrals (an option): one CTA per
//                  cell; the runs are staged into shared memory with bulk
//                  asynchronous copies (cp.async.bulk, completion on an mbarrier)
//                  and one thread per central walks them.
//
// Each thread keeps the k smallest squared distances in registers (sorted
// insertion).  Counts go to per-CTA shared-memory histograms (the per-thread
// buffers) added to the uint64 global histograms when the CTA finishes.
//
// The query in passes (ps_grid_opts.split): k_knn_vertex, the near kNN pass (the
// centrals sorted by the vertex-centred grid, each item against the 2 x 2 x 2
// cells around its vertex; k_query_warp on third-size cells), k_knn_list (the
// full-radius kNN of the centrals that pass lists) and k_rdf_sym.
#include <cstring>
#include <vector>

#include "ps_internal.cuh"
#include "ps_items.cuh"
#include "ps_sweep.cuh"

namespace ps {

struct QueryArgs {
  const float4* nrec;
  const uint32_t* nstart;
  const uint32_t* nsub;  // sub-cell starts (where the cells have sub-cells)
  const Geo* ngeo;
  const float4* crec;
  const uint32_t* cstart;
  const uint32_t* cwork;
  const uint2* witem;
  const uint2* whi;   // very heavy items (taken before those of witem)
  uint32_t work_cap;  // capacity of witem (light items grow from its end)
  Geo* cgeo;
  int stencil;
  double r0, dr;
  uint32_t n_bins;
  uint32_t n_k;
  uint32_t k_need;     // max requested k
  uint32_t stage_cap;  // float4 records per staging chunk (CTA kernel)
  uint32_t ks[PS_MAX_KLIST];
  uint64_t* rdf;
  uint64_t* knn;
  uint64_t* meta;
  float* kth;
  uint32_t* nwithin;
  int64_t n;  // ions in the cloud (stride of kth)
  // passes of the split query (zero / null for the combined one)
  float emax_near;        // > 0: kNN within this squared range only; a central with fewer than k_need
                          // neighbours there is marked in need[] instead of being counted
  uint32_t* need;         // per central record: 1 = needs the full-radius search (near pass writes it)
  int fallback;           // 1: only the centrals marked in need[] (the full-radius kNN pass)
  uint32_t* next_front;   // work counters of the front (heavy) and back (light) items
  uint32_t* next_light;
  // whether a central is among its own candidates: every one (self_all), or by its type
  int self_all;
  const uint8_t* type;
  Mask nbr;
  float one;  // 1.0f, opaque to the compiler (see dist2_x2_fma)
  int sweep;  // 1: the RDF of a dense cloud is left to k_rdf_sym (see sweep_pays)
  // bin lookup table (lut_shift = 0: none): cell c covers the float32 bit patterns
  // [(lut_base + c) << lut_shift, (lut_base + c + 1) << lut_shift), at most one interior edge each
  uint32_t lut_shift, lut_base, lut_n;
  // half-width of each stencil row (dy, dz), at [(dz + s) (2s + 1) + dy + s]: the row's cells
  // cx - w .. cx + w can hold a record within r_cut of the cell's records, the others cannot
  // (-1: none); w = s unless the cell is small against r_cut (see row_widths)
  int8_t row_w[kMaxRuns];
};

__device__ __forceinline__ Search search_of(const QueryArgs& a) { return Search{a.nrec, a.nstart, a.nsub, a.stencil, a.row_w}; }

struct SmemLayout {
  uint32_t off_E, off_lut, off_rdf, off_knn, off_kmeta, off_stage, total;
  bool priv;
};

constexpr uint32_t kLutMax = 4096;  // entries of the bin lookup table (uint32)

constexpr uint32_t kPrivBins = 512;  // up to this many bins each warp keeps its own 32-bit RDF row

__host__ __device__ inline SmemLayout smem_layout(uint32_t n_bins, uint32_t n_k, bool rdf, uint32_t stage_cap,
                                                  bool allow_priv = false, uint32_t lut_n = 0) {
  SmemLayout L;
  uint32_t o = 0;
  L.priv = allow_priv && rdf && n_bins <= kPrivBins;
  L.off_E = o;
  o += (n_bins + 1) * 4;
  L.off_lut = o;
  o += rdf ? lut_n * 4 : 0;
  o = (o + 7u) & ~7u;
  L.off_rdf = o;
  o += rdf ? (L.priv ? 8 * (n_bins + 1) * 4 : n_bins * 8) : 0;  // (bin n_bins: see FastBins)
  o = (o + 7u) & ~7u;
  L.off_knn = o;
  o += n_k * n_bins * 4;
  L.off_kmeta = o;
  o += n_k * 2 * 4;
  o = (o + 15u) & ~15u;
  L.off_stage = o;
  o += stage_cap * 16;
  L.total = o;
  return L;
}

// Per-CTA result buffers in shared memory.
template <bool RDF>
struct Hist {
  float* sE;
  unsigned long long* s_rdf;  // CTA row, 64-bit: per-CTA pair counts can pass 2^32 on large clouds
  // or one 32-bit row per warp (priv), flushed by its warp before it could pass 2^31; bin 0 may stand
  // below zero between a flush and the removal of the centrals that met themselves
  uint32_t* s_rdfw;
  bool priv;
  uint32_t* s_knn;            // per-CTA central counts stay below n < 2^32
  uint32_t* s_kmeta;
  uint32_t* lut;              // bin lookup table (see QueryArgs)
  uint32_t lut_shift, lut_base, lut_mask;
  float Emax, E0, r0f, inv_dr;
  uint32_t nb;

  __device__ void init(const QueryArgs& a, unsigned char* smem, uint32_t stage_cap, bool allow_priv = false) {
    const SmemLayout L = smem_layout(a.n_bins, a.n_k, RDF, stage_cap, allow_priv, a.lut_n);
    sE = reinterpret_cast<float*>(smem + L.off_E);
    lut = reinterpret_cast<uint32_t*>(smem + L.off_lut);
    lut_shift = RDF ? a.lut_shift : 0u;
    lut_base = a.lut_base;
    lut_mask = (1u << lut_shift) - 1u;
    priv = L.priv;
    s_rdf = reinterpret_cast<unsigned long long*>(smem + L.off_rdf);
    s_rdfw = reinterpret_cast<uint32_t*>(smem + L.off_rdf) + (threadIdx.x >> 5) * (a.n_bins + 1);
    s_knn = reinterpret_cast<uint32_t*>(smem + L.off_knn);
    s_kmeta = reinterpret_cast<uint32_t*>(smem + L.off_kmeta);
    nb = a.n_bins;
    // edge table: the same double formula as the host, E[b] = (float)((r0 + b*dr)^2)
    for (uint32_t b = threadIdx.x; b <= nb; b += blockDim.x) {
      const double e = __dadd_rn(a.r0, __dmul_rn((double)b, a.dr));
      sE[b] = __double2float_rn(__dmul_rn(e, e));
    }
    if (RDF) {
      if (priv)
        for (uint32_t b = threadIdx.x; b < 8 * (nb + 1); b += blockDim.x) reinterpret_cast<uint32_t*>(s_rdf)[b] = 0;
      else
        for (uint32_t b = threadIdx.x; b < nb; b += blockDim.x) s_rdf[b] = 0ull;
    }
    for (uint32_t b = threadIdx.x; b < a.n_k * nb; b += blockDim.x) s_knn[b] = 0;
    for (uint32_t b = threadIdx.x; b < 2 * a.n_k; b += blockDim.x) s_kmeta[b] = 0;
    __syncthreads();
    if (RDF && lut_shift) {
      // entry c = b0 << 17 | off: b0 the largest b < nb with E[b] <= the smallest value of cell c
      // (0 below E[0]); off the low lut_shift bits of the next interior edge E[b0 + 1] if it lies
      // in the cell (at most one does), else 2^16, above every low part
      for (uint32_t c = threadIdx.x; c < a.lut_n; c += blockDim.x) {
        const uint32_t c0 = (lut_base + c) << lut_shift;
        const float v = __uint_as_float(c0);
        uint32_t lo = 0, hi = nb;  // invariant: E[lo] <= v or lo == 0; E[hi] > v or hi == nb
        while (hi - lo > 1) {
          const uint32_t mid = (lo + hi) >> 1;
          if (sE[mid] <= v)
            lo = mid;
          else
            hi = mid;
        }
        uint32_t off = 1u << 16;
        if (lo + 1 < nb) {
          const uint32_t e = __float_as_uint(sE[lo + 1]);
          if (e >= c0 && e - c0 <= lut_mask) off = e & lut_mask;
        }
        lut[c] = lo << 17 | off;
      }
      __syncthreads();
    }
    Emax = sE[nb];
    E0 = sE[0];
    r0f = (float)a.r0;
    inv_dr = (float)(1.0 / a.dr);
  }

  // bin b in [0, nb) with E[b] <= d2 < E[b+1] for E[0] <= d2 < E[nb]: from the lookup table (the
  // cell of d2's bit pattern holds at most one interior edge, so the bin is the entry or the next
  // one), else from an approximate square root checked against the edges
  // (d2 >= 0 below E[nb]; the table's first cell lies wholly below E[1], so values below the
  // table take its entry, bin 0)
  __device__ __forceinline__ uint32_t bin(float d2) const {
    if (lut_shift) {
      const uint32_t u = __float_as_uint(d2);
      const uint32_t e = lut[max((int32_t)(u >> lut_shift) - (int32_t)lut_base, 0)];
      return (e >> 17) + ((u & lut_mask) >= (e & 0x1FFFFu) ? 1u : 0u);
    }
    return bin_index(d2, sE, nb, r0f, inv_dr);
  }

  // one in-range pair (d2 < Emax) of weight w: the RDF bin, or the count below E[0].  The pairs
  // binned are not counted here: the flushes add the rows' sums to the meta array.
  __device__ __forceinline__ void pair_w(float d2, uint32_t w, uint32_t& below) {
    if (!RDF) return;
    if (E0 == 0.f && priv) {  // r0 = 0: every pair (d2 >= 0) is binned (uniform branch)
      atomicAdd(&s_rdfw[bin(d2)], w);
      return;
    }
    const bool in = d2 >= E0;
    const uint32_t b = bin(in ? d2 : E0);
    if (priv)
      atomicAdd(&s_rdfw[b], in ? w : 0u);
    else
      atomicAdd(&s_rdf[b], (unsigned long long)(in ? w : 0u));
    below += in ? 0u : w;
  }
  __device__ __forceinline__ void pair(const QueryArgs& a, float d2, uint32_t& below) { pair_w(d2, 1u, below); }

  // one in-range pair of weight w counted straight into the global histogram (and into binned)
  __device__ __forceinline__ void pair_global(const QueryArgs& a, float d2, uint32_t w, uint64_t& binned,
                                              uint32_t& below) {
    if (!RDF) return;
    if (d2 >= E0) {
      atomicAdd((unsigned long long*)&a.rdf[bin(d2)], (unsigned long long)w);
      binned += w;
    } else {
      below += w;
    }
  }

  // the k-th distance D of one central for the q-th requested k
  __device__ __forceinline__ void kth(const QueryArgs& a, uint32_t q, float D, uint32_t idx) {
    if (a.kth) a.kth[(int64_t)q * a.n + idx] = D;
    uint32_t* sp;
    if (!(D < Emax))
      sp = &s_kmeta[2 * q];
    else if (D < E0)
      sp = &s_kmeta[2 * q + 1];
    else
      sp = &s_knn[q * nb + bin_index(D, sE, nb, r0f, inv_dr)];
    atomicAdd(sp, 1u);
  }

  // one warp adds its private RDF row to the global histogram (and its sum to the pair count)
  // and clears it
  __device__ void flush_warp(const QueryArgs& a) {
    if (!RDF || !priv) return;
    __syncwarp();
    unsigned long long tot = 0;
    for (uint32_t b = threadIdx.x & 31; b < nb; b += 32)
      if (s_rdfw[b]) {
        const unsigned long long v = (unsigned long long)(long long)(int32_t)s_rdfw[b];
        tot += v;
        atomicAdd((unsigned long long*)&a.rdf[b], v);
        s_rdfw[b] = 0;
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if ((threadIdx.x & 31) == 0 && tot) atomicAdd((unsigned long long*)&a.meta[PS_META_N_PAIRS], tot);
    __syncwarp();
  }

  // add the shared counters to the global histograms and clear them (whole CTA); the
  // per-warp rows are summed in the CTA first, one global atomic per bin and CTA
  __device__ void flush(const QueryArgs& a) {
    __syncthreads();
    unsigned long long tot = 0;  // pairs binned in this CTA's rows
    if (RDF && priv) {
      uint32_t* rows = reinterpret_cast<uint32_t*>(s_rdf);
      const uint32_t nw = blockDim.x >> 5;
      for (uint32_t b = threadIdx.x; b < nb; b += blockDim.x) {
        unsigned long long sum = 0;
        for (uint32_t w = 0; w < nw; ++w) sum += (unsigned long long)(long long)(int32_t)rows[w * (nb + 1) + b], rows[w * (nb + 1) + b] = 0;
        if (sum) atomicAdd((unsigned long long*)&a.rdf[b], sum);
        tot += sum;
      }
    }
    if (RDF && !priv)
      for (uint32_t b = threadIdx.x; b < nb; b += blockDim.x)
        if (s_rdf[b]) tot += s_rdf[b], atomicAdd((unsigned long long*)&a.rdf[b], s_rdf[b]), s_rdf[b] = 0;
    if (RDF) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
      if ((threadIdx.x & 31) == 0 && tot) atomicAdd((unsigned long long*)&a.meta[PS_META_N_PAIRS], tot);
    }
    for (uint32_t b = threadIdx.x; b < a.n_k * nb; b += blockDim.x)
      if (s_knn[b]) atomicAdd((unsigned long long*)&a.knn[b], (unsigned long long)s_knn[b]), s_knn[b] = 0;
    for (uint32_t b = threadIdx.x; b < 2 * a.n_k; b += blockDim.x)
      if (s_kmeta[b])
        atomicAdd((unsigned long long*)&a.meta[PS_META_HEAD + b], (unsigned long long)s_kmeta[b]), s_kmeta[b] = 0;
    __syncthreads();
  }
};

// pair counters of the whole CTA (every thread calls it): summed in the warp, then in shared
// memory, one global atomic per counter and CTA
__device__ __forceinline__ void add_pair_counters(const QueryArgs& a, uint64_t binned, uint64_t below) {
  // binned: only the pairs counted straight into the global histogram (the shared rows' pairs
  // are added by the flushes); below: pairs with d2 < E[0]
  __shared__ unsigned long long s_pc[2];
  if (threadIdx.x == 0) s_pc[0] = 0, s_pc[1] = 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    binned += __shfl_xor_sync(0xffffffffu, binned, o);
    below += __shfl_xor_sync(0xffffffffu, below, o);
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    if (binned) atomicAdd(&s_pc[0], (unsigned long long)binned);
    if (below) atomicAdd(&s_pc[1], (unsigned long long)below);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_pc[0]) atomicAdd((unsigned long long*)&a.meta[PS_META_N_PAIRS], s_pc[0]);
    if (s_pc[1]) atomicAdd((unsigned long long*)&a.meta[PS_META_N_BELOW], s_pc[1]);
  }
}

// Near kNN pass of the query in passes (vertex != 0): the central list is sorted by the grid
// of cells centred on the vertices of the neighbour grid (vg: origin half a cell lower, one more
// cell per axis), so the centrals of item cell c are those nearest to vertex V = c's coordinates,
// and the 2 x 2 x 2 neighbour cells V - 1 .. V along each axis hold every record within half a
// cell of each of them: 4 rows of 2 cells, ~8 cells of candidates instead of the 27 around a
// central's cell.  Run r < 4 of that block:
__device__ __forceinline__ void vertex_run(const QueryArgs& a, const Geo& ng, const Geo& vg, uint32_t c, uint32_t r,
                                           uint32_t& src, uint32_t& len) {
  src = 0;
  len = 0;
  if (r >= 4) return;
  const int vx = (int)(c % vg.dims[0]), vy = (int)((c / vg.dims[0]) % vg.dims[1]), vz = (int)(c / (vg.dims[0] * vg.dims[1]));
  const int y = vy - 1 + (int)(r & 1u), z = vz - 1 + (int)(r >> 1);
  const int xlo = max(vx - 1, 0), xhi = min(vx, (int)ng.dims[0] - 1);
  if (y < 0 || z < 0 || y >= (int)ng.dims[1] || z >= (int)ng.dims[2] || xlo > xhi) return;
  const uint32_t row = ((uint32_t)z * ng.dims[1] + (uint32_t)y) * ng.dims[0];
  src = a.nstart[row + xlo];
  len = a.nstart[row + xhi + 1] - src;
}

// The squared reach of central p in vertex cell c: the distance from p to the nearest face of
// its block (cells V - 1 and V along each axis, faces at u = V - 1 and u = V + 1 in the
// neighbour grid's cell coordinate u = (x - origin) * inv_h), less a slack for the float32
// rounding of the cell coordinates of p and of any record (a few ulps of u, below slack cells),
// times the cell edge, shrunk by 2^-12 before and after squaring: every record outside the
// block has d2 above it, so a k-th distance below it is the k-th distance over the whole cloud.
// Capped at E[nb].
__device__ __forceinline__ float vertex_reach(const Geo& ng, const Geo& vg, uint32_t c, const float4& p, float slack,
                                              float h_eff, float Emax) {
  const uint32_t v[3] = {c % vg.dims[0], (c / vg.dims[0]) % vg.dims[1], c / (vg.dims[0] * vg.dims[1])};
  const float pc[3] = {p.x, p.y, p.z};
  float m = INFINITY;
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const float u = __fmul_rn(__fsub_rn(pc[ax], ng.origin[ax]), ng.inv_h);
    m = fminf(m, fminf(__fsub_rn(u, (float)v[ax] - 1.0f), __fsub_rn((float)v[ax] + 1.0f, u)));
  }
  const float r = __fmul_rn(fmaxf(__fsub_rn(m, slack), 0.0f), h_eff);
  return fminf(__fmul_rn(__fmul_rn(r, r), 1.0f - 1.0f / 4096.0f), Emax);
}

// Lists the centrals (positions in the central list) of the lanes with miss set, warp-aggregated
// (all 32 lanes call it).
__device__ __forceinline__ void list_append(const QueryArgs& a, bool miss, uint32_t pos, uint32_t lane) {
  const uint32_t m = __ballot_sync(0xffffffffu, miss);
  if (!m) return;
  uint32_t at = 0;
  if (lane == 0) at = atomicAdd(&a.cgeo->list_n, (uint32_t)__popc(m));
  at = __shfl_sync(0xffffffffu, at, 0);
  if (miss) a.need[at + __popc(m & ((1u << lane) - 1u))] = pos;
}

__device__ __forceinline__ float4 far_record() { return make_float4(INFINITY, INFINITY, INFINITY, __uint_as_float(~0u)); }

// ---------------------------------------------------------------------------
// warp kernel
//   heavy items (cells with at least kHeavy centrals or more than kSparseCand candidates, batches of up
//     to 32 centrals): one to sixteen lanes per central (item_lanes).  The candidates are read 64 at
//     a time, the stencil's rows nearest first, and kept only within range of the bounding box of the item's centrals (the
//     histogram's range, or for kNN alone the largest k-th distance so far); the kept ones are
//     compacted into a ring of 128 in shared memory as interleaved pairs and tested 32 or 64 at a
//     time, two per packed test.  Candidates further from the box than every current k-th distance skip
//     the kNN part of the test.
//   light items (the other cells with centrals): the warp takes 32 items at a
//     time and gives each of their centrals a thread of its own that walks its
//     own stencil (the records of neighbouring centrals' cells hit in L1).
// ---------------------------------------------------------------------------
constexpr uint32_t kRowLaneCap = 1u << 25;     // per-central increments of the 32-bit warp row, then global
constexpr int kNoRdf = 0, kRdfGeneral = 1, kRdfDirect = 2;

// Bound by instruction issue, and on small or clustered clouds by the chain of one item.  Where the
// RDF is left to the sweep (a.sweep, dense clouds) only the kNN is done here: k = 10, 1e5-ion
// cylinder, 2 nm cells, 0.325 ms walking every record of the 27 cells, 0.163 ms with the sub-cells out of
// reach left out.  Sparse neighbours (3e6-ion needle, Al about Sc, RDF and k = 10: 0.354 ms, before 0.494):
// 75 instructions per 32 tests, of which the bins take 16, the near tests 18, the insertions 17.
// Near candidates are tested a second time for the queue: one loop for both spills at 64 registers
// (0.347 ms there, but 0.174 -> 0.193 ms where the kNN is alone).  In-range counts without the RDF are
// taken beside the kNN (5e5-ion needle, k = 16, r = 1 nm: 0.511 -> 0.456 ms).  Lists of more than 12, and the
// lists of 8 and more lanes, stop at the tighter bound over a central's lanes (5e4 ions, k = 32: 0.126 -> 0.117 ms;
// shorter lists of few lanes: it costs what it saves); those of up to 16 run 3 CTAs per SM (3e6-ion needle, Al about Sc, k = 16: 0.447 -> 0.406 ms),
// longer ones 2 (5e5-ion needle, k = 32: 0.757 against 0.783 ms with 3).
template <int KMAX, int MODE>
__global__ void __launch_bounds__(256, KMAX <= 12 ? 4 : (KMAX <= 16 ? 3 : 2)) k_query_warp(const __grid_constant__ QueryArgs a) {
  constexpr bool RDF = MODE != kNoRdf;
  griddep_wait();
  griddep_launch();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float4 s_buf[8][kRing];            // per warp: ring of kept candidates, as interleaved pairs
  __shared__ float s_kq[8][32 * kHalf + 32];    // per warp: kNN insertion queue, [slot][lane] + a spare row
  constexpr int KK = KMAX > 0 ? KMAX : 1;
  const bool swept = a.sweep && sweep_pays(*a.ngeo, *a.cgeo);  // RDF and in-range counts are the sweep's
  if (KMAX == 0 && swept) return;                              // nothing is left to do here
  Hist<RDF> H{};
  H.init(a, smem, 0, true);
  FastBins fb;
  if (MODE == kRdfDirect) fb.init(a.n_bins, a.dr, H.sE);
  const uint32_t row_base = smem_u32(H.s_rdfw) - 4u * kMagicBits;
  const unsigned long long one2 = f2_pack(a.one, a.one);
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t wcount = 0;  // increments of this warp's private row since its last flush (uniform)
  const Geo ng = *a.ngeo;
  const uint32_t n_hi = a.cgeo->work_n4, n_front = n_hi + a.cgeo->work_n2, n_light = a.cgeo->work_n3;
  const Search S = search_of(a);
  const float u_slack = item_slack(ng);
  const bool rdf_here = RDF && !swept;
  uint32_t* const nwithin = swept ? nullptr : a.nwithin;
  const float erange = a.emax_near > 0.f ? a.emax_near : H.Emax;  // squared search range of this pass
  uint64_t my_binned = 0;  // pairs counted straight into the global histogram
  uint32_t my_below = 0;   // pairs below E[0]
  float* bf = reinterpret_cast<float*>(s_buf[w]);
  float* kq = s_kq[w];
  const uint32_t q0 = smem_u32(kq + lane);

  // ---- items from the front: dense cells, the very heavy ones first ----
  for (;;) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(a.next_front, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_front) break;
    const uint2 it = item < n_hi ? a.whi[item] : a.witem[item - n_hi];
    const uint32_t c = it.x, first = it.y >> 6, cnt = it.y & 63u;
    const uint32_t c0 = a.cstart[c] + first;
    // L lanes per central (items of dense clusters, small clouds, a cell's partial last item): lane
    // sub of a central tests the pairs t = sub mod L
    const uint32_t L = item_lanes(cnt);
    const uint32_t lg = 31u - __clz(L);
    const uint32_t sub = lane & (L - 1u), ci = lane >> lg;
    bool valid = ci < cnt;
    if (a.fallback && valid) valid = a.need[c0 + ci] != 0u;
    if (a.fallback && __ballot_sync(0xffffffffu, valid) == 0u) continue;  // no central of this item to redo
    // lanes without a central never hit (their distances are infinite or NaN)
    float4 p = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    if (valid) p = a.crec[c0 + ci];
    const uint32_t pidx = valid ? __float_as_uint(p.w) : ~0u;
    const float emax = erange;
    const unsigned long long px = f2_pack(p.x, p.x), py = f2_pack(p.y, p.y), pz = f2_pack(p.z, p.z);
    ItemBox box;
    box.set(p, valid, ng, u_slack);
    float top[KK];
#pragma unroll
    for (int t = 0; t < KK; ++t) top[t] = INFINITY;
    uint32_t within = 0;
    // bound of the kNN insertions: the range and the k-th distance of the lane's central
    float thr = KMAX > 0 ? emax : -INFINITY;
    float near_max = fmaxf(thr, 0.f);  // the largest over the warp
    const bool all = rdf_here || nwithin != nullptr;  // every in-range pair counts, not the nearest alone
    // items whose lanes share centrals take 64 candidates at a time, so that each lane has enough of them
    const uint32_t nb = L > 1u ? 64u : 32u;
    ItemRing ring{bf, 0, 0, 0};

    // tests the nb ring slots from the head, of which n hold candidates
    auto batch = [&](uint32_t n) __attribute__((always_inline)) {
      const ulonglong2* rp = reinterpret_cast<const ulonglong2*>(bf) + (ring.head & (kRing - 1u));
      const uint32_t n_pr = (n + 1) >> 1;
      const bool near = KMAX > 0 && (int32_t)(ring.near_to - ring.head) > 0;
      // without the RDF the near candidates' in-range counts are taken where their kNN is
      if (all && !(MODE == kNoRdf && near)) {
        // two pairs of candidates at a time (beyond the last there are far ones to the end of the batch)
        const ulonglong2 *pa = rp + 2 * sub, *pb = pa + 2 * L;
#pragma unroll 1
        for (uint32_t t0 = 0; t0 < n_pr; t0 += 2 * L, pa += 4 * L, pb += 4 * L) {
          const ulonglong2 xy0 = pa[0], xy1 = pb[0];
          const unsigned long long z0 = pa[1].x, z1 = pb[1].x;
          const unsigned long long d20 = dist2_x2_fma(px, py, pz, xy0.x, xy0.y, z0, one2);
          const unsigned long long d21 = dist2_x2_fma(px, py, pz, xy1.x, xy1.y, z1, one2);
          float d[4];
          f2_unpack(d20, d[0], d[1]);
          f2_unpack(d21, d[2], d[3]);
          if (MODE == kRdfDirect && rdf_here) {
            const uint32_t x = fb.count2(d20, row_base) | fb.count2(d21, row_base);
            if (__any_sync(0xffffffffu, x != 0u)) {
              fb.settle2(d20, row_base);
              fb.settle2(d21, row_base);
            }
          }
          if (MODE == kRdfGeneral && rdf_here) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (d[e] < emax && __float_as_uint(reinterpret_cast<const float*>(e < 2 ? pa : pb)[6 + (e & 1)]) != pidx)
                H.pair(a, d[e], my_below);
          }
          if (nwithin != nullptr)
            within += (uint32_t)(d[0] < emax) + (uint32_t)(d[1] < emax) + (uint32_t)(d[2] < emax) + (uint32_t)(d[3] < emax);
        }
        __syncwarp();
      }
      if (near) {
        // candidates below the lane's bound go to its queue column (unconditional stores at the next
        // slot, kept only if counted), inserted every 16 pairs of the lanes
#pragma unroll 1
        for (uint32_t t0 = 0; t0 < n_pr; t0 += 8 * L) {
          uint32_t qa = q0;
          const uint32_t t1 = min(n_pr, t0 + 8 * L);
          const ulonglong2* pk = rp + 2 * (t0 + sub);
#pragma unroll 2
          for (uint32_t t = t0 + sub; t < t1; t += L, pk += 2 * L) {
            const ulonglong2 xy = pk[0], zw = pk[1];
            float da, db, wa, wb;
            f2_unpack(dist2_x2_fma(px, py, pz, xy.x, xy.y, zw.x, one2), da, db);
            f2_unpack(zw.y, wa, wb);
            if (MODE == kNoRdf && nwithin != nullptr) within += (uint32_t)(da < emax) + (uint32_t)(db < emax);
            queue_push_other(qa, da, thr, __float_as_uint(wa), pidx);
            queue_push_other(qa, db, thr, __float_as_uint(wb), pidx);
          }
          __syncwarp();
          const uint32_t qn = (qa - q0) >> 7, m = __reduce_max_sync(0xffffffffu, qn);
          for (uint32_t q = 0; q < m; ++q)
            if (q < qn) topk_insert(top, queue_at(q0, q));
          float kth = top[KK - 1];  // an upper bound of the central's k-th distance in each of its lanes
          if (KK > 12 || L >= 8u)
            kth = topk_bound(top, L);
          else
            for (uint32_t o = 1; o < L; o <<= 1) kth = fminf(kth, __shfl_xor_sync(0xffffffffu, kth, o));
          thr = fminf(kth, emax);
        }
        near_max = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(valid ? thr : 0.f)));
      }
      if (RDF && H.priv) {
        wcount += 32u * 64u;
        if (wcount >= (1ull << 30)) {
          H.flush_warp(a);
          wcount = 0;
        }
      }
    };

    item_scan(S, ng, c, box, ring, nb, all, emax, near_max, batch, [](float) { return true; });
    if (all) {
      // the centrals met themselves once each, at d2 = 0 (a non-finite one did not, nor any where the range
      // squared is 0 in float32)
      bool self = valid && sub == 0 && emax > 0.f && dist2(p.x, p.y, p.z, p.x, p.y, p.z) == 0.f;
      if (self && !a.self_all) self = in_mask(a.nbr, a.type[pidx]);
      within -= (uint32_t)self;
      if (MODE == kRdfDirect && rdf_here) {
        const uint32_t n_self = __popc(__ballot_sync(0xffffffffu, self));
        if (lane == 0 && n_self) red_shared(row_base + 4u * kMagicBits, 0u - n_self);
      }
    }
    // merge the sorted lists of the L lanes of each central (disjoint candidate subsets): the smallest head
    // is taken k_need times, rank by rank into the queue buffer, a column per central.  (Merging pairs of
    // lists by insertion takes lg L rounds of up to KK insertions: ~1000 instructions at 16 lanes and KK =
    // 10, ~8000 at 32, against ~250 and ~1400.  Thin clouds, where most items hold one to three centrals: 5e4-ion
    // cylinder, third-size cells, r = 1 nm, k = 32, whole call 0.61 -> 0.42 ms, k = 10 with per-ion counts
    // 0.253 -> 0.238; 1e6 ions, half-size cells, r = 1.5 nm, 5 % of them central 0.578 -> 0.553 ms.)
    const uint32_t n_col = 32u >> lg;
    if (L > 1u) {
      for (uint32_t o = 1; o < L; o <<= 1) within += __shfl_xor_sync(0xffffffffu, within, o);
      if constexpr (KMAX > 0) {
        const uint32_t group = ((1u << L) - 1u) << (lane & ~(L - 1u));
        __syncwarp();
#pragma unroll 1
        for (uint32_t rank = 0; rank < a.k_need; ++rank) {
          float m = top[0];
          for (uint32_t o = 1; o < L; o <<= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
          const uint32_t heads = __ballot_sync(0xffffffffu, top[0] == m) & group;
          if ((int)lane == __ffs(heads) - 1) {
#pragma unroll
            for (int t = 0; t + 1 < KK; ++t) top[t] = top[t + 1];
            top[KK - 1] = INFINITY;
          }
          if (sub == 0) kq[rank * n_col + ci] = m;
        }
        __syncwarp();
      }
    }
    auto ranked = [&](uint32_t i) -> float { return L > 1u ? kq[i * n_col + ci] : topk_get(top, i); };
    if (valid && sub == 0) {
      if (nwithin) nwithin[pidx] = within;
      if (KMAX > 0) {
        const float kd = ranked(a.k_need - 1);
        const bool found = !(a.emax_near > 0.f) || kd < a.emax_near;
        if (a.emax_near > 0.f) a.need[c0 + ci] = found ? 0u : 1u;
        if (found)
          for (uint32_t q = 0; q < a.n_k; ++q) H.kth(a, q, ranked(a.ks[q] - 1), pidx);
      }
    }
  }

  // ---- items from the back: sparse cells, one thread per central ----
  // central record and cell of the taken items' centrals (<= 32 * 15, kHeavy - 1 per item)
  static_assert(PS_K_MAX * 16 <= 32 * kHalf + 32, "ranks of two lanes per central in the queue buffer");
  static_assert(32 * (kHeavy - 1) <= 4 * kRing && 32 * (kHeavy - 1) <= 32 * kHalf + 32, "light items taken at once");
  uint32_t* cl_rec = reinterpret_cast<uint32_t*>(s_buf[w]);
  uint32_t* cl_cell = reinterpret_cast<uint32_t*>(s_kq[w]);
  const int st = a.stencil;
  // items per take: enough that every warp of the grid gets work when the list is short
  const uint32_t n_warps = gridDim.x * (blockDim.x >> 5);
  const uint32_t take = min(32u, max(1u, (n_light + n_warps - 1) / n_warps));
  for (;;) {
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(a.next_light, take);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base >= n_light) break;
    uint32_t c = 0, f = 0, cnt = 0;
    if (lane < take && base + lane < n_light) {
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
    for (uint32_t q = 0; q < cnt; ++q) cl_rec[inc - cnt + q] = f + q, cl_cell[inc - cnt + q] = c;
    __syncwarp();
    for (uint32_t r0 = 0; r0 < total; r0 += 32) {
      bool valid = r0 + lane < total;
      if (a.fallback && valid) valid = a.need[cl_rec[r0 + lane]] != 0u;
      uint32_t rowc = 0;  // increments of the warp row by this lane
      if (valid) {
        const uint32_t ce = cl_cell[r0 + lane];
        const float4 p = __ldg(a.crec + cl_rec[r0 + lane]);
        const uint32_t pidx = __float_as_uint(p.w);
        const uint32_t cx = ce % ng.dims[0], cy = (ce / ng.dims[0]) % ng.dims[1], cz = ce / (ng.dims[0] * ng.dims[1]);
        float top[KK];
#pragma unroll
        for (int t = 0; t < KK; ++t) top[t] = INFINITY;
        uint32_t within = 0;
        for (int dz = -st; dz <= st; ++dz)
          for (int dy = -st; dy <= st; ++dy) {
            uint32_t j0 = 0, nj = 0;
            row_run(S, ng, cx, (int)cy + dy, (int)cz + dz, row_width(S, dy, dz), j0, nj);
            const uint32_t j1 = j0 + nj;
            for (uint32_t j = j0; j < j1; ++j) {
              const float4 q = __ldg(a.nrec + j);
              const float d2 = dist2(p.x, p.y, p.z, q.x, q.y, q.z);
              if (d2 < erange && __float_as_uint(q.w) != pidx) {
                ++within;
                if (rdf_here) {
                  if (within <= kRowLaneCap) {
                    if (MODE == kRdfDirect)
                      fb.count1(d2, row_base);
                    else
                      H.pair(a, d2, my_below);
                  }
                  else
                    H.pair_global(a, d2, 1u, my_binned, my_below);
                }
                if (KMAX > 0 && d2 < top[KK - 1]) topk_insert(top, d2);
              }
            }
          }
        rowc = within < kRowLaneCap ? within : kRowLaneCap;
        if (nwithin) nwithin[pidx] = within;
        if (KMAX > 0) {
          const bool found = !(a.emax_near > 0.f) || topk_get(top, a.k_need - 1) < a.emax_near;
          if (a.emax_near > 0.f) a.need[cl_rec[r0 + lane]] = found ? 0u : 1u;
          if (found)
            for (uint32_t q = 0; q < a.n_k; ++q) H.kth(a, q, topk_get(top, a.ks[q] - 1), pidx);
        }
      }
      if (RDF) {
        // a round adds at most 32 * 2^25 = 2^30 to the row: flushed at 2^30, it stays below 2^31
        wcount += __reduce_add_sync(0xffffffffu, rowc);
        if (wcount >= (1ull << 30)) {
          H.flush_warp(a);
          wcount = 0;
        }
      }
    }
    __syncwarp();  // cl is rewritten next
  }
  H.flush(a);
  add_pair_counters(a, my_binned, my_below);
}

// ---------------------------------------------------------------------------
// CTA kernel: one CTA per dense cell, runs staged in shared memory by bulk copies
// ---------------------------------------------------------------------------
template <int KMAX, bool RDF>
__global__ void __launch_bounds__(256) k_query_cta(const __grid_constant__ QueryArgs a) {
  griddep_wait();
  griddep_launch();
  const Search S = search_of(a);
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint64_t bar;
  __shared__ uint32_t s_item;
  __shared__ uint32_t s_run_src[kMaxRuns], s_run_len[kMaxRuns];
  __shared__ int s_timeout;
  constexpr int KK = KMAX > 0 ? KMAX : 1;

  Hist<RDF> H;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
    s_timeout = 0;
  }
  H.init(a, smem, a.stage_cap);
  float4* s_cand =
      reinterpret_cast<float4*>(smem + smem_layout(a.n_bins, a.n_k, RDF, a.stage_cap, false, a.lut_n).off_stage);
  const uint32_t tid = threadIdx.x;
  const Geo ng = *a.ngeo;
  const uint32_t work_n = a.cgeo->work_n;
  const uint32_t n_runs = (2 * a.stencil + 1) * (2 * a.stencil + 1);
  uint32_t phase = 0, stuck_phase = 0;
  uint64_t my_binned = 0;
  uint32_t my_below = 0;

  for (;;) {
    if (tid == 0) s_item = atomicAdd(&a.cgeo->work_next, 1u);
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= work_n || s_timeout) break;
    const uint32_t c = a.cwork[item];
    const uint32_t c0 = a.cstart[c], n_c = a.cstart[c + 1] - c0;
    if (tid < n_runs) cell_run(S, ng, c, tid, s_run_src[tid], s_run_len[tid]);
    __syncthreads();

    for (uint32_t cb = 0; cb < n_c; cb += blockDim.x) {
      const uint32_t ci = cb + tid;
      const bool valid = ci < n_c;
      float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
      if (valid) p = a.crec[c0 + ci];
      const uint32_t pidx = __float_as_uint(p.w);
      float top[KK];
#pragma unroll
      for (int t = 0; t < KK; ++t) top[t] = INFINITY;
      uint32_t within = 0;

      // walk the runs in chunks of at most stage_cap records (padded to a multiple of 8 with far records)
      uint32_t r = 0, ro = 0;
      while (r < n_runs) {
        uint32_t chunk = 0;
        uint32_t rr = r, rro = ro;
        while (rr < n_runs && chunk < a.stage_cap) {
          const uint32_t len = s_run_len[rr];
          const uint32_t take = min(len - rro, a.stage_cap - chunk);
          chunk += take;
          rro += take;
          if (rro >= len) ++rr, rro = 0;
        }
        if (chunk == 0) break;
        const uint32_t padded = (chunk + 7u) & ~7u;
        if (tid == 0) {
          for (uint32_t t = chunk; t < padded; ++t) s_cand[t] = far_record();
          mbar_arrive_expect_tx(&bar, chunk * 16u);
          uint32_t dst = 0, q = r, qo = ro;
          while (q < n_runs && dst < chunk) {
            const uint32_t len = s_run_len[q];
            const uint32_t take = min(len - qo, chunk - dst);
            if (take) bulk_g2s(s_cand + dst, a.nrec + s_run_src[q] + qo, take * 16u, &bar);
            dst += take;
            qo += take;
            if (qo >= len) ++q, qo = 0;
          }
        }
        r = rr;
        ro = rro;
        if (!mbar_wait_bounded(&bar, phase, kWaitLimitNs)) s_timeout = 1;
        const uint32_t this_phase = phase;
        phase ^= 1u;

        if (valid) {
          for (uint32_t t0 = 0; t0 < padded; t0 += 8) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const float4 q = s_cand[t0 + u];
              const float d2 = dist2(p.x, p.y, p.z, q.x, q.y, q.z);
              if (d2 < H.Emax && __float_as_uint(q.w) != pidx) {
                ++within;
                H.pair(a, d2, my_below);
                if (KMAX > 0) topk_insert(top, d2);
              }
            }
          }
        }
        __syncthreads();  // the chunk buffer is reused next
        if (s_timeout) {  // uniform after the barrier: issue no more copies
          stuck_phase = this_phase;
          break;
        }
      }
      if (s_timeout) break;
      if (valid) {
        if (a.nwithin) a.nwithin[pidx] = within;
        if (KMAX > 0)
          for (uint32_t q = 0; q < a.n_k; ++q) H.kth(a, q, topk_get(top, a.ks[q] - 1), pidx);
      }
    }
    __syncthreads();  // s_item and the run table are rewritten next
  }
  if (s_timeout) {
    // the copies of the phase that timed out may still be in flight into this CTA's shared
    // memory: wait for them once more (bounded) before the CTA exits
    if (tid == 0) mbar_wait_bounded(&bar, stuck_phase, kWaitLimitNs);
    __syncthreads();
  }
  H.flush(a);
  add_pair_counters(a, my_binned, my_below);
  if (tid == 0 && s_timeout) atomicCAS((int*)&a.cgeo->status, 0, (int)PS_ERR_TIMEOUT);
}

// ---------------------------------------------------------------------------
// symmetric RDF pass: every unordered pair of neighbour records once (sweep_pairs)
// ---------------------------------------------------------------------------
// Bound by instruction issue and the shared-memory pipe (ncu, 2e5 cylinder: 77 % of the issue slots,
// two bank cycles per increment).  FAST (r0 = 0, at most kPrivBins bins; the host's rule in run_query):
// two 32-bit rows per warp, for pairs of weight 1 and 2, and one increment per test by every
// lane.  With the candidates cut down to those near the staged records two of five tests hit, and a
// warp list of the hits (ballots, counts, a store and a load each) costs more than the idle lanes.
// Measured, all-all, one box (ms): 1e8-ion needle 192.8 -> 76.7, 8e6-ion needle 14.95 -> 5.85,
// 2e5 cylinder 0.504 -> 0.232 (before: full half stencils, warp list of hits, bin table).
// Otherwise (r0 > 0 or more bins): the general bins of Hist, a branch per hit.
// WITHIN (direct bins): also the in-range neighbours of every record, in record order, into `wacc`: a
// candidate's lane counts its hits, the hits of a staged record are counted over the warp.
template <bool FAST, bool WITHIN>
__global__ void __launch_bounds__(256, WITHIN ? 3 : 4) k_rdf_sym(const QueryArgs a, const __grid_constant__ SweepArgs sw,
                                                                 uint32_t* __restrict__ wacc) {
  griddep_wait();
  griddep_launch();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SweepBuf s_sweep[8];
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (a.sweep && !sweep_pays(*a.ngeo, *a.cgeo)) return;
  SweepBuf& buf = s_sweep[w];
  uint64_t wcount = 0;  // bound on the increments of this warp's rows since their last flush (uniform)
  if constexpr (FAST) {
    const uint32_t nb = a.n_bins, stride = nb + 1;  // bin n_bins: out of range
    float* sE = reinterpret_cast<float*>(smem);
    uint32_t* rows = reinterpret_cast<uint32_t*>(sE + stride);  // [8][2][stride]
    for (uint32_t b = threadIdx.x; b <= nb; b += blockDim.x) {
      const double e = __dadd_rn(a.r0, __dmul_rn((double)b, a.dr));
      sE[b] = __double2float_rn(__dmul_rn(e, e));
    }
    for (uint32_t b = threadIdx.x; b < 16 * stride; b += blockDim.x) rows[b] = 0;
    __syncthreads();
    FastBins fb;
    fb.init(a.n_bins, a.dr, sE);
    uint32_t* row1 = rows + 2 * w * stride;
    const uint32_t a1 = smem_u32(row1), base1 = a1 - 4u * kMagicBits, base2 = base1 + 4u * stride;
    const unsigned long long one2 = f2_pack(sw.one, sw.one);
    const float Emax = sE[nb];
    uint32_t* wrec = rows + 16 * stride + w * kSweepRec;  // WITHIN: hits of the staged records
    if (WITHIN)
      for (uint32_t r = lane; r < kSweepRec; r += 32) wrec[r] = 0;
    auto tile = [&](uint32_t n_pr, uint32_t, uint32_t nc, bool) __attribute__((always_inline)) {
      const float4 far = make_float4(INFINITY, INFINITY, INFINITY, __uint_as_float(kCandSingle));
      const float4 c0 = lane < nc ? buf.cand[lane] : far, c1 = lane + 32 < nc ? buf.cand[lane + 32] : far;
      const uint32_t k0 = __float_as_uint(c0.w), k1 = __float_as_uint(c1.w);
      const uint32_t b0 = k0 == kCandBoth ? base2 : base1, b1 = k1 == kCandBoth ? base2 : base1;
      const unsigned long long x0 = f2_pack(c0.x, c0.x), y0 = f2_pack(c0.y, c0.y), z0 = f2_pack(c0.z, c0.z);
      const unsigned long long x1 = f2_pack(c1.x, c1.x), y1 = f2_pack(c1.y, c1.y), z1 = f2_pack(c1.z, c1.z);
      const ulonglong2* rxy = reinterpret_cast<const ulonglong2*>(buf.rxy);
      const ulonglong2* rz = reinterpret_cast<const ulonglong2*>(buf.rz);
      uint32_t hits0 = 0, hits1 = 0;
#pragma unroll 1
      for (uint32_t k = 0; k < n_pr; k += 2) {  // 4 records against the lane's 2 candidates
        const ulonglong2 xy = rxy[k], xy2 = rxy[k + 1], zz = rz[k >> 1];
        const unsigned long long d0 = dist2_x2_fma(xy.x, xy.y, zz.x, x0, y0, z0, one2);
        const unsigned long long d1 = dist2_x2_fma(xy.x, xy.y, zz.x, x1, y1, z1, one2);
        const unsigned long long d2 = dist2_x2_fma(xy2.x, xy2.y, zz.y, x0, y0, z0, one2);
        const unsigned long long d3 = dist2_x2_fma(xy2.x, xy2.y, zz.y, x1, y1, z1, one2);
        const uint32_t x = fb.count2(d0, b0) | fb.count2(d1, b1) | fb.count2(d2, b0) | fb.count2(d3, b1);
        if (__any_sync(0xffffffffu, x != 0u)) {
          fb.settle2(d0, b0);
          fb.settle2(d1, b1);
          fb.settle2(d2, b0);
          fb.settle2(d3, b1);
        }
        if (WITHIN) {
          // of each of the four records, and of the lane's two candidates
          float e0[4], e1[4];
          f2_unpack(d0, e0[0], e0[1]), f2_unpack(d2, e0[2], e0[3]);
          f2_unpack(d1, e1[0], e1[1]), f2_unpack(d3, e1[2], e1[3]);
          uint32_t n = 0;
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i) {
            const bool h0 = e0[i] < Emax, h1 = e1[i] < Emax;
            hits0 += h0, hits1 += h1;
            const uint32_t v = __popc(__ballot_sync(0xffffffffu, h0)) + __popc(__ballot_sync(0xffffffffu, h1));
            if (lane == i) n = v;
          }
          if (lane < 4) wrec[2 * k + lane] += n;
        }
      }
      // the staged records met themselves once each, at d2 = 0
      const uint32_t self = __popc(__ballot_sync(0xffffffffu, k0 == kCandSelf)) +
                            __popc(__ballot_sync(0xffffffffu, k1 == kCandSelf));
      if (self && lane == 0) red_shared(a1, 0u - self);
      if (WITHIN) {  // (the block's own records count their neighbours in it as staged records)
        if (lane < nc && (k0 == kCandBoth || k0 == kCandSingle) && hits0) atomicAdd(wacc + buf.cidx[lane], hits0);
        if (lane + 32 < nc && (k1 == kCandBoth || k1 == kCandSingle) && hits1) atomicAdd(wacc + buf.cidx[lane + 32], hits1);
      }
      wcount += 2u * kSweepTile * n_pr;
      if (wcount >= (1ull << 31)) {
        __syncwarp();
        unsigned long long tot = 0;
        for (uint32_t b = lane; b < nb; b += 32) {
          const unsigned long long v = row1[b] + 2ull * row1[stride + b];
          if (v) atomicAdd((unsigned long long*)&a.rdf[b], v);
          tot += v;
          row1[b] = row1[stride + b] = 0;
        }
        if (tot) atomicAdd((unsigned long long*)&a.meta[PS_META_N_PAIRS], tot);
        __syncwarp();
        wcount = 0;
      }
    };
    if constexpr (WITHIN)
      sweep_pairs<true>(sw, buf, tile, [&](uint32_t m, bool) __attribute__((always_inline)) {
        __syncwarp();
        for (uint32_t r = lane; r < kSweepRec; r += 32) {
          if (r < m && wrec[r]) atomicAdd(wacc + buf.ridx[r], wrec[r]);
          wrec[r] = 0;
        }
        __syncwarp();
      });
    else
      sweep_pairs<false>(sw, buf, tile);
    __syncthreads();
    unsigned long long tot = 0;
    for (uint32_t b = threadIdx.x; b < nb; b += blockDim.x) {
      unsigned long long sum = 0;
      for (uint32_t r = 0; r < 8; ++r) sum += rows[2 * r * stride + b] + 2ull * rows[(2 * r + 1) * stride + b];
      if (sum) atomicAdd((unsigned long long*)&a.rdf[b], sum);
      tot += sum;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0 && tot) atomicAdd((unsigned long long*)&a.meta[PS_META_N_PAIRS], tot);
  } else {
    Hist<true> H{};
    H.init(a, smem, 0, true);
    const float Emax = H.Emax;
    uint32_t my_below = 0;
    sweep_pairs<true>(sw, buf, [&](uint32_t, uint32_t m, uint32_t nc, bool) __attribute__((always_inline)) {
      const float* rxy = reinterpret_cast<const float*>(buf.rxy);
      const float* rz = reinterpret_cast<const float*>(buf.rz);
      for (uint32_t h = lane; h < nc; h += 32) {
        const float4 q = buf.cand[h];
        const uint32_t j = buf.cidx[h], wt = __float_as_uint(q.w) == kCandBoth ? 2u : 1u;
        for (uint32_t k = 0; k < m; ++k) {
          const float* p = rxy + (k >> 1) * 4 + (k & 1u);
          const float d2 = dist2(p[0], p[2], rz[k], q.x, q.y, q.z);
          if (d2 < Emax && buf.ridx[k] != j) H.pair_w(d2, wt, my_below);
        }
      }
      __syncwarp();
      wcount += 2u * kSweepTile * m;
      if (wcount >= (1ull << 30)) {
        H.flush_warp(a);
        wcount = 0;
      }
    });
    H.flush(a);
    add_pair_counters(a, 0, my_below);
  }
}

template <bool FAST, bool WITHIN>
static int launch_rdf_sym(const ps_grid* g, const QueryArgs& qa, const SweepArgs& sw, uint32_t smem, uint32_t* wacc,
                          cudaStream_t s) {
  auto k = k_rdf_sym<FAST, WITHIN>;
  PS_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int per_sm = 0;
  PS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 256, smem));
  if (per_sm < 1) return fail(PS_ERR_UNSUPPORTED, "symmetric RDF kernel does not fit on an SM");
  PS_LAUNCH(PS_KID_RDF_SYM, s, PS_CUDA(launch_pdl(k, g->num_sms * per_sm, 256, smem, s, qa, sw, wacc)));
  return PS_OK;
}

// ---------------------------------------------------------------------------
// near kNN pass on the vertex-centred central list
// ---------------------------------------------------------------------------
constexpr uint32_t kQueue = 40;  // queue rows per lane; inserted when fewer than 16 are free
constexpr uint32_t kVertexSmem = 8 * (16 * 16 + 16 * 8 + (kQueue + 1) * 32 * 4);  // the kernel's static shared memory

// One warp per item (up to 32 centrals of a vertex cell, one to sixteen lanes each), its candidates the
// records of the 2 x 2 x 2 cells around the vertex, staged 32 at a time as interleaved pairs.  A sorted
// insertion costs ~25 instructions for the whole warp whichever lanes need it, so the candidates
// are filtered first: by the central's reach and by the radius that holds k + 3 sqrt(k) records
// at the block's density (about 20 of 240 candidates at k = 10), and the few left are queued and
// inserted together.  A central with fewer than k records there is listed for the full search, as
// one whose k-th distance is beyond its reach.  The central itself stays in (distance 0): the
// list is one longer and rank k is its entry k, so that no test compares indexes.  KMAX > k_need.
// Bound by issue (ncu, 8e6-ion needle: 81 % of the slots).  All-all, k = 10, one box (ms): 8e6-ion needle
// 1.94 -> 1.42, the 1e8-ion one 25.4 -> 20.5 (before: an insertion queue drained every 16 candidates, the
// central compared by index; 1.65 and 21.5 with the strides of shared centrals in the common loop).
template <int KMAX>
__global__ void __launch_bounds__(256, KMAX <= 13 ? 4 : 2) k_knn_vertex(const __grid_constant__ QueryArgs a) {
  griddep_wait();
  griddep_launch();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float4 s_xy[8][16];
  __shared__ float2 s_z[8][16];
  __shared__ float s_kq[8][(kQueue + 1) * 32];
  static_assert(sizeof(s_xy) + sizeof(s_z) + sizeof(s_kq) == kVertexSmem, "run_query asks whether this fits");
  Hist<false> H{};
  H.init(a, smem, 0, true);
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* kq = s_kq[w];
  const uint32_t q0 = smem_u32(kq + lane);
  const Geo ng = *a.ngeo, vg = *a.cgeo;
  const uint32_t n_items = vg.work_n2;
  const unsigned long long one2 = f2_pack(a.one, a.one);
  // rounding slack of a cell coordinate (cells) and the cell edge for vertex_reach
  const float slack = (float)max(ng.dims[0], max(ng.dims[1], ng.dims[2])) * 5.0e-7f + 1.0e-6f;
  const float h_eff = __fmul_rn(__fdiv_rn(1.0f, ng.inv_h), 1.0f - 1.0f / 4096.0f);
  const float k_f = (float)a.k_need, want = (k_f + 3.f * sqrtf(k_f) + 1.f) * 0.238732415f;  // 3 / (4 pi)
  for (;;) {
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(a.next_front, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= n_items) break;
    const uint2 it = a.witem[item];
    const uint32_t c = it.x, cnt = it.y & 63u, c0 = a.cstart[c] + (it.y >> 6);
    const uint32_t L = item_lanes(cnt), lg = 31u - __clz(L);
    const uint32_t sub = lane & (L - 1u), ci = lane >> lg;
    const bool valid = ci < cnt;
    // the four runs of the block: their records as one list
    uint32_t rs = 0, rl = 0;
    vertex_run(a, ng, vg, c, lane, rs, rl);
    const uint32_t s0 = __shfl_sync(0xffffffffu, rs, 0), s1 = __shfl_sync(0xffffffffu, rs, 1),
                   s2 = __shfl_sync(0xffffffffu, rs, 2), s3 = __shfl_sync(0xffffffffu, rs, 3);
    const uint32_t e0 = __shfl_sync(0xffffffffu, rl, 0), e1 = e0 + __shfl_sync(0xffffffffu, rl, 1),
                   e2 = e1 + __shfl_sync(0xffffffffu, rl, 2), n_cand = e2 + __shfl_sync(0xffffffffu, rl, 3);
    auto fetch = [&](uint32_t pos) -> float4 {
      if (pos >= n_cand) return make_float4(INFINITY, INFINITY, INFINITY, 0.f);
      const uint32_t j = pos < e1 ? (pos < e0 ? s0 + pos : s1 + (pos - e0)) : (pos < e2 ? s2 + (pos - e1) : s3 + (pos - e2));
      return __ldg(a.nrec + j);
    };
    float4 nxt = fetch(lane);
    float4 p = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    float thr = 0.f;
    if (valid) {
      p = a.crec[c0 + ci];
      // (cells of the block inside the grid: at least 1 of 8)
      const float r0 = ng.h * cbrtf(want * 8.f / (float)max(n_cand, 1u));
      thr = fminf(vertex_reach(ng, vg, c, p, slack, h_eff, H.Emax), r0 * r0);
    }
    const unsigned long long px = f2_pack(p.x, p.x), py = f2_pack(p.y, p.y), pz = f2_pack(p.z, p.z);
    float top[KMAX];
#pragma unroll
    for (int t = 0; t < KMAX; ++t) top[t] = INFINITY;
    uint32_t qa = q0;  // the next slot of this lane's queue column
    auto insert = [&](uint32_t m) __attribute__((always_inline)) {
      const uint32_t qn = (qa - q0) >> 7;
#pragma unroll 1
      for (uint32_t q = 0; q < m; ++q)
        if (q < qn) topk_insert(top, queue_at(q0, q));
      qa = q0;
    };
    float* sxy = reinterpret_cast<float*>(s_xy[w]);
    float* sz = reinterpret_cast<float*>(s_z[w]);
    for (uint32_t b = 0; b < n_cand; b += 32) {
      __syncwarp();
      {
        float* d = sxy + (lane >> 1) * 4 + (lane & 1u);
        d[0] = nxt.x, d[2] = nxt.y, sz[lane] = nxt.z;
      }
      __syncwarp();
      nxt = fetch(b + 32 + lane);
#pragma unroll 1
      for (uint32_t hb = 0; hb < 16; hb += 8) {
        auto test = [&](uint32_t t) __attribute__((always_inline)) {
          const ulonglong2 xy = *reinterpret_cast<const ulonglong2*>(&s_xy[w][t]);
          const unsigned long long zz = *reinterpret_cast<const unsigned long long*>(&s_z[w][t]);
          float da, db;
          f2_unpack(dist2_x2_fma(px, py, pz, xy.x, xy.y, zz, one2), da, db);
          queue_push(qa, da, thr);
          queue_push(qa, db, thr);
        };
        if (L == 1u) {  // constant offsets: half the instructions of the loop below
#pragma unroll
          for (uint32_t t = 0; t < 8; ++t) test(hb + t);
        } else {
#pragma unroll 1
          for (uint32_t t = hb + sub; t < hb + 8; t += L) test(t);
        }
        const uint32_t m = __reduce_max_sync(0xffffffffu, qa - q0) >> 7;
        if (m > kQueue - 16u) {
          insert(m);
          thr = fminf(thr, top[KMAX - 1]);
        }
      }
    }
    insert(__reduce_max_sync(0xffffffffu, qa - q0) >> 7);
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
    bool miss = false;
    if (valid && sub == 0) {
      miss = !(topk_get(top, a.k_need) < INFINITY);  // entry 0 is the central itself
      if (!miss)
        for (uint32_t q = 0; q < a.n_k; ++q) H.kth(a, q, topk_get(top, a.ks[q]), __float_as_uint(p.w));
    }
    list_append(a, miss, c0 + ci, lane);
  }
  H.flush(a);
}

template <int KMAX>
static int launch_knn_vertex(const ps_grid* g, const QueryArgs& qa, uint32_t smem, cudaStream_t s) {
  auto k = k_knn_vertex<KMAX>;
  int per_sm = 0;
  PS_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  PS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 256, smem));
  if (per_sm < 1) return fail(PS_ERR_UNSUPPORTED, "near kNN kernel does not fit on an SM");
  PS_LAUNCH(PS_KID_QUERY, s, PS_CUDA(launch_pdl(k, g->num_sms * per_sm, 256, smem, s, qa)));
  return PS_OK;
}

static int dispatch_knn_vertex(const ps_grid* g, const QueryArgs& qa, uint32_t smem, cudaStream_t s) {
  const uint32_t k = qa.k_need;
  if (k <= 1) return launch_knn_vertex<2>(g, qa, smem, s);
  if (k <= 2) return launch_knn_vertex<3>(g, qa, smem, s);
  if (k <= 4) return launch_knn_vertex<5>(g, qa, smem, s);
  if (k <= 8) return launch_knn_vertex<9>(g, qa, smem, s);
  if (k <= 10) return launch_knn_vertex<11>(g, qa, smem, s);
  if (k <= 12) return launch_knn_vertex<13>(g, qa, smem, s);
  if (k <= 16) return launch_knn_vertex<17>(g, qa, smem, s);
  return launch_knn_vertex<33>(g, qa, smem, s);
}

// ---------------------------------------------------------------------------
// full-radius kNN of the centrals the near pass could not settle
// ---------------------------------------------------------------------------
// Full-radius kNN of the centrals listed by the near pass: one lane per listed central, in two
// tiers: (A) the 27 cells around its cell (every record within one cell of it; the central's
// reach is its distance to the faces of that block, less the rounding slack), then, for the
// warps with a central whose k-th distance is not within that reach, (B) the rest of its stencil
// (the outer cells of the 9 inner rows and the outer rows).  Each tier walks its rows (nearest
// first) with the k_need smallest d2 below E[nb] kept through the per-lane queue; fewer than k of
// them: not found (INF).
template <int KMAX>
__global__ void __launch_bounds__(256) k_knn_list(const __grid_constant__ QueryArgs a) {
  griddep_wait();
  griddep_launch();
  const Search S = search_of(a);
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float s_kq[8][17 * 32];
  Hist<false> H{};
  H.init(a, smem, 0, true);
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float* kq = s_kq[w];
  const Geo ng = *a.ngeo;
  const float Emax = H.Emax;
  const uint32_t n_list = a.cgeo->list_n;
  const int s = a.stencil, n_rows = (2 * s + 1) * (2 * s + 1);
  const float slack = (float)max(ng.dims[0], max(ng.dims[1], ng.dims[2])) * 5.0e-7f + 1.0e-6f;
  const float h_eff = __fmul_rn(__fdiv_rn(1.0f, ng.inv_h), 1.0f - 1.0f / 4096.0f);
  const uint32_t n_warps = gridDim.x * (blockDim.x >> 5);
  for (uint32_t base = (blockIdx.x * (blockDim.x >> 5) + w) * 32u; base < n_list; base += n_warps * 32u) {
    const bool valid = base + lane < n_list;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
    int cc[3] = {0, 0, 0};
    float reach = -1.0f;
    if (valid) {
      p = a.crec[a.need[base + lane]];
      const float pc[3] = {p.x, p.y, p.z};
      float m = INFINITY;
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        const float u = __fmul_rn(__fsub_rn(pc[ax], ng.origin[ax]), ng.inv_h);
        int c = __float2int_rd(u);
        c = c < 0 ? 0 : (c >= (int)ng.dims[ax] ? (int)ng.dims[ax] - 1 : c);
        cc[ax] = c;
        m = fminf(m, fminf(__fsub_rn(u, (float)c - 1.0f), __fsub_rn((float)c + 2.0f, u)));
      }
      const float r = __fmul_rn(fmaxf(__fsub_rn(m, slack), 0.0f), h_eff);
      reach = fminf(__fmul_rn(__fmul_rn(r, r), 1.0f - 1.0f / 4096.0f), Emax);
    }
    const uint32_t pidx = valid ? __float_as_uint(p.w) : ~0u;
    float top[KMAX];
#pragma unroll
    for (int t = 0; t < KMAX; ++t) top[t] = INFINITY;
    // one x-run per lane: the records of cells xlo..xhi of row (y, z), for the lanes in `act`
    auto walk = [&](bool act, int y, int z, int xlo, int xhi) {
      uint32_t src = 0, len = 0;
      xlo = max(xlo, 0), xhi = min(xhi, (int)ng.dims[0] - 1);
      if (act && xlo <= xhi && y >= 0 && z >= 0 && y < (int)ng.dims[1] && z < (int)ng.dims[2]) {
        const uint32_t row = ((uint32_t)z * ng.dims[1] + (uint32_t)y) * ng.dims[0];
        src = a.nstart[row + xlo];
        len = a.nstart[row + xhi + 1] - src;
      }
      const uint32_t n_max = __reduce_max_sync(0xffffffffu, len);
      for (uint32_t t0 = 0; t0 < n_max; t0 += 16) {
        const float thr = fminf(top[KMAX - 1], Emax);  // in range only: fewer than k leaves INF
        uint32_t qn = 0;
#pragma unroll 4
        for (uint32_t u = 0; u < 16; ++u) {
          const uint32_t t = t0 + u;
          float4 q = far_record();
          if (t < len) q = __ldg(a.nrec + src + t);
          const float d2 = dist2(p.x, p.y, p.z, q.x, q.y, q.z);
          kq[qn * 32 + lane] = d2;
          qn += (d2 < thr && __float_as_uint(q.w) != pidx) ? 1u : 0u;
        }
        const uint32_t m = __reduce_max_sync(0xffffffffu, qn);
        for (uint32_t q = 0; q < m; ++q)
          if (q < qn) topk_insert(top, kq[q * 32 + lane]);
        __syncwarp();
      }
    };
    // tier A: the 9 inner rows over cx - 1 .. cx + 1 (the first 9 rows of the nearest-first order)
    for (int r = 0; r < 9; ++r)
      walk(valid, cc[1] + c_row_dy[r], cc[2] + c_row_dz[r], cc[0] - 1, cc[0] + 1);
    const bool more = valid && !(topk_get(top, a.k_need - 1) < reach);
    if (__ballot_sync(0xffffffffu, more)) {
      // tier B: the outer cells of the inner rows, then the outer rows, each within its width
      for (int r = 0; r < 9; ++r) {
        const int dy = c_row_dy[r], dz = c_row_dz[r], wd = valid ? row_width(S, dy, dz) : -1;
        walk(more && wd >= 2, cc[1] + dy, cc[2] + dz, cc[0] - wd, cc[0] - 2);
        walk(more && wd >= 2, cc[1] + dy, cc[2] + dz, cc[0] + 2, cc[0] + wd);
      }
      for (int r = 9; r < n_rows; ++r) {
        const int dy = c_row_dy[r], dz = c_row_dz[r], wd = valid ? row_width(S, dy, dz) : -1;
        walk(more && wd >= 0, cc[1] + dy, cc[2] + dz, cc[0] - wd, cc[0] + wd);
      }
    }
    if (valid)
      for (uint32_t q = 0; q < a.n_k; ++q) H.kth(a, q, topk_get(top, a.ks[q] - 1), pidx);
  }
  H.flush(a);
}

template <int KMAX>
static int launch_knn_list(const ps_grid* g, const QueryArgs& qa, uint32_t smem, cudaStream_t s) {
  auto k = k_knn_list<KMAX>;
  int per_sm = 0;
  PS_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  PS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 256, smem));
  if (per_sm < 1) return fail(PS_ERR_UNSUPPORTED, "full-radius kNN kernel does not fit on an SM");
  PS_LAUNCH(PS_KID_KNN_FULL, s, PS_CUDA(launch_pdl(k, g->num_sms * per_sm, 256, smem, s, qa)));
  return PS_OK;
}

static int dispatch_knn_list(const ps_grid* g, const QueryArgs& qa, uint32_t smem, cudaStream_t s) {
  const uint32_t k = qa.k_need;
  if (k <= 1) return launch_knn_list<1>(g, qa, smem, s);
  if (k <= 2) return launch_knn_list<2>(g, qa, smem, s);
  if (k <= 4) return launch_knn_list<4>(g, qa, smem, s);
  if (k <= 8) return launch_knn_list<8>(g, qa, smem, s);
  if (k <= 10) return launch_knn_list<10>(g, qa, smem, s);
  if (k <= 12) return launch_knn_list<12>(g, qa, smem, s);
  if (k <= 16) return launch_knn_list<16>(g, qa, smem, s);
  return launch_knn_list<32>(g, qa, smem, s);
}

// Writes n_central and the device status into the meta array, and the in-range counts that the sweep
// took (wacc, record order; each central met itself once) to their ions.
__global__ void __launch_bounds__(256) k_query_epilogue(const Geo* __restrict__ ngeo, const Geo* __restrict__ cgeo,
                                                        uint64_t* meta, const float4* __restrict__ nrec,
                                                        const uint32_t* __restrict__ pfx,
                                                        const uint32_t* __restrict__ wacc, uint32_t* __restrict__ nwithin) {
  griddep_wait();
  griddep_launch();
  if (wacc != nullptr && sweep_pays(*ngeo, *cgeo)) {
    const uint32_t n = ngeo->n_sel;
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
      if (pfx[j + 1] == pfx[j]) continue;
      const float4 p = __ldg(nrec + j);
      const bool self = dist2(p.x, p.y, p.z, p.x, p.y, p.z) == 0.f;
      nwithin[__float_as_uint(p.w)] = wacc[j] - (uint32_t)self;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    meta[PS_META_N_CENTRAL] = cgeo->n_sel;
    int st = cgeo->status;
    if (st == 0) st = ngeo->status;
    meta[PS_META_STATUS] = (uint64_t)(uint32_t)st;
  }
}

template <int KMAX, int MODE>
static int launch_query(const ps_grid* g, const QueryArgs& qa, uint32_t smem_cta, uint32_t smem_warp, cudaStream_t s) {
  const uint32_t kid = qa.fallback ? PS_KID_KNN_FULL : PS_KID_QUERY;
  constexpr bool RDF = MODE != kNoRdf;
  auto kw = k_query_warp<KMAX, MODE>;
  PS_CUDA(cudaFuncSetAttribute(kw, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_warp));
  int per_sm_w = 0;
  PS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_w, kw, 256, smem_warp));
  if (per_sm_w < 1) return fail(PS_ERR_UNSUPPORTED, "query kernel does not fit on an SM");
  if (g->dense_min != 0xFFFFFFFFu) {
    auto kc = k_query_cta<KMAX, RDF>;
    PS_CUDA(cudaFuncSetAttribute(kc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_cta));
    int per_sm_c = 0;
    PS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_c, kc, 256, smem_cta));
    if (per_sm_c < 1) return fail(PS_ERR_UNSUPPORTED, "query kernel does not fit on an SM");
    PS_LAUNCH(kid, s, PS_CUDA(launch_pdl(kc, g->num_sms * per_sm_c, 256, smem_cta, s, qa)));
  }
  PS_LAUNCH(kid, s, PS_CUDA(launch_pdl(kw, g->num_sms * per_sm_w, 256, smem_warp, s, qa)));
  PS_CUDA(cudaGetLastError());
  return PS_OK;
}

template <int MODE>
static int dispatch_k(const ps_grid* g, const QueryArgs& qa, uint32_t sc, uint32_t sw, cudaStream_t s) {
  const uint32_t k = qa.k_need;
  if (k == 0) return MODE != kNoRdf ? launch_query<0, MODE>(g, qa, sc, sw, s) : PS_OK;
  if (k <= 1) return launch_query<1, MODE>(g, qa, sc, sw, s);
  if (k <= 2) return launch_query<2, MODE>(g, qa, sc, sw, s);
  if (k <= 4) return launch_query<4, MODE>(g, qa, sc, sw, s);
  if (k <= 8) return launch_query<8, MODE>(g, qa, sc, sw, s);
  if (k <= 10) return launch_query<10, MODE>(g, qa, sc, sw, s);
  if (k <= 12) return launch_query<12, MODE>(g, qa, sc, sw, s);
  if (k <= 16) return launch_query<16, MODE>(g, qa, sc, sw, s);
  return launch_query<32, MODE>(g, qa, sc, sw, s);
}

// Parameters of the bin lookup table: a bit shift S <= 16 at which the interior edges
// E[1..nb-1] fall in strictly increasing cells of the float32 bit pattern (bits >> S), so that a
// cell holds at most one edge, whose low S bits its entry carries; the table covers the cells from
// the one below E[1]'s to E[nb]'s.  The largest such S gives the smallest table.  None when the
// table would exceed kLutMax entries, two edges coincide or nb >= 2^15.
static void choose_lut(ps_bins bins, QueryArgs& qa) {
  qa.lut_shift = qa.lut_base = qa.lut_n = 0;
  const uint32_t nb = bins.n_bins;
  if (nb < 2 || nb >= (1u << 15)) return;
  std::vector<uint32_t> Eb(nb + 1);
  for (uint32_t b = 0; b <= nb; ++b) {
    const double e = bins.r0 + (double)b * bins.dr;
    const float f = (float)(e * e);
    memcpy(&Eb[b], &f, 4);
  }
  for (int S = 16; S >= 1; --S) {
    bool ok = (Eb[1] >> S) >= 1;
    for (uint32_t b = 2; b < nb && ok; ++b) ok = (Eb[b] >> S) > (Eb[b - 1] >> S);
    if (!ok) continue;
    const uint32_t base = (Eb[1] >> S) - 1, n = (Eb[nb] >> S) - base + 1;
    if (n <= kLutMax) {
      qa.lut_shift = (uint32_t)S;
      qa.lut_base = base;
      qa.lut_n = n;
    }
    return;
  }
}

int run_query(ps_grid* g, const float* dsrf, const uint64_t ctr_mask[4], float dsrf_min, ps_bins bins,
              const uint32_t* ks, uint32_t n_k, uint64_t* d_rdf, uint64_t* d_knn, uint64_t* d_meta, float* d_kth,
              uint32_t* d_nwithin, cudaStream_t s) {
  QueryArgs qa;
  memset(&qa, 0, sizeof(qa));
  qa.nrec = g->nbr.rec;
  qa.nstart = g->nbr.start;
  qa.nsub = g->nbr.count;
  qa.ngeo = g->nbr.geo;
  qa.crec = g->ctr.rec;
  qa.cstart = g->ctr.start;
  qa.cwork = g->ctr.work;
  qa.witem = g->ctr.witem;
  qa.whi = g->nbr_witem;
  qa.work_cap = g->item_cap;
  qa.cgeo = g->ctr.geo;
  qa.stencil = g->stencil;
  row_widths(g->stencil, g->cell_scale, qa.row_w);
  qa.r0 = bins.r0;
  qa.dr = bins.dr;
  qa.n_bins = bins.n_bins;
  qa.n_k = n_k;
  qa.k_need = 0;
  for (uint32_t q = 0; q < n_k; ++q) {
    qa.ks[q] = ks[q];
    if (ks[q] > qa.k_need) qa.k_need = ks[q];
  }
  qa.rdf = d_rdf;
  qa.knn = d_knn;
  qa.meta = d_meta;
  qa.kth = d_kth;
  qa.nwithin = d_nwithin;
  qa.n = g->n;
  qa.next_front = &g->ctr.geo->work_next2;
  qa.next_light = &g->ctr.geo->work_next3;
  choose_lut(bins, qa);

  const bool rdf = d_rdf != nullptr;
  // direct bins: r0 = 0, a warp's row of counts at most 2 KB, and edges and range far from the limits
  // of float32 (the approximate root flushes subnormals)
  const double stop = bins.r0 + (double)bins.n_bins * bins.dr;
  const bool direct = bins.r0 == 0.0 && bins.n_bins <= kPrivBins && bins.dr > 1e-15 && stop < 1e15;
  ZeroOut z;  // the outputs are zeroed by the central-list reset kernel
  z.p[0] = d_meta;
  z.n[0] = PS_META_LEN(n_k);
  if (rdf) z.p[1] = d_rdf, z.n[1] = bins.n_bins;
  if (n_k) z.p[2] = d_knn, z.n[2] = n_k * bins.n_bins;
  // one-pass queries: the sweep takes dense clouds (sweep_pays); its in-range counts, in record order, in
  // the counting sort's index list, free until the next build
  const bool in_passes = g->split && centrals_in_neighbours(g, ctr_mask) && rdf && d_nwithin == nullptr && g->stencil >= 2 &&
                         g->dense_min == 0xFFFFFFFFu;
  const bool sweep = !in_passes && rdf && centrals_in_neighbours(g, ctr_mask) && g->dense_min == 0xFFFFFFFFu &&
                     (direct || d_nwithin == nullptr);
  uint32_t* wacc = sweep && d_nwithin != nullptr ? g->sel : nullptr;
  if (wacc) z.p[3] = reinterpret_cast<uint64_t*>(wacc), z.n[3] = (uint32_t)(((uint64_t)g->n + 1) / 2);

  const bool subset = centrals_in_neighbours(g, ctr_mask);
  qa.self_all = subset;
  qa.type = g->type;
  for (int w = 0; w < 4; ++w) qa.nbr.w[w] = g->nbr_mask[w];
  qa.one = 1.0f;
  int dev_smem = 0;
  PS_CUDA(cudaDeviceGetAttribute(&dev_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, g->device));
  // the query in passes, and its near kNN pass on the vertex-centred central list (two-cell
  // stencils; the ranks of that counting sort take one word per central of the cell arrays; its queues
  // take 3 KB more than k_query_warp's may, which does the pass where the kNN histograms nearly fill an SM,
  // such as 32 k values of 1,419 to 1,440 bins)
  const bool split = in_passes;
  const bool vertex = split && n_k > 0 && g->stencil == 2 && (uint64_t)g->n <= (uint64_t)g->cell_cap &&
                      smem_layout(bins.n_bins, n_k, false, 0, true).total + kVertexSmem <= (uint32_t)dev_smem;
  int rc = build_central_list(g, dsrf, ctr_mask, dsrf_min, s, z, true, vertex, !split || n_k > 0,
                              split ? kSweep : (sweep ? kSweepIfDense : kNoSweep));
  if (rc) return rc;

  // staging budget of the CTA kernel: two CTAs per SM
  const SmemLayout base = smem_layout(bins.n_bins, n_k, rdf, 0, false, qa.lut_n);
  const uint32_t budget = (uint32_t)dev_smem / 2 - 2048;
  if (base.total + 16 * 1024 > (uint32_t)dev_smem - 1024)
    return fail(PS_ERR_UNSUPPORTED, "too many bins x k values for shared memory");
  uint32_t stage_bytes = budget > base.total + 16 * 1024 ? budget - base.total : 16 * 1024;
  qa.stage_cap = (stage_bytes / 16) & ~7u;
  const uint32_t smem_cta = smem_layout(bins.n_bins, n_k, rdf, qa.stage_cap, false, qa.lut_n).total;
  const uint32_t smem_warp = smem_layout(bins.n_bins, n_k, rdf, 0, true, qa.lut_n).total;
  // the RDF over unordered pairs
  auto run_rdf_sym = [&]() -> int {
    QueryArgs qs = qa;
    qs.n_k = 0;
    SweepArgs sw = sweep_args(g, &g->ctr.geo->sym_next);
    sw.range = (float)(stop * stop);
    if (!direct)
      return launch_rdf_sym<false, false>(g, qs, sw, smem_layout(bins.n_bins, 0, true, 0, true, qa.lut_n).total, nullptr, s);
    const uint32_t smem = (bins.n_bins + 1) * 4 * 17;
    if (d_nwithin == nullptr) return launch_rdf_sym<true, false>(g, qs, sw, smem, nullptr, s);
    return launch_rdf_sym<true, true>(g, qs, sw, smem + 8 * kSweepRec * 4, g->sel, s);
  };
  if (split) {
    // the query in passes: (1) kNN near each central, centrals with fewer than k_need
    // neighbours there set apart; (2) their full-radius kNN; (3) the RDF over unordered pairs
    if (n_k > 0) {
      QueryArgs qn = qa;
      qn.need = g->sel;  // free between a build and the next one (the counting sort's index list)
      const uint32_t smem_knn = smem_layout(bins.n_bins, n_k, false, 0, true).total;
      if (vertex) {
        // the 2 x 2 x 2 cells around each central's nearest vertex, each central within its own
        // reach; the others listed for k_knn_list
        rc = dispatch_knn_vertex(g, qn, smem_knn, s);
        if (rc) return rc;
        rc = dispatch_knn_list(g, qn, smem_knn, s);
        if (rc) return rc;
      } else {
        // the 27 cells around each central's cell, within the cell edge
        const double rk = (double)g->r_cut * (double)g->cell_scale;
        const float Emax = (float)(stop * stop), Ek = (float)(rk * rk);
        qn.emax_near = Ek < Emax ? Ek : Emax;
        qn.stencil = 1;
        row_widths(1, 1.0, qn.row_w);
        rc = dispatch_k<kNoRdf>(g, qn, smem_cta, smem_layout(bins.n_bins, n_k, false, 0, true).total, s);
        if (rc) return rc;
        // the full radius for the centrals it marked
        QueryArgs qf = qa;
        qf.fallback = 1;
        qf.need = g->sel;
        qf.next_front = &g->ctr.geo->work_next2b;
        qf.next_light = &g->ctr.geo->work_next3b;
        rc = dispatch_k<kNoRdf>(g, qf, smem_cta, smem_layout(bins.n_bins, n_k, false, 0, true).total, s);
        if (rc) return rc;
      }
    }
    rc = run_rdf_sym();
    if (rc) return rc;
  } else if (n_k > 0 || rdf) {
    if (sweep) {
      qa.sweep = 1;
      rc = run_rdf_sym();
      if (rc) return rc;
    }
    rc = !rdf    ? dispatch_k<kNoRdf>(g, qa, smem_cta, smem_warp, s)
         : direct ? dispatch_k<kRdfDirect>(g, qa, smem_cta, smem_warp, s)
                  : dispatch_k<kRdfGeneral>(g, qa, smem_cta, smem_warp, s);
    if (rc) return rc;
  }
  PS_LAUNCH(PS_KID_EPILOGUE, s,
            PS_CUDA(launch_pdl(k_query_epilogue, wacc ? g->num_sms * 8 : 1, wacc ? 256 : 32, 0, s, g->nbr.geo, g->ctr.geo, d_meta,
                               g->nbr.rec, reinterpret_cast<const uint32_t*>(g->cr), (const uint32_t*)wacc, d_nwithin)));
  PS_CUDA(cudaGetLastError());
  return PS_OK;
}

}  // namespace ps
