// k_assign.cu - scalars and gridding of galaxies and randoms (Sec. III.A).
//
// Interpolation of the objects to the grid nodes (eq. mapFFT) with CIC, TSC or
// PCS (the paper's fourth-order) weights, as a counting sort by 16^3-cell tile followed by accumulation in
// shared memory:
//   count    per object: FKP weight and the partial sums of the scalars (W,
//            sum w^2, sum w^3, sum nbar w^2, sum nbar^2 w^3, for alpha, I_22,
//            I_33, N_0, S_3: eqs. I22def, N0true, Noise0) in double-single
//            arithmetic per thread and FP64 across threads,
//            the geometry check and one count for the object's tile (block
//            histogram in shared memory);
//   scan     tile offsets (exclusive prefix sum);
//   scatter  each object's (x, y, z, value) to its tile's segment, value =
//            w for galaxies and -alpha w for randoms (and the w^2-weighted
//            value for F^w, eq. SNbisp2), with the L^ab sums (eq. Lab);
//   tiles    one block per tile: every tap is rounded once to a 2^-40
//            fixed-point integer and added in shared memory over the tile and
//            its one-cell halo, then the nonzero cells are added to the grid.
// Integer sums make the grid independent of the order of the objects and of
// the blocks (deterministic, identical alone or inside a batch).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "fkp_internal.h"

namespace fkp {

constexpr int kTile = 16;            // cells per tile side
// Objects per work item of the tile accumulation: a tile's objects are split
// into items of at most this many, so that the few tiles of the densest
// parts of a survey do not hold up the end of the launch.
constexpr int kAccumChunk = 8160;
constexpr int kAccumThreads = 512;
// Region a tile's objects reach, from one cell below the tile: the tile
// plus one halo cell on each side for CIC and TSC, and one more above for
// PCS (taps c-1 .. c+2 of the centre cell c)
// (the second grid of an interlaced pair reaches one cell further down).
template <int P>
__host__ __device__ constexpr int reg_side(bool second) { return (P == 4 ? kTile + 3 : kTile + 2) + (second ? 1 : 0); }
template <int P>
__host__ __device__ constexpr int reg_cells(bool second) { return reg_side<P>(second) * reg_side<P>(second) * reg_side<P>(second); }

int assign_tiles_per_axis(int N) { return (N + kTile - 1) / kTile; }

// Centre cell of an object along one axis, u = (x - origin)/H: TSC taps
// c-1..c+1 around c = floor(u + 1/2); CIC taps c, c+1 with c = floor(u); PCS
// taps c-1..c+2 with c = floor(u).  The count, the scatter and the accumulation
// of an object must agree on its cell (its taps lie in its tile's region), also
// where u + 1/2 is within a rounding of a whole number, so every kernel takes it
// from here, with the roundings written out: left to the compiler, the product
// may join the sum in one FMA in one kernel and not in another.
template <int P>
__device__ __forceinline__ int centre_index(float x, float origin, float invH) {
  const float r = __fsub_rn(x, origin);
  return (int)floorf(P == 3 ? __fmaf_rn(r, invH, 0.5f) : __fmul_rn(r, invH));
}

// The centre cell along the three axes.  Returns false when a tap would leave
// [1, N-2] (non-periodic) or the position is not finite.
template <int P>
__device__ __forceinline__ bool centre_cell(const GeomDev& g, float px, float py, float pz, int& cx, int& cy,
                                            int& cz) {
  const float ux = (px - g.ox) * g.invH, uy = (py - g.oy) * g.invH, uz = (pz - g.oz) * g.invH;
  const int N = g.N;
  auto cells = [&] {
    cx = centre_index<P>(px, g.ox, g.invH);
    cy = centre_index<P>(py, g.oy, g.invH);
    cz = centre_index<P>(pz, g.oz, g.invH);
  };
  if (!g.periodic) {
    if (!(ux >= 0.f && ux < (float)N && uy >= 0.f && uy < (float)N && uz >= 0.f && uz < (float)N)) return false;
    cells();
    const int lo = P == 2 ? 1 : 2, hi = P == 4 ? N - 4 : N - 3;
    return cx >= lo && cy >= lo && cz >= lo && cx <= hi && cy <= hi && cz <= hi;
  }
  if (!(fabsf(ux) < 1e8f && fabsf(uy) < 1e8f && fabsf(uz) < 1e8f)) return false;
  cells();
  return true;
}

// i mod N in [0, N): indices within one box of the grid (all but periodic
// positions several boxes away) take the compare-and-add path, not a division.
__device__ __forceinline__ int wrapN(int i, int N) {
  if (i >= 0 && i < N) return i;
  if (i < 0 && i >= -N) return i + N;
  if (i >= N && i < 2 * N) return i - N;
  i %= N;
  return i < 0 ? i + N : i;
}

__device__ __forceinline__ int tile_of(int cx, int cy, int cz, int N, int ntx) {
  return ((wrapN(cz, N) / kTile) * ntx + wrapN(cy, N) / kTile) * ntx + wrapN(cx, N) / kTile;
}

// ---------------------------------------------------------------------------

// One launch for both catalogs: the first nbg blocks take the galaxies, the
// others the randoms (a launch for the galaxies alone leaves most SMs idle:
// 2e4 galaxies and 2e5 randoms took 19 + 26 us one after the other).  Each
// block owns a contiguous chunk of objects (the same chunks as the scatter
// launch on the same catalogs): its counts go to a shared-memory histogram
// over all tiles, written out whole as the block's row of bh.  TWO: the objects'
// cells in the second grid g2 of an interlaced pair are checked too.
constexpr int kBinThreads = 1024;

// f(x, y, z, nbar, w or 0) for the objects of [i0, i1).  WIDE: in runs of four
// per thread, one 16-byte load per array where every array of the catalog starts
// on a 16-byte boundary (chunks start at multiples of four) and four loads of 4
// bytes otherwise: the objects come to each thread in the same order either way,
// so its sums do not depend on where the caller's arrays lie.  Otherwise one by
// one.  3.57e7 objects, 512^3: the count launch and the scans behind it 0.55 ->
// 0.41 ms; the scatter gains nothing (four objects of a thread go to four places
// one after the other: 1.59 -> 1.64 ms with the accumulation) and takes them one
// by one.
template <bool WIDE, class F>
__device__ __forceinline__ void each_object(const CatDev& c, long long i0, long long i1, F&& f) {
  if (WIDE) {
    const long long n4 = i0 + ((i1 - i0) & ~3ll);
    const unsigned long long al = (unsigned long long)c.x | (unsigned long long)c.y | (unsigned long long)c.z |
                                  (unsigned long long)c.nbar | (unsigned long long)c.w;  // c.w may be null
    const bool wide = (al & 15) == 0;
    auto load4 = [](const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); };
    auto load1 = [](const float* p) { return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3)); };
#pragma unroll 1
    for (long long i = i0 + 4 * (long long)threadIdx.x; i < n4; i += 4 * (long long)blockDim.x) {
      float4 x, y, z, nb, w = make_float4(0.f, 0.f, 0.f, 0.f);
      if (wide) {
        x = load4(c.x + i); y = load4(c.y + i); z = load4(c.z + i); nb = load4(c.nbar + i);
        if (c.w) w = load4(c.w + i);
      } else {
        x = load1(c.x + i); y = load1(c.y + i); z = load1(c.z + i); nb = load1(c.nbar + i);
        if (c.w) w = load1(c.w + i);
      }
      f(x.x, y.x, z.x, nb.x, w.x);
      f(x.y, y.y, z.y, nb.y, w.y);
      f(x.z, y.z, z.z, nb.z, w.z);
      f(x.w, y.w, z.w, nb.w, w.w);
    }
    i0 = n4;
  }
#pragma unroll 4
  for (long long i = i0 + threadIdx.x; i < i1; i += blockDim.x)
    f(__ldg(c.x + i), __ldg(c.y + i), __ldg(c.z + i), __ldg(c.nbar + i), c.w ? __ldg(c.w + i) : 0.f);
}

template <int P, bool TWO>
__global__ void __launch_bounds__(kBinThreads) k_bin_count(CatDev cg, CatDev cr, int nbg, GeomDev g, GeomDev g2,
                                                           int ntx, int ntiles, double* __restrict__ part,
                                                           int* __restrict__ bh, int* __restrict__ err) {
  const int is_ran = (int)blockIdx.x >= nbg;
  const CatDev& c = is_ran ? cr : cg;
  extern __shared__ int hist[];
  __shared__ double sh[32];
  for (int t = threadIdx.x; t < ntiles; t += blockDim.x) hist[t] = 0;
  __syncthreads();
  FFSum s_w, s_w2, s_w3, s_nw2, s_n2w3;
  bool bad = false, apart = false;
  const int nblk = is_ran ? (int)gridDim.x - nbg : nbg, blk = is_ran ? (int)blockIdx.x - nbg : (int)blockIdx.x;
  const long long chunk = ((c.n + nblk - 1) / nblk + 3) & ~3ll;
  const long long i0 = blk * chunk < c.n ? blk * chunk : c.n;
  const long long i1 = i0 + chunk < c.n ? i0 + chunk : c.n;
  each_object<true>(c, i0, i1, [&](float px, float py, float pz, float nb, float wc) {
    const FF w = fkp_weight_ff(c.w != nullptr, wc, nb, g.P_fkp, g.P_fkp_lo);
    const FF w2 = ff_mul(w, w);
    const FF w3 = ff_mul(w2, w);
    s_w.add(w);
    s_w2.add(w2);
    s_w3.add(w3);
    if (is_ran) {
      const FF nw2 = ff_mul(w2, nb);
      s_nw2.add(nw2);
      s_n2w3.add(ff_mul(ff_mul(w3, nb), nb));
    }
    int cx, cy, cz;
    const bool in = centre_cell<P>(g, px, py, pz, cx, cy, cz);
    if (in)
      atomicAdd(hist + tile_of(cx, cy, cz, g.N, ntx), 1);
    else
      bad = true;
    if (TWO) {
      int dx, dy, dz;
      if (!in || !centre_cell<P>(g2, px, py, pz, dx, dy, dz)) bad = true;
      else if ((unsigned)(cx - dx) > 1u || (unsigned)(cy - dy) > 1u || (unsigned)(cz - dz) > 1u) apart = true;
    }
  });
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, 1);
  if (TWO && __syncthreads_or(apart) && threadIdx.x == 0) atomicOr(err + kErrApart, 1);
  int* row = bh + (size_t)blockIdx.x * ntiles;
  for (int t = threadIdx.x; t < ntiles; t += blockDim.x) row[t] = hist[t];
  double* out = part + (size_t)blockIdx.x * SC_NSUM;
  double v;
  if (!is_ran) {
    v = block_sum_f64(s_w.value(), sh);  if (threadIdx.x == 0) out[SC_G_W] = v;
    v = block_sum_f64(s_w2.value(), sh); if (threadIdx.x == 0) out[SC_G_W2] = v;
    v = block_sum_f64(s_w3.value(), sh); if (threadIdx.x == 0) out[SC_G_W3] = v;
  } else {
    v = block_sum_f64(s_w.value(), sh);    if (threadIdx.x == 0) out[SC_R_W] = v;
    v = block_sum_f64(s_w2.value(), sh);   if (threadIdx.x == 0) out[SC_R_W2] = v;
    v = block_sum_f64(s_w3.value(), sh);   if (threadIdx.x == 0) out[SC_R_W3] = v;
    v = block_sum_f64(s_nw2.value(), sh);  if (threadIdx.x == 0) out[SC_R_NW2] = v;
    v = block_sum_f64(s_n2w3.value(), sh); if (threadIdx.x == 0) out[SC_R_N2W3] = v;
  }
}

// Per tile t, over the rows of bh (one per block of the count launch,
// galaxies' blocks first): each row's entry becomes the exclusive prefix of
// the rows above it, and cnt[t] the tile's total.  A block takes 32 tiles (one
// 128-byte line per row) and cuts the rows among its 8 warps: 512^3, 304 rows
// of 32,768 tiles, 37 us with one thread per tile.
// The last block forms the scalars instead (ds not null): alpha, I_22, I_33,
// N_0, S_3 from the count blocks' FP64 partial sums, warp q the sum of
// quantity q in a fixed order (galaxy blocks [0, nbg), random blocks [nbg,
// nbg + nbr)); one thread per sum took 17 us.
__global__ void __launch_bounds__(256) k_tile_prefix(int* __restrict__ bh, int nrows, int ntiles,
                                                     int* __restrict__ cnt, const double* __restrict__ part, int nbg,
                                                     int nbr, long long ng, long long nr, int alpha_mode,
                                                     double* __restrict__ ds) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (ds && blockIdx.x == gridDim.x - 1) {
    __shared__ double tot[SC_NSUM];
    static_assert(SC_NSUM == 8, "one warp per sum");
    const bool gal = w <= SC_G_W3;
    const int b0 = gal ? 0 : nbg, nb = gal ? nbg : nbr;
    double v = 0.0;
    for (int b = lane; b < nb; b += 32) v += part[(size_t)(b0 + b) * SC_NSUM + w];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) tot[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      const double Wg = tot[SC_G_W], Wr = tot[SC_R_W];
      const double a = alpha_mode == 0 ? Wg / Wr : (double)ng / (double)nr;
      ds[DS_ALPHA] = a;
      ds[DS_I22] = a * tot[SC_R_NW2];
      ds[DS_I33] = a * tot[SC_R_N2W3];
      ds[DS_N0] = tot[SC_G_W2] + a * a * tot[SC_R_W2];
      ds[DS_N0FKP] = a * (1.0 + a) * tot[SC_R_W2];
      ds[DS_S3] = tot[SC_G_W3] - a * a * a * tot[SC_R_W3];
      ds[DS_WG] = Wg;
      ds[DS_WR] = Wr;
      ds[DS_NG] = (double)ng;
      ds[DS_NR] = (double)nr;
    }
    return;
  }
  __shared__ int sum[8][32];
  const int t = blockIdx.x * 32 + lane;
  const int per = (nrows + 7) / 8, r0 = w * per, r1 = min(nrows, r0 + per);
  int s = 0;
  if (t < ntiles) {
#pragma unroll 8
    for (int q = r0; q < r1; ++q) s += bh[(size_t)q * ntiles + t];
  }
  sum[w][lane] = s;
  __syncthreads();
  if (t >= ntiles) return;
  int run = 0;
  for (int k = 0; k < w; ++k) run += sum[k][lane];
  if (w == 7) cnt[t] = run + s;
#pragma unroll 8
  for (int q = r0; q < r1; ++q) {
    const int v = bh[(size_t)q * ntiles + t];
    bh[(size_t)q * ntiles + t] = run;
    run += v;
  }
}

// Exclusive scan of the tile counts into offsets (off[ntiles] = total), and
// of the tiles' work items (one per
// chunk objects or part of it) into item offsets (items[ntiles] = the
// number of items).  One block of 1024 threads walks the tiles in rounds of
// 1024 (coalesced loads, the next round's counts loaded during this round's
// warp-shuffle scan).
// occ (if not null) receives the rows that the occupied tiles reach (OccView),
// a tile counting as occupied when cnt or more (the cached random catalog's
// counts, or null) says so: a tile's objects reach its cells, one cell below
// and reach - kTile + 1 above, wrapped around a periodic box.  apart (with
// occ2): the flag of objects whose second-grid cells lie anywhere; the cached
// catalog's follows its counts.  The second grid then counts every row.
__global__ void __launch_bounds__(1024) k_scan_tiles(const int* __restrict__ cnt, int ntiles, int* __restrict__ off,
                                                     int* __restrict__ items, int chunk, const int* __restrict__ more, int ntx,
                                                     int N, int reach, int periodic, int* __restrict__ occ,
                                                     int* __restrict__ occ2, const int* __restrict__ apart) {
  __shared__ int wsum[32], wsumi[32];
  __shared__ int ty0[32], ty1[32];  // per plane of tiles: first and last occupied tile row
  __shared__ int zfirst, zlast;
  if (threadIdx.x < 32) {
    ty0[threadIdx.x] = 64;
    ty1[threadIdx.x] = -1;
  }
  if (threadIdx.x == 0) {
    zfirst = N;
    zlast = -1;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int carry = 0, carryi = 0;  // totals of the earlier rounds (the same in every thread)
  int c = (int)threadIdx.x < ntiles ? cnt[threadIdx.x] : 0;
  for (int base = 0; base < ntiles; base += 1024) {
    const int i = base + (int)threadIdx.x;
    const int cn = i + 1024 < ntiles ? cnt[i + 1024] : 0;
    const int ci = (c + chunk - 1) / chunk;
    if (occ) {
      // lanes of one row of tiles speak through their first occupied lane
      const bool full = i < ntiles && (c > 0 || (more && more[i] > 0));
      const unsigned m = __ballot_sync(0xffffffffu, full);
      const int q = i / ntx;
      const int q0 = __shfl_up_sync(0xffffffffu, q, 1);
      const unsigned starts = __ballot_sync(0xffffffffu, lane == 0 || q != q0);  // where a row begins in the warp
      if (full) {
        const unsigned upto = starts & (0xffffffffu >> (31 - lane));
        const int first = 31 - __clz(upto);  // this row's first lane
        if ((m & ((1u << lane) - 1u)) >> first == 0u) {
          const int tz = q / ntx, ty = q - tz * ntx;
          atomicMin(&ty0[tz], ty);
          atomicMax(&ty1[tz], ty);
        }
      }
    }
    int s = c, si = ci;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, s, o), vi = __shfl_up_sync(0xffffffffu, si, o);
      if (lane >= o) {
        s += v;
        si += vi;
      }
    }
    if (lane == 31) {
      wsum[warp] = s;
      wsumi[warp] = si;
    }
    __syncthreads();
    if (warp == 0) {
      int w = wsum[lane], wi = wsumi[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, w, o), vi = __shfl_up_sync(0xffffffffu, wi, o);
        if (lane >= o) {
          w += v;
          wi += vi;
        }
      }
      wsum[lane] = w;
      wsumi[lane] = wi;
    }
    __syncthreads();
    if (i < ntiles) {
      const int e = carry + (warp ? wsum[warp - 1] : 0) + s - c;
      off[i] = e;
      items[i] = carryi + (warp ? wsumi[warp - 1] : 0) + si - ci;
    }
    carry += wsum[31];
    carryi += wsumi[31];
    __syncthreads();
    c = cn;
  }
  if (threadIdx.x == 0) {
    off[ntiles] = carry;
    items[ntiles] = carryi;
  }
  if (!occ) return;
  // plane z = threadIdx.x (N <= 512): the hull of the rows of the tile planes
  // that reach it.  The second grid of an interlaced pair is filled from the
  // first grid's tiles, one cell further down (occ2).
  for (int low = 1; low <= (occ2 ? 2 : 1); ++low) {
    int* out = low == 1 ? occ : occ2;
    const bool all = low == 2 && (*apart || (more && more[ntiles]));
    const int z = threadIdx.x;
    __syncthreads();
    if (z == 0) {
      zfirst = N;
      zlast = -1;
    }
    __syncthreads();
    int y0 = N, y1 = 0;
    if (z < N) {
      for (int tz = 0; tz < ntx; ++tz) {
        if (ty1[tz] < 0) continue;
        const int a = tz * kTile - low, b = tz * kTile + reach;
        if (!((z >= a && z <= b) || (periodic && ((z - N >= a && z - N <= b) || (z + N >= a && z + N <= b))))) continue;
        const int ya = ty0[tz] * kTile - low, yb = ty1[tz] * kTile + reach;
        if (periodic && (ya < 0 || yb >= N)) {
          y0 = 0;
          y1 = N;
        } else {
          y0 = min(y0, max(ya, 0));
          y1 = max(y1, min(yb + 1, N));
        }
      }
      if (all) {
        y0 = 0;
        y1 = N;
      }
      if (y1 > y0) {
        atomicMin(&zfirst, z);
        atomicMax(&zlast, z);
      } else {
        y0 = y1 = 0;
      }
      out[4 + z] = y0 | (y1 << 16);
    }
    const int len = z < N ? y1 - y0 : 0;
    int sum = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, sum, o);
      if (lane >= o) sum += v;
    }
    if (lane == 31) wsum[warp] = sum;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += wsum[w];
    if (z < N) out[4 + N + z] = before + sum - len;
    if (z == N - 1) {
      out[0] = before + sum;
      out[1] = zlast < 0 ? 0 : zfirst;  // without objects: one plane of zeros
      out[2] = zlast < 0 ? 1 : zlast + 1;
      out[3] = 0;
    }
  }
}

// Each block owns the contiguous chunk of objects its count block counted:
// its range inside tile t's segment starts at off[t] plus the counts of the
// blocks before it (its row of the prefixed bh), so one pass over the chunk
// writes each object at the next slot of its tile's range.
// raw = 1 (randoms only): values w and w^2 without alpha, for the cached
// random grids that later mocks combine with their own alpha.
template <int P>
__global__ void __launch_bounds__(kBinThreads) k_bin_scatter(CatDev cg, CatDev cr, int nbg, int raw, GeomDev g,
                                                             int ntx, int ntiles, float obx, float oby, float obz,
                                                             const double* __restrict__ ds,
                                                             const int* __restrict__ off,
                                                             const int* __restrict__ bpref,
                                                             float4* __restrict__ xyzv, float* __restrict__ vw2,
                                                             double* __restrict__ labpart) {
  const int is_ran = (int)blockIdx.x >= nbg;
  const CatDev& c = is_ran ? cr : cg;
  extern __shared__ int hist[];
  __shared__ double sh[32];
  // alpha and alpha^2 as float pairs (hi + lo): each random's value is then
  // rounded once, at random, instead of carrying the FP32 rounding of alpha
  // into every random alike (a systematic scale of the random field)
  const double ad = raw ? 0.0 : ds[DS_ALPHA];
  const float alpha = (float)ad, alo = (float)(ad - (double)alpha);
  const float a2 = (float)(ad * ad), a2lo = (float)(ad * ad - (double)a2);
  const int nblk = is_ran ? (int)gridDim.x - nbg : nbg, blk = is_ran ? (int)blockIdx.x - nbg : (int)blockIdx.x;
  const long long chunk = ((c.n + nblk - 1) / nblk + 3) & ~3ll;
  const long long i0 = blk * chunk < c.n ? blk * chunk : c.n;
  const long long i1 = i0 + chunk < c.n ? i0 + chunk : c.n;
  const int* brow = bpref + (size_t)blockIdx.x * ntiles;
  for (int t = threadIdx.x; t < ntiles; t += blockDim.x) hist[t] = off[t] + brow[t];
  __syncthreads();
  KahanF lab[LAB_NSUM];
  each_object<false>(c, i0, i1, [&](float px, float py, float pz, float nb, float wc) {
    const float w = c.w ? wc : 1.0f / (1.0f + nb * g.P_fkp);
    int cx, cy, cz;
    if (centre_cell<P>(g, px, py, pz, cx, cy, cz)) {
      const int slot = atomicAdd(hist + tile_of(cx, cy, cz, g.N, ntx), 1);
      xyzv[slot] = make_float4(px, py, pz, is_ran && !raw ? -fmaf(alpha, w, alo * w) : w);
      if (vw2) {
        const float ww = w * w;
        vw2[slot] = is_ran && !raw ? fmaf(a2, ww, a2lo * ww) : ww;
      }
    }
    if (is_ran) {
      float hx, hy, hz;
      if (g.los_inf) {
        hx = g.lx; hy = g.ly; hz = g.lz;
      } else {
        const float dx = px - obx, dy = py - oby, dz = pz - obz;
        const float r2 = dx * dx + dy * dy + dz * dz;
        const float inv = r2 > 0.f ? rsqrtf(r2) : 0.f;
        hx = dx * inv; hy = dy * inv; hz = dz * inv;
      }
      lab[0].add(w * hx * hx);
      lab[1].add(w * hy * hy);
      lab[2].add(w * hz * hz);
      lab[3].add(w * hx * hy);
      lab[4].add(w * hy * hz);
      lab[5].add(w * hz * hx);
    }
  });
  if (is_ran) {
#pragma unroll
    for (int q = 0; q < LAB_NSUM; ++q) {
      const double v = block_sum_f64(lab[q].value(), sh);
      if (threadIdx.x == 0) labpart[(size_t)blk * LAB_NSUM + q] = v;
    }
  }
}

// Taps of an object along one axis: the first of its P cells and their weights,
// from its distance d = u - c to its centre cell c.
template <int P>
__device__ __forceinline__ void tap_weights(float x, float origin, float invH, int& i0, float* wt) {
  const int c = centre_index<P>(x, origin, invH);
  const float r = __fsub_rn(x, origin);
  const float d = P == 3 ? __fmaf_rn(r, invH, -(float)c) : __fsub_rn(__fmul_rn(r, invH), (float)c);
  i0 = P == 2 ? c : c - 1;
  if (P == 2) {
    wt[0] = 1.f - d;
    wt[1] = d;
  } else if (P == 3) {
    const float a = 0.5f - d, b = 0.5f + d;
    wt[0] = 0.5f * a * a;
    wt[1] = 0.75f - d * d;
    wt[2] = 0.5f * b * b;
  } else {
    // PCS: the cubic B-spline at distances 1 + d, d, 1 - d, 2 - d
    const float e = 1.f - d, d2 = d * d, d3 = d2 * d;
    wt[0] = e * e * e * (1.f / 6.f);
    wt[1] = (4.f - 6.f * d2 + 3.f * d3) * (1.f / 6.f);
    wt[2] = (1.f + 3.f * (d + d2 - d3)) * (1.f / 6.f);
    wt[3] = d3 * (1.f / 6.f);
  }
}

// x = round(v 2^40) as h 2^19 + l with FP32 arithmetic only (no conversion
// instructions): for |v| < 2, adding M = 1.5 2^23 to v 2^21 (one FMA, one
// rounding to nearest even) leaves h = round(v 2^21) in the low bits of the
// sum; the remainder v 2^21 - h is exact and lies in [-1/2, 1/2], and a
// second FMA leaves l = round((v 2^21 - h) 2^19) in [-2^18, 2^18] the same
// way.  h 2^19 + l is round(v 2^40), rounded to nearest even, exactly.
constexpr float kMagic = 12582912.0f;   // 1.5 2^23
constexpr int kMagicBits = 0x4B400000;  // its bit pattern
__device__ __forceinline__ void split_fixed(float v, int& h, int& l) {
  const float a = fmaf(v, 2097152.0f, kMagic);  // v 2^21 + M
  const float hf = a - kMagic;
  const float rem = fmaf(v, 2097152.0f, -hf);
  h = __float_as_int(a) - kMagicBits;
  l = __float_as_int(fmaf(rem, 524288.0f, kMagic)) - kMagicBits;
}

// x^_x^ea x^_y^eb x^_z^ec of the object at (o.x, o.y, o.z): its own line of
// sight about the observer (node 0 sits at origin - observer = (rx, ry, rz)
// from it), the fixed one for an observer at infinity; x^ = 0 at the
// observer itself.
__device__ __forceinline__ float ipow(float v, int e) {
  float r = 1.f;
  for (int k = 0; k < e; ++k) r *= v;
  return r;
}
__device__ __forceinline__ float object_moment(const GeomDev& g, const float4& o, int ea, int eb, int ec) {
  float hx = g.lx, hy = g.ly, hz = g.lz;
  if (!g.los_inf) {
    const float dx = (o.x - g.ox) + g.rx, dy = (o.y - g.oy) + g.ry, dz = (o.z - g.oz) + g.rz;
    const float r2 = dx * dx + dy * dy + dz * dz;
    const float inv = r2 > 0.f ? rsqrtf(r2) : 0.f;
    hx = dx * inv;
    hy = dy * inv;
    hz = dz * inv;
  }
  return ipow(hx, ea) * ipow(hy, eb) * ipow(hz, ec);
}

// Exponents (a, b, c) of the moment fields of a per-object plan: blockIdx.y picks the field, gridded N^3 cells after the one before
// (one launch for all 16: on a small survey a launch per field leaves most
// SMs idle, 128^3 and 2.2e5 objects 16 x 21 us).
struct MomentExp {
  unsigned long long a = 0, b = 0, c = 0;  // four bits per field
};

// One block per work item: up to chunk (<= kAccumChunk) objects of one tile (items in
// tile order; items[t] is tile t's first).  The tile's region, from one cell
// below the tile to the end of its reach (reg_side cells a side), covers the
// taps of every object whose centre cell lies in the tile.  Blocks past the
// last item return at once (the grid is sized from an upper bound).
//
// Each tap adds x = round(v 2^40) to its cell (v = w times the tap weight).
// Shared-memory adds of 64 bits are several times slower than adds of 32
// bits, and conversions to 64-bit integers run on a narrow pipe, so when the
// item allows it a cell is held as two signed 32-bit words from split_fixed:
// L sums the l (at most kAccumChunk < 2^13 terms of magnitude <= 2^18: |L| <
// 2^31) and H the h.  H stays exact while the item's sum S of |w| (an upper
// bound for any cell's sum of |v|, every tap weight being at most 1) is
// below 2^10 - 1: then |H| <= 2^21 S + 2^12 < 2^31.  split_fixed needs |v| <
// 2.  Items that fail either bound add x = round(v 2^40) as one 64-bit word
// instead.  Both forms give the exact integer sum of the x, so the grid does
// not depend on how the objects are split into items or in which order they
// are added.
//
// SECOND: the second grid of an interlaced pair (geometry g; the tiles are
// those of the first grid, whose origin is o1).  Its nodes lie half a cell
// further, so an object's centre cell there is its centre cell in the first
// grid or the one below: the region begins one cell lower, and the pair needs
// one count, scan and scatter instead of two (360^3 PCS, 3.5e7 randoms: 1.1 ms
// of 11.7).  A periodic box takes positions up to 1e8 cells away, where the two
// FP32 coordinates round apart (from 2^22 cells on their spacing is half a cell
// and more) and the second grid's cell may lie further down: such an object's
// taps go to the grid directly.
template <int P, bool W2, bool SECOND>
__global__ void __launch_bounds__(kAccumThreads, W2 ? 2 : 4) k_tile_accum(GeomDev g, float3 o1, int ntx, int ntiles,
                                                                        const int* __restrict__ off,
                                                                        const int* __restrict__ items,
                                                                        const float4* __restrict__ xyzv,
                                                                        const float* __restrict__ vw2,
                                                                        unsigned long long* __restrict__ grid,
                                                                        unsigned long long* __restrict__ gridw,
                                                                        int chunk, MomentExp xe,
                                                                        const double* __restrict__ labpart, int nlab,
                                                                        double* __restrict__ lab) {
  // the last block (one more than the items can be) sums L^ab instead, warp q
  // quantity q over the random blocks in a fixed order
  if (lab && blockIdx.x == gridDim.x - 1 && blockIdx.y == 0) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w >= LAB_NSUM) return;
    double v = 0.0;
    for (int b = lane; b < nlab; b += 32) v += labpart[(size_t)b * LAB_NSUM + w];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) lab[w] = v;
    return;
  }
  // moment field of a per-object plan (0: F)
  const int fld = blockIdx.y;
  const int ea = (int)(xe.a >> (4 * fld)) & 15, eb = (int)(xe.b >> (4 * fld)) & 15, ec = (int)(xe.c >> (4 * fld)) & 15;
  grid += (size_t)fld * g.N * g.N * g.N;
  constexpr int kLow = SECOND ? 2 : 1, kReg = reg_side<P>(SECOND), kReg3 = kReg * kReg * kReg;
  static_assert(kAccumChunk * 262144ll < 2147483648ll, "the low words would wrap");
  extern __shared__ unsigned long long reg[];
  __shared__ int s_tile;
  __shared__ float s_abs;
  __shared__ int s_max, s_apart;
  unsigned long long* regw = reg + kReg3;
  int* L = reinterpret_cast<int*>(reg);
  int* H = L + kReg3;
  int* Lw = reinterpret_cast<int*>(regw);
  int* Hw = Lw + kReg3;
  const int item = blockIdx.x;
  if (item >= items[ntiles]) return;
  if (threadIdx.x == 0) {
    // last tile whose first item is at or before this one
    int lo = 0, hi = ntiles - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (items[mid] <= item) lo = mid;
      else hi = mid - 1;
    }
    s_tile = lo;
    s_abs = 0.f;
    s_max = 0;
    s_apart = 0;
  }
  const int N = g.N;
  for (int i = threadIdx.x; i < kReg3; i += blockDim.x) {
    reg[i] = 0ull;
    if (W2) regw[i] = 0ull;
  }
  __syncthreads();
  const int t = s_tile;
  const int a = off[t] + (item - items[t]) * chunk;
  const int b = min(off[t + 1], a + chunk);
  const int tx = t % ntx, ty = (t / ntx) % ntx, tz = t / (ntx * ntx);
  const int lx0 = tx * kTile - kLow, ly0 = ty * kTile - kLow, lz0 = tz * kTile - kLow;
  // the item's objects are read twice: for the bounds, then for the taps
  float sa = 0.f, ma = 0.f;
  for (int i = a + threadIdx.x; i < b; i += kAccumThreads) {
    const float m = fmaxf(fabsf(xyzv[i].w), W2 ? fabsf(vw2[i]) : 0.f);
    sa += m;
    ma = fmaxf(ma, m);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sa += __shfl_xor_sync(0xffffffffu, sa, o);
    ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s_abs, sa);
    atomicMax(&s_max, __float_as_int(ma));  // non-negative: ordered as integers (NaN above +inf)
  }
  __syncthreads();
  // whether the P taps from (x, y, z) of the region lie in it
  auto inside = [](int x, int y, int z) {
    constexpr unsigned kLast = kReg - P;
    return (unsigned)x <= kLast && (unsigned)y <= kLast && (unsigned)z <= kLast;
  };
  // the bounds, with room for the rounding of the FP32 sums above
  const bool split = s_abs < 1000.f && __int_as_float(s_max) < 2.f;
  for (int i = a + threadIdx.x; i < b; i += kAccumThreads) {
    float4 o = xyzv[i];
    const float wv = W2 ? vw2[i] : 0.f;
    if (fld > 0) o.w *= object_moment(g, o, ea, eb, ec);  // |x^ products| <= 1: the bounds hold
    int ix, iy, iz;
    float wx[P], wy[P], wz[P];
    tap_weights<P>(o.x, g.ox, g.invH, ix, wx);
    tap_weights<P>(o.y, g.oy, g.invH, iy, wy);
    tap_weights<P>(o.z, g.oz, g.invH, iz, wz);
    // taps relative to the region (periodic positions may lie one box away)
    int cx = ix + (P >= 3 ? 1 : 0), cy = iy + (P >= 3 ? 1 : 0), cz = iz + (P >= 3 ? 1 : 0);
    if (SECOND) {  // the centre cell that chose the tile
      cx = centre_index<P>(o.x, o1.x, g.invH);
      cy = centre_index<P>(o.y, o1.y, g.invH);
      cz = centre_index<P>(o.z, o1.z, g.invH);
    }
    const int rx = ix - (cx - wrapN(cx, N)) - lx0;
    const int ry = iy - (cy - wrapN(cy, N)) - ly0;
    const int rz = iz - (cz - wrapN(cz, N)) - lz0;
    if (SECOND && !inside(rx, ry, rz)) {
      s_apart = 1;  // left for the loop below
      continue;
    }
    if (split) {
#pragma unroll
      for (int p = 0; p < P; ++p) {
#pragma unroll
        for (int q = 0; q < P; ++q) {
          const float wzy = wz[p] * wy[q];
          const int base = ((rz + p) * kReg + (ry + q)) * kReg + rx;
#pragma unroll
          for (int r = 0; r < P; ++r) {
            const float tw = wzy * wx[r];
            int h, l;
            split_fixed(o.w * tw, h, l);
            atomicAdd(L + base + r, l);
            atomicAdd(H + base + r, h);
            if (W2) {
              split_fixed(wv * tw, h, l);
              atomicAdd(Lw + base + r, l);
              atomicAdd(Hw + base + r, h);
            }
          }
        }
      }
    } else {
#pragma unroll
      for (int p = 0; p < P; ++p) {
#pragma unroll
        for (int q = 0; q < P; ++q) {
          const float wzy = wz[p] * wy[q];
          const int base = ((rz + p) * kReg + (ry + q)) * kReg + rx;
#pragma unroll
          for (int r = 0; r < P; ++r) {
            const float tw = wzy * wx[r];
            atomicAdd(reg + base + r, (unsigned long long)__float2ll_rn(o.w * tw * kFixScaleF));
            if (W2) atomicAdd(regw + base + r, (unsigned long long)__float2ll_rn(wv * tw * kFixScaleF));
          }
        }
      }
    }
  }
  __syncthreads();
  if (SECOND && s_apart) {
#pragma unroll 1
    for (int i = a + threadIdx.x; i < b; i += kAccumThreads) {
      const float4 o = xyzv[i];
      const float wv = W2 ? vw2[i] : 0.f;
      int ix, iy, iz;
      float wx[P], wy[P], wz[P];
      tap_weights<P>(o.x, g.ox, g.invH, ix, wx);
      tap_weights<P>(o.y, g.oy, g.invH, iy, wy);
      tap_weights<P>(o.z, g.oz, g.invH, iz, wz);
      const int cx = centre_index<P>(o.x, o1.x, g.invH), cy = centre_index<P>(o.y, o1.y, g.invH),
                cz = centre_index<P>(o.z, o1.z, g.invH);
      if (inside(ix - (cx - wrapN(cx, N)) - lx0, iy - (cy - wrapN(cy, N)) - ly0, iz - (cz - wrapN(cz, N)) - lz0))
        continue;
#pragma unroll
      for (int p = 0; p < P; ++p)
#pragma unroll
        for (int q = 0; q < P; ++q) {
          const float wzy = wz[p] * wy[q];
          const size_t row = ((size_t)wrapN(iz + p, N) * N + wrapN(iy + q, N)) * N;
#pragma unroll
          for (int r = 0; r < P; ++r) {
            const float tw = wzy * wx[r];
            const size_t gi = row + wrapN(ix + r, N);
            atomicAdd(grid + gi, (unsigned long long)__float2ll_rn(o.w * tw * kFixScaleF));
            if (W2) atomicAdd(gridw + gi, (unsigned long long)__float2ll_rn(wv * tw * kFixScaleF));
          }
        }
    }
  }
  for (int i = threadIdx.x; i < kReg3; i += blockDim.x) {
    unsigned long long v, vw = 0ull;
    if (split) {
      v = (unsigned long long)((long long)H[i] * 524288ll + (long long)L[i]);
      if (W2) vw = (unsigned long long)((long long)Hw[i] * 524288ll + (long long)Lw[i]);
    } else {
      v = reg[i];
      if (W2) vw = regw[i];
    }
    if (v == 0ull && vw == 0ull) continue;
    const int lx = i % kReg, ly = (i / kReg) % kReg, lz = i / (kReg * kReg);
    const size_t gi = ((size_t)wrapN(lz0 + lz, N) * N + wrapN(ly0 + ly, N)) * N + wrapN(lx0 + lx, N);
    if (v) atomicAdd(grid + gi, v);
    if (W2 && vw) atomicAdd(gridw + gi, vw);
  }
}

// F = G - alpha R and F^w = G^w + alpha^2 R^w (eqs. mapFFT, SNbisp2) from the
// galaxies' fixed-point grids G, G^w and the cached random grids R = sum_r w W,
// R^w = sum_r w^2 W: each random term is rounded once to the grid's 2^-40
// fixed point, so the result is as deterministic as a direct gridding.
__global__ void __launch_bounds__(256) k_combine_randoms(unsigned long long* __restrict__ grid,
                                                         const unsigned long long* __restrict__ rgrid,
                                                         unsigned long long* __restrict__ gridw,
                                                         const unsigned long long* __restrict__ rgridw,
                                                         const double* __restrict__ ds, long long n) {
  const double a = ds[DS_ALPHA];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    grid[i] = (unsigned long long)((long long)grid[i] - __double2ll_rn(a * (double)(long long)__ldg(rgrid + i)));
    if (gridw)
      gridw[i] = (unsigned long long)((long long)gridw[i] +
                                      __double2ll_rn(a * a * (double)(long long)__ldg(rgridw + i)));
  }
}

// ---------------------------------------------------------------------------
// launch wrappers
// ---------------------------------------------------------------------------

cudaError_t launch_combine_randoms(unsigned long long* grid, const unsigned long long* rgrid,
                                   unsigned long long* gridw, const unsigned long long* rgridw, const double* ds,
                                   long long n, int nsm, cudaStream_t s) {
  long long nb = (n + 255) / 256;
  if (nb > (long long)nsm * 16) nb = (long long)nsm * 16;
  k_combine_randoms<<<(int)nb, 256, 0, s>>>(grid, rgrid, gridw, rgridw, ds, n);
  return cudaGetLastError();
}

// Both catalogs in one launch, nbg + nbr blocks (nbg = 0: no galaxies, nbr = 0:
// the randoms are cached); part and bh: their nbg + nbr rows; g2: NULL, or the
// second grid of an interlaced pair, whose box limits are checked too.
cudaError_t launch_bin_count(const CatDev& gal, const CatDev& ran, int nbg, int nbr, const GeomDev& g,
                             const GeomDev* g2, double* part, int* bh, int* err, cudaStream_t s) {
  const int ntx = assign_tiles_per_axis(g.N);
  const int ntiles = ntx * ntx * ntx;
  const size_t sm = sizeof(int) * ntiles;
  const int nblk = nbg + nbr;
#define FKP_BC(PP, TWO)                                                                                             \
  do {                                                                                                              \
    raise_smem_limit((const void*)k_bin_count<PP, TWO>, sm);                                                        \
    k_bin_count<PP, TWO><<<nblk, kBinThreads, sm, s>>>(gal, ran, nbg, g, g2 ? *g2 : g, ntx, ntiles, part, bh, err); \
  } while (0)
#define FKP_BCP(PP)                                \
  do {                                             \
    if (g2) FKP_BC(PP, true); else FKP_BC(PP, false); \
  } while (0)
  if (g.assign == 2) FKP_BCP(2);
  else if (g.assign == 3) FKP_BCP(3);
  else FKP_BCP(4);
#undef FKP_BCP
#undef FKP_BC
  return cudaGetLastError();
}

// ds: NULL, or where the scalars go (formed from the nbg + nbr rows of part).
cudaError_t launch_tile_prefix(int* bh, int nrows, int ntiles, int* cnt, const double* part, int nbg, int nbr,
                               long long ng, long long nr, int alpha_mode, double* ds, cudaStream_t s) {
  k_tile_prefix<<<(ntiles + 31) / 32 + (ds ? 1 : 0), 256, 0, s>>>(bh, nrows, ntiles, cnt, part, nbg, nbr, ng, nr,
                                                                  alpha_mode, ds);
  return cudaGetLastError();
}

// Objects per work item of the tile accumulation: kAccumChunk for large
// catalogs (an item pays for clearing its region and adding it to the grid),
// less where that would leave SMs without an item: about eight items per SM,
// at least 512 objects (64^3, 2.2e5 objects: 33 us with one item per tile; with the
// other launches merged, the whole 64^3 mock 294 -> 237 us).
int accum_chunk(long long nobj, int nsm) {
  const long long c = nobj / (8ll * nsm);
  return (int)std::max<long long>(512, std::min<long long>(kAccumChunk, c));
}

cudaError_t launch_scan_tiles(const int* cnt, int ntiles, int* off, int* items, int chunk, cudaStream_t s,
                              const GeomDev& g, const int* more, int* occ, int* occ2, const int* err) {
  k_scan_tiles<<<1, 1024, 0, s>>>(cnt, ntiles, off, items, chunk, more, assign_tiles_per_axis(g.N), g.N,
                                  g.assign == 4 ? kTile + 1 : kTile, g.periodic, occ, occ2, err + kErrApart);
  return cudaGetLastError();
}

// off: the tile offsets; bpref: the nbg + nbr prefixed count rows.
cudaError_t launch_bin_scatter(const CatDev& gal, const CatDev& ran, int nbg, int nbr, const GeomDev& g,
                               const double obs[3], const double* ds, const int* off, const int* bpref, float4* xyzv,
                               float* vw2, double* labpart, cudaStream_t s, int raw) {
  const int ntx = assign_tiles_per_axis(g.N);
  const int ntiles = ntx * ntx * ntx;
  const size_t sm = sizeof(int) * ntiles;
  const int nblk = nbg + nbr;
#define FKP_SC(PP)                                                                                                 \
  do {                                                                                                             \
    raise_smem_limit((const void*)k_bin_scatter<PP>, sm);                                                          \
    k_bin_scatter<PP><<<nblk, kBinThreads, sm, s>>>(gal, ran, nbg, raw, g, ntx, ntiles, (float)obs[0],             \
                                                    (float)obs[1], (float)obs[2], ds, off, bpref, xyzv, vw2, labpart); \
  } while (0)
  if (g.assign == 2) FKP_SC(2);
  else if (g.assign == 3) FKP_SC(3);
  else FKP_SC(4);
#undef FKP_SC
  return cudaGetLastError();
}

// first: NULL, or the first grid of the interlaced pair whose second grid is g;
// nobj: the objects scattered into tile order (bounds the number of items);
// mt: the moment table of a per-object plan, or NULL; lab: NULL, or where the
// L^ab sums of the nlab rows of labpart go.
cudaError_t launch_tile_accum(const GeomDev& g, const int* off, const int* items, long long nobj, int chunk,
                              const float4* xyzv, const float* vw2, unsigned long long* grid,
                              unsigned long long* gridw, cudaStream_t s, const GeomDev* first, const MomentTable* mt,
                              const double* labpart, int nlab, double* lab) {
  MomentExp xe;
  static_assert(kMaxFields <= 16, "four bits per field in 64");
  for (int q = 0; mt && q < mt->nfields; ++q) {
    xe.a |= (unsigned long long)mt->e[q][0] << (4 * q);
    xe.b |= (unsigned long long)mt->e[q][1] << (4 * q);
    xe.c |= (unsigned long long)mt->e[q][2] << (4 * q);
  }
  const int ntx = assign_tiles_per_axis(g.N);
  const int ntiles = ntx * ntx * ntx;
  // every non-empty tile has one item that may be partial, the rest are full
  const long long nitems = std::min<long long>((long long)ntiles, nobj) + nobj / chunk + (lab ? 1 : 0);
  if (nitems <= 0) return cudaSuccess;
  if (nitems > INT32_MAX) return cudaErrorInvalidValue;
  const bool w2 = gridw != nullptr;
  const dim3 blocks((unsigned)nitems, mt ? mt->nfields : 1);
#define FKP_TA(PP, WW, SS)                                                                               \
  do {                                                                                                   \
    const size_t sm = sizeof(unsigned long long) * reg_cells<PP>(SS) * (WW ? 2 : 1);                     \
    raise_smem_limit((const void*)k_tile_accum<PP, WW, SS>, sm);                                         \
    k_tile_accum<PP, WW, SS><<<blocks, kAccumThreads, sm, s>>>(g, o1, ntx, ntiles, off, items, xyzv, vw2, grid, \
                                                               gridw, chunk, xe, labpart, nlab, lab);    \
  } while (0)
#define FKP_TAP(PP)                                                        \
  do {                                                                     \
    if (first) { if (w2) FKP_TA(PP, true, true); else FKP_TA(PP, false, true); } \
    else { if (w2) FKP_TA(PP, true, false); else FKP_TA(PP, false, false); }     \
  } while (0)
  const float3 o1 = first ? make_float3(first->ox, first->oy, first->oz) : make_float3(0.f, 0.f, 0.f);
  if (g.assign == 2) FKP_TAP(2);
  else if (g.assign == 3) FKP_TAP(3);
  else FKP_TAP(4);
#undef FKP_TAP
#undef FKP_TA
  return cudaGetLastError();
}

}  // namespace fkp
