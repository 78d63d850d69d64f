// k_contract_tc.cu - the triangle contraction of eq. Factorize on the
// tcgen05 tensor cores.
//
//   T^(l)(a,b,c) = sum_x F_a^(l)(x) F_b^(0)(x) F_c^(0)(x)
//
// is the skinny GEMM D[(b,c), (l,a)] = sum_x A[(b,c), x] B[(l,a), x] with
// A = the Khatri-Rao products F_b^(0) F_c^(0) and B = the shell fields.  Each
// FP32 operand v is split into BF16 v_hi = bf16(v), v_lo = bf16(v - v_hi); the
// three products hi*hi + hi*lo + lo*hi are accumulated in FP32 in tensor
// memory (the lo*lo term and the rounding of lo, each ~2^-18 relative, are
// dropped: a per-product error of random sign, which over N^3 points
// random-walks to ~2^-17 sqrt(sum_x t^2) on a triangle sum).  The 3-way
// split v = v_hi + v_mid + v_lo keeps the six products whose order is at most
// 2^-16 (hh, hm, mh, hl, lh, mm), for a per-term error near FP32 rounding:
// the triangle sums cancel strongly (sum |t| >> |sum t|), so the 3-way split
// is the accurate mode and the 2-way split the fast one.
//
// What bounds it, and the layout that follows from that.  The MMA work is
// small (a tile of 128 pairs needs only the fields a that close a triangle
// with one of them: the field rows are ordered a-major, so a tile's fields
// are one run of rows and one descriptor, 320 columns in all for 37 shells
// and three multipoles, where a (l,a) x (b,c) tiling issues 768); the cost is
// shared memory: building the products and feeding the operands.  So
//   - the pair products never touch shared memory: a thread owns a pair (a
//     tensor-memory lane), forms 32 points of its product in registers, splits
//     them and stores the BF16 parts to tensor memory (tcgen05.st), from where
//     the MMA reads its A operand;
//   - only the field operand B is staged in shared memory (its K-major parts,
//     21 KB per chunk of 32 points at 111 fields), built once per chunk for
//     all tiles of the block;
//   - the chunk's FP32 fields arrive as one TMA box (32 points x all fields,
//     128-byte swizzle: eight lanes reading one 16-byte column of eight
//     consecutive fields hit distinct banks).
// 24 warps, each with one role, meet on mbarriers: three warpgroups build A,
// each for a third of the tiles and into its own tensor-memory stage, with a
// warp each that issues those tiles' MMAs (one warp for all tiles sets the
// pace with its waits and commits: 29.1 ms at 360^3); one warpgroup builds B,
// one drains the accumulators, one warp issues the TMA loads.
// Tensor memory (512 columns): 176 accumulator columns, 176 columns of the
// running sums of the drained accumulators, 144 of A stages; tiles are
// packed into groups of at most 176 columns, one block per (group, K slice).
//
// Accumulation in tensor memory rounds (its error grows with the run length),
// so a tile's accumulator is drained - added with round to nearest to the
// running FP32 sum in tensor memory - after every run of tc_run(tiles) chunks
// (36 accumulating MMAs for three tiles and the 3-way split).  The tiles of a
// block drain at different chunks, so the tensor pipe seldom waits.  At the end of the slice the sums go
// to per-slice partials, summed over slices in FP64 by k_tc_reduce.
//
// Measured (3-way split, GB300): 37 shells x 3 multipoles on 360^3 48.3 ms with
// the products built into shared memory for (l,a) x (b,c) tiles of 128 x 256,
// 21.0 ms here (16.1 ms with the MMAs left out, 18.5 without the B build); 27
// shells x 1 on 512^3 83.7 -> 26.5 ms.  A chunk takes about 1,900 cycles of
// which a warpgroup computes 900: what is left is the handoffs (waits of 80 to
// 170 cycles each) between the roles.  The triangle sums are closer to the FP64
// ones than with runs of 96 MMAs (T_l 1.1e-6 to 1.8e-6 -> 0.5e-6 to 1.3e-6 over
// grids of 64^3 to 512^3, every split).
#include <algorithm>
#include <numeric>
#include <vector>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "fkp_internal.h"

namespace fkp {

constexpr int kTcM = 128;              // MMA rows: pairs (b, c) per tile
constexpr int kTcRows = 128;           // fields (l, a) at most
constexpr int kTcCols = 176;           // accumulator columns of a group of tiles
constexpr int kTcKC = 32;              // K points per chunk
constexpr int kTcSliceTarget = 2048;   // chunks per K slice, at most (about)
constexpr int kTcRing = 4;             // chunks of fields in flight
constexpr int kTcAWg = 3;              // warpgroups that build A, and warps that issue MMAs
constexpr int kTcThreads = (kTcAWg + 2) * 128 + (kTcAWg + 1) * 32;
constexpr int kTcPartRow = kTcRows + 16;           // rows of a B part (a tile's last rows may be padding)
constexpr int kTcPartBytes = kTcPartRow * kTcKC * 2;  // one BF16 part of B: 9 KB

// Chunks per accumulation run of a block with T tiles: a multiple of T when
// T <= 4, so that at most one tile drains per chunk, and 8 at most.
__host__ __device__ constexpr int tc_run(int T) { return T <= 2 ? 4 : (T <= 8 ? T : 8); }

// K slicing: the fewest whole waves of the SMs (groups x slices CTAs, one per
// SM at a time) whose slices hold at most about kTcSliceTarget chunks; slices
// of equal length (the last one shorter), none empty.
void tc_slicing(long long N3, int ngroups, int nsm, int* nslices, int* chunks) {
  const long long total = (N3 + kTcKC - 1) / kTcKC;
  const long long per_wave = (long long)nsm * kTcSliceTarget;
  const long long waves = std::max<long long>(1, (total * ngroups + per_wave - 1) / per_wave);
  long long ns = std::max<long long>(1, waves * nsm / std::max(1, ngroups));
  ns = std::min(ns, std::max<long long>(1, total));
  const long long ch = (total + ns - 1) / ns;
  *chunks = (int)ch;
  *nslices = (int)((total + ch - 1) / ch);
}
int tc_rows() { return kTcRows; }

// The tiles of a set of outputs.  Output o is the sum of field arow[o] = l S +
// a times the pair (fb, fc)[o].  Pairs are sorted by their first shell (the
// shells a that close with a pair begin there), cut into tiles of 128, and
// the tiles packed into groups of at most kTcCols accumulator columns.
TcPlan tc_plan(int S, int nl, const std::vector<int>& arow, const std::vector<short2>& pair) {
  TcPlan P;
  const int no = (int)arow.size();
  std::vector<int> ord(no);
  std::iota(ord.begin(), ord.end(), 0);
  auto key = [&](int o) { return ((pair[o].x % S) * 4 + pair[o].x / S) * S + pair[o].y; };
  std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) { return key(a) < key(b); });
  std::vector<int> idx(no, 0);
  std::vector<short2> list;
  for (int q = 0; q < no; ++q) {
    if (q == 0 || key(ord[q]) != key(ord[q - 1])) list.push_back(pair[ord[q]]);
    idx[ord[q]] = (int)list.size() - 1;
  }
  const int nt = ((int)list.size() + kTcM - 1) / kTcM;
  // each tile's run of field rows r = a nl + l, from a multiple of 8 (the
  // swizzle's period), a multiple of 16 columns
  auto row_of = [&](int o) { return (arow[o] % S) * nl + arow[o] / S; };
  std::vector<int> lo(nt, 1 << 20), hi(nt, -1);
  for (int o = 0; o < no; ++o) {
    const int t = idx[o] / kTcM, r = row_of(o);
    lo[t] = std::min(lo[t], r);
    hi[t] = std::max(hi[t], r);
  }
  std::vector<TcTile> tiles(nt);
  int cb = 0;
  for (int t = 0; t < nt; ++t) {
    tiles[t].r0 = lo[t] / 8 * 8;
    tiles[t].n = (hi[t] - tiles[t].r0) / 16 * 16 + 16;
    tiles[t].cb = cb;
    tiles[t].tile = t;
    cb += tiles[t].n;
  }
  P.ncols = cb;
  // first fit, widest first, each tile into the emptiest group that holds it
  std::vector<int> by(nt);
  std::iota(by.begin(), by.end(), 0);
  std::stable_sort(by.begin(), by.end(), [&](int a, int b) { return tiles[a].n > tiles[b].n; });
  int total = 0;
  for (auto& t : tiles) total += t.n;
  std::vector<int> used;
  for (int g = 0; g < std::max(1, (total + kTcCols - 1) / kTcCols); ++g) { P.groups.push_back(TcGroup{}); used.push_back(0); }
  for (int t : by) {
    int best = -1;
    for (int g = 0; g < (int)used.size(); ++g)
      if (used[g] + tiles[t].n <= kTcCols && (best < 0 || used[g] < used[best])) best = g;
    if (best < 0) { best = (int)used.size(); P.groups.push_back(TcGroup{}); used.push_back(0); }
    TcGroup& G = P.groups[best];
    tiles[t].col = used[best];
    used[best] += tiles[t].n;
    G.t[G.T++] = tiles[t];
  }
  P.groups.erase(std::remove_if(P.groups.begin(), P.groups.end(), [](const TcGroup& g) { return g.T == 0; }), P.groups.end());
  list.resize((size_t)nt * kTcM, make_short2(0, 0));  // padding lanes: any field (their rows of D are not read)
  P.pairs = list;
  P.off.resize(no);
  for (int o = 0; o < no; ++o) {
    const TcTile& t = tiles[idx[o] / kTcM];
    P.off[o] = (t.cb + row_of(o) - t.r0) * kTcM + idx[o] % kTcM;
  }
  return P;
}

// ---------------------------------------------------------------------------
// tcgen05 / TMEM wrappers
// ---------------------------------------------------------------------------

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A * B^T, A (BF16, 2 values per 32-bit column, lane = row) in
// tensor memory, B K-major BF16 in shared memory, FP32 accumulate.
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate, uint32_t elected) {
  asm volatile(
      "{\n .reg .pred p, e;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 e, %5, 0;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(elected)
      : "memory");
}

// 1 in one lane of the (converged) warp, 0 in the others.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
  return e;
}

__device__ __forceinline__ void umma_commit(uint64_t* bar, uint32_t elected) {
  asm volatile(
      "{\n .reg .pred e;\n setp.ne.b32 e, %1, 0;\n"
      " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_u32(bar)),
      "r"(elected)
      : "memory");
}

// 16 consecutive 32-bit columns of this warp's 32 tensor-memory lanes: load
// without the wait, the wait that completes every load in flight (naming the
// registers, so that no use of them moves ahead of it), and store.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Box of a 2-D tensor map to shared memory, completing on bar.
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// Shared-memory matrix descriptor: K-major operand with the 64-byte swizzle.
// Each row holds the chunk's 32 K values (64 bytes); 8 rows form a 512-byte
// swizzle atom (512 between atoms); the K steps of 16 advance the start
// address by 32 bytes within the rows.  Descriptor version 1, layout type
// SWIZZLE_64B (4) in bits 61-63.
// The address field counts 16-byte units in the low 14 bits (shared memory is
// far smaller than their reach), so an offset is added to the low word.
constexpr uint32_t kDescLo = 1u << 16, kDescHi = (512u >> 4) | (1u << 14) | (4u << 29);
__device__ __forceinline__ uint64_t sdesc(uint32_t lo) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(kDescHi));
  return d;
}

// Instruction descriptor for kind::f16: D FP32, A and B BF16, both K-major, M = 128.
__device__ __forceinline__ uint32_t tc_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTcM >> 4) << 24);
}

// Byte offset of the 16-byte segment (row, k-group kg) of an operand tile in
// the 64-byte-swizzled K-major layout: row r at 64 r, its 16-byte chunk kg
// stored at chunk kg ^ ((r >> 1) & 3) (address bits 4-5 XOR bits 7-8).  A
// quarter-warp storing 8 consecutive rows of one kg hits 8 distinct 16-byte
// bank groups.
__device__ __forceinline__ int canon_off(int row, int kg) {
  return row * 64 + ((kg ^ ((row >> 1) & 3)) << 4);
}

// Packed FP32 pairs.
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)));
  return *reinterpret_cast<float2*>(&r);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)));
  return *reinterpret_cast<float2*>(&r);
}

// BF16 split of two values into NS parts (each part the BF16 rounding of the
// remainder): w[p] packs part p of both.
template <int NS>
__device__ __forceinline__ void split2(float2 r, uint32_t* w) {
#pragma unroll
  for (int p = 0; p < NS; ++p) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(r.x, r.y);
    w[p] = *reinterpret_cast<const uint32_t*>(&h);
    if (p + 1 < NS) r = sub2(r, make_float2(__uint_as_float(w[p] << 16), __uint_as_float(w[p] & 0xffff0000u)));
  }
}

// ---------------------------------------------------------------------------

struct TcShared {
  uint64_t ring_full[kTcRing], ring_empty[kTcRing];
  uint64_t a_full[kTcAWg], a_empty[kTcAWg];
  uint64_t b_full[2], b_empty[2];
  uint64_t acc_full[kTcMaxTiles], acc_empty[kTcMaxTiles];
  uint64_t done[kTcAWg];
  uint32_t tmem;
  uint32_t packed[kTcMaxTiles];
  int abort;
  TcGroup g;
};

// A bounded wait by a warp (all lanes leave it together, with one answer);
// once one gives up (the error word is set) every other wait of the block
// gives up too.  A poll suspends the warp for up to kTcPollNs, so that waiting
// warps do not crowd the shared-memory pipe.
constexpr unsigned kTcPolls = 1u << 18, kTcPollNs = 20000;
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity, volatile int* abort, int* err) {
  for (unsigned it = 0; it < kTcPolls; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(kTcPollNs)
        : "memory");
    if (__all_sync(0xffffffffu, ok)) return true;
    if ((it & 15) == 15 && __any_sync(0xffffffffu, *abort)) return false;
  }
  *abort = 1;
  if ((threadIdx.x & 31) == 0) atomicOr(err, 16);
  return false;
}

template <int NS>
__global__ void __launch_bounds__(kTcThreads, 1) k_contract_tc(const __grid_constant__ CUtensorMap map, int nf, int S,
                                                               int nl, const TcGroup* __restrict__ groups,
                                                               const short2* __restrict__ pairs, long long nchunks,
                                                               int chunks, int ncols, float* __restrict__ part,
                                                               int* __restrict__ err) {
  extern __shared__ unsigned char smdyn[];
  unsigned char* smraw = smdyn + ((1024u - (smem_u32(smdyn) & 1023u)) & 1023u);  // the swizzles need 1024
  __shared__ TcShared sh;
  __shared__ short2 spair[kTcMaxTiles * kTcM];
  constexpr int kStageCols = NS * (kTcKC / 2);
  constexpr int kBStage = NS * kTcPartBytes;
  constexpr uint32_t kSum = kTcCols, kA0 = 2 * kTcCols;
  static_assert(2 * kTcCols + kTcAWg * kStageCols <= 512, "tensor memory columns");
  const int slot_bytes = (nf * kTcKC * 4 + 1023) & ~1023;
  unsigned char* ring = smraw;                            // kTcRing x [nf][32] FP32, 128-byte swizzle
  unsigned char* bst = smraw + kTcRing * slot_bytes;      // 2 x NS parts of B
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const long long c0 = (long long)blockIdx.y * chunks;
  const int nch = (int)(nchunks - c0 < chunks ? nchunks - c0 : chunks);
  if (tid == 0) {
    sh.g = groups[blockIdx.x];
    sh.abort = 0;
    for (int i = 0; i < groups[blockIdx.x].T; ++i) {
      const TcTile& t = groups[blockIdx.x].t[i];
      sh.packed[i] = (uint32_t)(t.col / 16) | (uint32_t)(t.r0 / 8) << 4 | (uint32_t)(t.n / 16) << 9;
    }
    for (int i = 0; i < kTcRing; ++i) {
      mbar_init(&sh.ring_full[i], 1);
      mbar_init(&sh.ring_empty[i], 4 * groups[blockIdx.x].T + 4);
    }
    for (int i = 0; i < kTcAWg; ++i) {
      mbar_init(&sh.a_full[i], 4);
      mbar_init(&sh.a_empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.b_full[i], 4);
      mbar_init(&sh.b_empty[i], groups[blockIdx.x].T < kTcAWg ? groups[blockIdx.x].T : kTcAWg);
    }
    for (int i = 0; i < kTcMaxTiles; ++i) {
      mbar_init(&sh.acc_full[i], 1);
      mbar_init(&sh.acc_empty[i], 4);
    }
    for (int i = 0; i < kTcAWg; ++i) mbar_init(&sh.done[i], 1);
    mbar_fence_init();
  }
  // rows of B past the last field stay zero
  for (int i = tid; i < 2 * kBStage / 16; i += kTcThreads) reinterpret_cast<uint4*>(bst)[i] = make_uint4(0, 0, 0, 0);
  if (warp == 0) {
    tmem_alloc(&sh.tmem, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  fence_proxy_async();
  __syncthreads();
  tc_fence_after();
  const int T = sh.g.T, R = tc_run(T);
  for (int i = tid; i < T * kTcM; i += kTcThreads) spair[i] = pairs[sh.g.t[i / kTcM].tile * kTcM + i % kTcM];
  __syncthreads();
  const uint32_t tm = sh.tmem;
  volatile int* ab = &sh.abort;

  if (warp < 4 * kTcAWg) {
    // ---- A: products of the pairs of the tiles t = w mod kTcAWg, in warpgroup
    // w's own stage of tensor memory, which MMA warp w reads
    const int row = tid & 127;
    const uint32_t lane_base = (uint32_t)(warp & 3) << 21;  // (warp % 4) * 32 lanes, in bits 16 and up
    const int wg = warp >> 2;
    const uint32_t stage = tm + lane_base + kA0 + wg * kStageCols;
    int t = wg, q = 0;
    for (int c = wg < T ? 0 : nch; c < nch; ++q) {
      const int s = c % kTcRing;
      const short2 bc = spair[t * kTcM + row];
      if (!tc_wait(&sh.ring_full[s], (uint32_t)(c / kTcRing) & 1, ab, err)) break;
      const unsigned char* pb = ring + s * slot_bytes + bc.x * 128;
      const unsigned char* pc = ring + s * slot_bytes + bc.y * 128;
      const int xb = bc.x & 7, xc = bc.y & 7;
      uint32_t w[NS][16];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 u = *reinterpret_cast<const float4*>(pb + ((j ^ xb) << 4));
        const float4 v = *reinterpret_cast<const float4*>(pc + ((j ^ xc) << 4));
        uint32_t o[NS];
        split2<NS>(mul2(make_float2(u.x, u.y), make_float2(v.x, v.y)), o);
#pragma unroll
        for (int p = 0; p < NS; ++p) w[p][2 * j] = o[p];
        split2<NS>(mul2(make_float2(u.z, u.w), make_float2(v.z, v.w)), o);
#pragma unroll
        for (int p = 0; p < NS; ++p) w[p][2 * j + 1] = o[p];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.ring_empty[s]);
      if (q > 0 && !tc_wait(&sh.a_empty[wg], (uint32_t)(q - 1) & 1, ab, err)) break;
      tc_fence_after();
#pragma unroll
      for (int p = 0; p < NS; ++p) tmem_st16(stage + p * 16, w[p]);
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.a_full[wg]);
      t += kTcAWg;
      if (t >= T) {
        t = wg;
        ++c;
      }
    }
  } else if (warp < 4 * (kTcAWg + 1)) {
    // ---- B: thread r splits field row r = a nl + l (field l S + a) into its K-major parts
    const int r = tid & 127;
    const bool act = r < nf;
    const int f = act ? (r % nl) * S + r / nl : 0;
    for (int c = 0; c < nch; ++c) {
      const int s = c % kTcRing, b = c & 1;
      if (!tc_wait(&sh.ring_full[s], (uint32_t)(c / kTcRing) & 1, ab, err)) break;
      if (c >= 2 && !tc_wait(&sh.b_empty[b], (uint32_t)((c >> 1) - 1) & 1, ab, err)) break;
      if (act) {
        const unsigned char* pf = ring + s * slot_bytes + f * 128;
        unsigned char* dst = bst + b * kBStage;
#pragma unroll
        for (int kg = 0; kg < 4; ++kg) {
          const float4 u = *reinterpret_cast<const float4*>(pf + (((2 * kg) ^ (f & 7)) << 4));
          const float4 v = *reinterpret_cast<const float4*>(pf + (((2 * kg + 1) ^ (f & 7)) << 4));
          uint32_t w[4][NS];
          split2<NS>(make_float2(u.x, u.y), w[0]);
          split2<NS>(make_float2(u.z, u.w), w[1]);
          split2<NS>(make_float2(v.x, v.y), w[2]);
          split2<NS>(make_float2(v.z, v.w), w[3]);
#pragma unroll
          for (int p = 0; p < NS; ++p)
            *reinterpret_cast<uint4*>(dst + p * kTcPartBytes + canon_off(r, kg)) =
                make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
        }
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sh.b_full[b]);
        mbar_arrive(&sh.ring_empty[s]);
      }
    }
  } else if (warp < 4 * (kTcAWg + 2)) {
    // ---- drains: accumulator of a finished run added to the tile's running sum
    const uint32_t base = tm + ((uint32_t)(warp & 3) << 21);
    uint32_t z[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) z[k] = 0u;
    for (int col = 0; col < kTcCols; col += 16) tmem_st16(base + kSum + col, z);
    tmem_wait_st();
    uint32_t par = 0;  // bit t: parity of tile t's next drain
    bool ok = true;
    int cr1 = R > 1 ? 1 : 0;  // (c + 1) mod R
    for (int c = 0; c < nch && ok; ++c) {
      for (int t = 0; t < T && ok; ++t) {
        if (c + 1 < nch && cr1 != (t < R ? t : t - R)) continue;
        ok = tc_wait(&sh.acc_full[t], (par >> t) & 1, ab, err);
        if (!ok) break;
        par ^= 1u << t;
        tc_fence_after();
        const uint32_t col = base + sh.g.t[t].col;
        for (int k = 0; k < sh.g.t[t].n; k += 16) {
          uint32_t v[16], u[16];
          tmem_ld16(col + k, v);
          tmem_ld16(col + kSum + k, u);
          tmem_wait_ld(v);
          tmem_wait_ld(u);
#pragma unroll
          for (int m = 0; m < 16; ++m) u[m] = __float_as_uint(__uint_as_float(u[m]) + __uint_as_float(v[m]));
          tmem_st16(col + kSum + k, u);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.acc_empty[t]);
      }
      if (++cr1 == R) cr1 = 0;
    }
    // the slice's sums: [slice][column][pair]
    if (ok) {
      for (int t = 0; t < T; ++t) {
        float* dst = part + ((size_t)blockIdx.y * ncols + sh.g.t[t].cb) * kTcM + (tid & 127);
        for (int k = 0; k < sh.g.t[t].n; k += 16) {
          uint32_t u[16];
          tmem_ld16(base + kSum + sh.g.t[t].col + k, u);
          tmem_wait_ld(u);
#pragma unroll
          for (int m = 0; m < 16; ++m) dst[(size_t)(k + m) * kTcM] = __uint_as_float(u[m]);
        }
      }
    }
  } else if (warp < 4 * (kTcAWg + 2) + kTcAWg) {
    // ---- MMAs: warp m issues those of the tiles t = m mod kTcAWg (a tile's are
    // in order that way).  The whole warp walks the jobs with warp-uniform
    // values (the operands are then in uniform registers), one lane issues.
    const int m = warp - 4 * (kTcAWg + 2);
    const uint32_t el = elect_one();
    // products (i, j) of A part i and B part j whose order is at most 2^-16
    constexpr int NP = NS == 2 ? 3 : 6;
    constexpr int pi[6] = {0, 0, 1, 0, 2, 1};
    constexpr int pj[6] = {0, 1, 0, 2, 0, 1};
    const uint32_t tmu = __shfl_sync(0xffffffffu, tm, 0);
    uint32_t par = 0;  // bit t: parity of the drain that tile t's next run waits for
    int q = 0, cr = 0, cr1 = R > 1 ? 1 : 0;  // job, c mod R, (c + 1) mod R
    const uint32_t bb0 = kDescLo | (smem_u32(bst) >> 4);
    bool ok = m < T;
    for (int c = 0; c < nch && ok; ++c) {
      const int b = c & 1;
      ok = tc_wait(&sh.b_full[b], (uint32_t)(c >> 1) & 1, ab, err);
      for (int t = m; t < T && ok; t += kTcAWg, ++q) {
        const int tr = t < R ? t : t - R;
        const bool first = c == 0 || cr == tr;
        // columns / 16, first row / 8 and width / 16 of the tile
        const uint32_t pk = __shfl_sync(0xffffffffu, sh.packed[t], 0);
        const uint32_t d = tmu + (pk & 15) * 16, a = tmu + kA0 + m * kStageCols;
        const uint32_t br = bb0 + b * (kBStage >> 4) + ((pk >> 4) & 31) * 32, id = tc_idesc((pk >> 9) * 16);
        ok = tc_wait(&sh.a_full[m], (uint32_t)q & 1, ab, err);
        if (ok && first && c > 0) {
          ok = tc_wait(&sh.acc_empty[t], (par >> t) & 1, ab, err);
          par ^= 1u << t;
        }
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int ks = 0; ks < kTcKC / 16; ++ks)
#pragma unroll
          for (int k = 0; k < NP; ++k)
            umma_bf16_ts(d, a + pi[k] * 16 + ks * 8, sdesc(br + ((pj[k] * kTcPartBytes + ks * 32) >> 4)), id,
                         (!first || ks > 0 || k > 0) ? 1u : 0u, el);
        umma_commit(&sh.a_empty[m], el);
        if (c + 1 == nch || cr1 == tr) umma_commit(&sh.acc_full[t], el);
      }
      if (ok) umma_commit(&sh.b_empty[b], el);
      cr = cr1;
      if (++cr1 == R) cr1 = 0;
    }
    // every MMA issued has finished before the tensor memory is freed
    umma_commit(&sh.done[m], el);
    mbar_wait(&sh.done[m], 0, err, 16);
    __syncwarp();
  } else {
    // ---- TMA: one box of fields per chunk
    const uint32_t bytes = (uint32_t)nf * kTcKC * 4;
    int c = 0;
    for (; c < nch; ++c) {
      const int s = c % kTcRing;
      if (c >= kTcRing && !tc_wait(&sh.ring_empty[s], (uint32_t)(c / kTcRing - 1) & 1, ab, err)) break;
      if (lane == 0) {
        mbar_expect_tx(&sh.ring_full[s], bytes);
        tma_load_2d(ring + s * slot_bytes, &map, (int)((c0 + c) * kTcKC), 0, &sh.ring_full[s]);
      }
      __syncwarp();
    }
    // copies in flight have landed before the block ends
    for (int k = c > kTcRing ? c - kTcRing : 0; k < c; ++k)
      mbar_wait(&sh.ring_full[k % kTcRing], (uint32_t)(k / kTcRing) & 1, err, 16);
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tm, 512);
}

// out[o] = sum over slices of the partials at off[o] (-1: 0).  A block takes 32
// outputs: 8 threads each sum every eighth slice, then in a fixed order.
__global__ void __launch_bounds__(256) k_tc_reduce(const float* __restrict__ part, int nslices, long long stride,
                                                   const int* __restrict__ off, int nout, double* __restrict__ out) {
  __shared__ double sh[8][33];
  const int o = blockIdx.x * 32 + threadIdx.x;
  const int p = o < nout ? off[o] : -1;
  double s = 0.0;
  if (p >= 0)
    for (int k = threadIdx.y; k < nslices; k += 8) s += (double)__ldg(part + k * stride + p);
  sh[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && o < nout) {
    for (int k = 1; k < 8; ++k) s += sh[k][threadIdx.x];
    out[o] = s;
  }
}

template <int NS>
static cudaError_t run_tc(const CUtensorMap& map, int nf, int S, int nl, const TcGroup* groups, int ngroups,
                          const short2* pairs, long long nchunks, int chunks, int nslices, int ncols, float* part,
                          int* err, cudaStream_t s) {
  const size_t sm = (size_t)kTcRing * ((nf * kTcKC * 4 + 1023) & ~1023) + 2 * NS * (size_t)kTcPartBytes + 1024;
  const cudaError_t e = raise_smem_limit((const void*)k_contract_tc<NS>, sm);
  if (e != cudaSuccess) return e;
  k_contract_tc<NS><<<dim3(ngroups, nslices), kTcThreads, sm, s>>>(map, nf, S, nl, groups, pairs, nchunks, chunks,
                                                                   ncols, part, err);
  return cudaGetLastError();
}

// I: the nf = nl S shell fields of N3 points each.
cudaError_t launch_contract_tc(const float* I, long long N3, int S, int nl, const TcGroup* groups, int ngroups,
                               const short2* pairs, int ncols, float* part, int* err, int nslices, int chunks,
                               int nsplit, cudaStream_t s) {
  const int nf = nl * S;
  typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                             const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                             CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qr;
  const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &qr);
  if (e != cudaSuccess) return e;
  if (qr != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
  // x = the points (a multiple of 8 of them: every field starts on a 16-byte
  // boundary; chunks start at multiples of 32; points past the end read as 0)
  CUtensorMap map;
  const cuuint64_t dim[2] = {(cuuint64_t)N3, (cuuint64_t)nf}, stride[1] = {(cuuint64_t)N3 * 4};
  const cuuint32_t box[2] = {kTcKC, (cuuint32_t)nf}, one[2] = {1, 1};
  if (reinterpret_cast<Encode>(fn)(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(I), dim, stride, box,
                                   one, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const long long nchunks = (N3 + kTcKC - 1) / kTcKC;
  return nsplit == 2 ? run_tc<2>(map, nf, S, nl, groups, ngroups, pairs, nchunks, chunks, nslices, ncols, part, err, s)
                     : run_tc<3>(map, nf, S, nl, groups, ngroups, pairs, nchunks, chunks, nslices, ncols, part, err, s);
}

cudaError_t launch_tc_reduce(const float* part, int nslices, int ncols, const int* off, int nout, double* out,
                             cudaStream_t s) {
  k_tc_reduce<<<(nout + 31) / 32, dim3(32, 8), 0, s>>>(part, nslices, (long long)ncols * kTcM, off, nout, out);
  return cudaGetLastError();
}

}  // namespace fkp
