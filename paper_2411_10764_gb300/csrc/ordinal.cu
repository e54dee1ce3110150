// Feature ordinals and the ordinal walk (layout and exactness: ordinal.cuh).
// XGBoost gbtree prediction (Sec. 3, Table 3) over rows, the caller's or those a
// decoded batch was written to: k_ordinals turns them into ordinals, k_walk_ord
// walks these.
#include <algorithm>
#include <cmath>

#include "ordinal.cuh"
#include "walk.cuh"

namespace mlt {
namespace {

using namespace walk;

constexpr int kOrdThreads = 1024;
constexpr int kOrdMaxCta = 1024;
constexpr int kOrdDeepUnit = 8;    // trees a tree group takes at a time
constexpr int kOrdDeepFlight = 4;  // trees a thread walks at once
constexpr size_t kSmPerSm = 228 * 1024;
constexpr size_t kCtaReserve = 1024;
constexpr size_t kStaticSmem = 1024;

// `steps` compares from the bucket's start: p += 2^k entries wherever the
// last of them is still <= x.  One load, one compare and one predicated add
// each (the offsets are immediates).
template <int K, int S>
__device__ __forceinline__ void ord_step(uint32_t (&p)[S], const float (&x)[S]) {
  float t[S];
#pragma unroll
  for (int r = 0; r < S; ++r)
    asm("ld.shared.f32 %0, [%1 + %2];" : "=f"(t[r]) : "r"(p[r]), "n"((4 << K) - 4));
#pragma unroll
  for (int r = 0; r < S; ++r)
    asm("{\n\t.reg .pred q;\n\tsetp.le.f32 q, %1, %2;\n\t@q add.u32 %0, %0, %3;\n\t}"
        : "+r"(p[r])
        : "f"(t[r]), "f"(x[r]), "n"(4 << K));
}
template <int S>
__device__ __forceinline__ void ord_search(uint32_t steps, uint32_t (&p)[S], const float (&x)[S]) {
  switch (steps) {
    case 13: ord_step<12>(p, x); [[fallthrough]];
    case 12: ord_step<11>(p, x); [[fallthrough]];
    case 11: ord_step<10>(p, x); [[fallthrough]];
    case 10: ord_step<9>(p, x); [[fallthrough]];
    case 9: ord_step<8>(p, x); [[fallthrough]];
    case 8: ord_step<7>(p, x); [[fallthrough]];
    case 7: ord_step<6>(p, x); [[fallthrough]];
    case 6: ord_step<5>(p, x); [[fallthrough]];
    case 5: ord_step<4>(p, x); [[fallthrough]];
    case 4: ord_step<3>(p, x); [[fallthrough]];
    case 3: ord_step<2>(p, x); [[fallthrough]];
    case 2: ord_step<1>(p, x); [[fallthrough]];
    case 1: ord_step<0>(p, x); break;
    default: break;
  }
}

// Rows without 16-byte alignment: a warp takes 32 rows and 8 features, a lane one
// feature of every fourth row (slot r: row 4 r + lane / 8), so a load covers
// four rows' 32 bytes where four scalar loads of a half row each touched 16
// lines.  Neighbouring lanes then exchange ordinals: an even lane stores the
// pair's word of slots 0, 2, 4, 6, the odd one of slots 1, 3, 5, 7.  300,007 x
// 101 with missing values, whole call: 540 us with scalar loads of half rows,
// 503 so.
template <bool HALF>
__device__ __forceinline__ void ord_unaligned(const OrdArgs& a, const OrdFeature* feat, uint32_t sm, int first, int f0,
                                              int nf, long long block, long long count, int F2, int F8) {
  const int lane = threadIdx.x & 31, h = lane & 7;
  const bool mine = f0 + h < nf;
  float x[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const long long i = block * 32 + r * 4 + (lane >> 3);
    const bool in = i < count && mine;
    const long long row = in ? (a.rows ? static_cast<long long>(a.rows[i]) : i) : 0;
    x[r] = in ? __ldg(a.feats + row * a.F + first + f0 + h) : 0.0f;
    if (HALF) x[r] = __half2float(__float2half_rn(x[r]));
  }
  const float4 o0 = __ldg(reinterpret_cast<const float4*>(feat + f0 + h));
  const uint4 o1 = __ldg(reinterpret_cast<const uint4*>(feat + f0 + h) + 1);
  const uint32_t base = __float_as_uint(o0.z), shift = __float_as_uint(o0.w);
  const uint32_t thr = sm + o1.z, lut = sm + o1.w;
  uint32_t p[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const uint32_t d = __float_as_uint(__fadd_rn(fmaxf(x[r], o0.x), o0.y)) - base;
    p[r] = thr + lds_u16(lut + min(d >> shift, o1.x) * 2u) * 4u;
  }
  ord_search(__shfl_sync(0xFFFFFFFFu, o1.y >> 8, 0), p, x);  // the compares of all eight features
  bool nan = false;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const bool missing = x[r] != x[r];
    nan |= missing;
    p[r] = missing ? kOrdNan : (p[r] - thr) >> 2;
  }
  const bool odd = lane & 1;
  uint32_t* dst = a.out + (block * F2 + ((first + f0 + h) >> 1)) * 32 + (lane >> 3);
#pragma unroll
  for (int r = 0; r < 8; r += 2) {
    // the even lane gives slot r + 1 and gets the odd lane's slot r
    const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, odd ? p[r] : p[r + 1], 1);
    const uint32_t word = odd ? (other | p[r + 1] << 16) : (p[r] | other << 16);
    if (f0 + (h & ~1) < nf) dst[(odd ? r + 1 : r) * 4] = word;
  }
  const bool any = __any_sync(0xFFFFFFFFu, nan);
  if (lane == 0) a.nan_flags[block * F8 + ((first + f0) >> 3)] = any ? 1 : 0;
}

// A CTA holds one feature group's thresholds and lookup tables in shared
// memory.  A warp takes 16 S rows and 8 features (one 32-byte sector of each
// row) at a time: lanes 2i and 2i + 1 read the two halves of a row's sector
// together (16 lines a load, where a lane per row would touch 32), so an even
// lane searches features 0-3 and an odd one 4-7, S rows of a feature together
// (S chains in flight; its parameters are read once for them).
// Groups get CTAs in proportion to their features.  Bound: the L1 data pipe,
// about 14 wavefronts of table loads and 5 of row loads per 32 values.  V's
// ordinals of 1,048,576 x 128 take 0.315 ms (0.344 with four rows a lane; 0.72
// with a lane per row and feature parameters per row pair).  S is 8, or 4 where
// that leaves warps without work (20,011 x 47, whole call: 71.3 us with 8, 69.7
// with 4).
template <bool VEC, bool HALF, int S>
__global__ void __launch_bounds__(kOrdThreads, 1) k_ordinals(const __grid_constant__ OrdArgs a) {
  constexpr int kRows = VEC ? S / 2 : 1;  // blocks of 32 rows a warp takes together
  static_assert(VEC || S == 8, "unaligned rows: 8 slots of 4 rows");
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long bar, never;  // never completed (self-test)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int gi = 0;
  for (int hi = a.n_groups; gi + 1 < hi;) {
    const int mid = (gi + hi) >> 1;
    if (blockIdx.x >= a.first_cta[mid])
      gi = mid;
    else
      hi = mid;
  }
  const int slab = blockIdx.x - a.first_cta[gi], slabs = a.first_cta[gi + 1] - a.first_cta[gi];
  const OrdGroup g = a.groups[gi];
  if (tid == 0) {
    mbar_init(smem_u32(&bar), 1);
    mbar_init(smem_u32(&never), 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (tid == 0 && g.bytes > 0) {  // thresholds are static: before waiting on earlier kernels
    mbar_expect_tx(smem_u32(&bar), g.bytes);
    bulk_copy_g2s(smem_u32(smem), a.image + g.off, g.bytes, smem_u32(&bar));
  }
  pdl_wait();
  pdl_trigger();
  const bool skip = a.stream && *reinterpret_cast<volatile const unsigned*>(&a.stream->done);
  const long long count = skip ? 0 : a.count ? static_cast<long long>(*a.count) : a.n;
  const long long blocks = (count + 31) >> 5;
  const int F2 = (a.F + 1) >> 1, F8 = (a.F + 7) >> 3;
  const int nf = static_cast<int>(g.count), chunks = (nf + 7) >> 3;
  const uint32_t items = static_cast<uint32_t>((blocks + kRows - 1) / kRows) * chunks;  // n x F fits memory
  const OrdFeature* feat = a.features + g.first;
  const uint32_t step = slabs * (blockDim.x >> 5);
  const uint32_t sm = smem_u32(smem);
  // every warp waits for the copy, also one without rows: it must land before
  // the CTA's shared memory is released.  A CTA that gives up leaves the buffer's
  // earlier contents in its share, so it marks the call's ordinals as failed: the
  // walk then takes no candidate as valid.
  const bool stall = a.stall_ns > 0 && blockIdx.x == 0;
  const bool here = stall ? mbar_wait_bounded_ns(smem_u32(&never), 0u, a.stall_ns)
                          : g.bytes == 0 || mbar_wait_bounded(smem_u32(&bar), 0u);
  if (!__all_sync(0xFFFFFFFFu, here)) {
    if (g.bytes > 0) mbar_wait_bounded(smem_u32(&bar), 0u);
    if (lane == 0) {
      atomicOr(a.failed, 1u);
      atomicOr(a.err, kErrWaitTimeout);
    }
    return;
  }
  for (uint32_t it = warp * slabs + slab; it < items; it += step) {
    const uint32_t s32 = it / static_cast<uint32_t>(chunks);
    const int f0 = static_cast<int>(it - s32 * chunks) * 8;
    const long long sb = s32;
    if constexpr (!VEC) {
      ord_unaligned<HALF>(a, feat, sm, static_cast<int>(g.first), f0, nf, sb, count, F2, F8);
      continue;
    }
    // row slot r of this lane: row 16 r + lane / 2 of the item; features h0 .. h0 + 3
    const int h0 = f0 + (lane & 1) * 4;
    float x[4][S];  // [feature][row slot]
#pragma unroll
    for (int r = 0; r < S; ++r) {
      const long long i = sb * (kRows * 32) + r * 16 + (lane >> 1);
      const bool in = i < count && h0 < nf;
      const long long row = in ? (a.rows ? static_cast<long long>(a.rows[i]) : i) : 0;
      const float* src = a.feats + row * a.F + g.first + h0;
      const float4 v = in ? __ldg(reinterpret_cast<const float4*>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
      x[0][r] = v.x;
      x[1][r] = v.y;
      x[2][r] = v.z;
      x[3][r] = v.w;
    }
    // ordinals of a row slot: words of pairs (h0, h0 + 1) and (h0 + 2, h0 + 3)
    uint32_t* dst = a.out + (sb * kRows * F2 + ((g.first + h0) >> 1)) * 32 + (lane >> 1);
    uint32_t missing = 0;  // bits: row slots of this lane that hold a missing value
    uint32_t word[S];
#pragma unroll
    for (int h = 0; h < 4; ++h) {  // the table is padded to a multiple of 8 features
      const float4 o0 = __ldg(reinterpret_cast<const float4*>(feat + h0 + h));
      const uint4 o1 = __ldg(reinterpret_cast<const uint4*>(feat + h0 + h) + 1);
      const uint32_t base = __float_as_uint(o0.z), shift = __float_as_uint(o0.w);
      const uint32_t thr = sm + o1.z, lut = sm + o1.w;
      uint32_t p[S];
#pragma unroll
      for (int r = 0; r < S; ++r) {
        if (HALF) x[h][r] = __half2float(__float2half_rn(x[h][r]));
        const uint32_t d = __float_as_uint(__fadd_rn(fmaxf(x[h][r], o0.x), o0.y)) - base;
        p[r] = thr + lds_u16(lut + min(d >> shift, o1.x) * 2u) * 4u;
      }
      // lanes 2i search feature h0 + h, lanes 2i + 1 feature h0 + h + 4, which
      // has the same number of steps
      ord_search(__shfl_sync(0xFFFFFFFFu, o1.y & 0xFFu, 0), p, x[h]);
      bool nan = false;
#pragma unroll
      for (int r = 0; r < S; ++r) nan |= x[h][r] != x[h][r];
      if (nan) {
#pragma unroll
        for (int r = 0; r < S; ++r)
          if (x[h][r] != x[h][r]) {
            p[r] = thr + kOrdNan * 4u;
            missing |= 1u << r;
          }
      }
      // (p - thr) / 4 of the pair in the low and high halves
#pragma unroll
      for (int r = 0; r < S; ++r)
        word[r] = (h & 1) == 0 ? (p[r] - thr) >> 2 : word[r] + ((p[r] - thr) << 14);
      if ((h & 1) == 1 && h0 + h - 1 < nf) {
        // row slots 2b, 2b + 1 are the halves of block b of the item
#pragma unroll
        for (int r = 0; r < S; ++r)
          if (sb * kRows + (r >> 1) < blocks) dst[((r >> 1) * F2 + (h >> 1)) * 32 + (r & 1) * 16] = word[r];
      }
    }
    missing = __reduce_or_sync(0xFFFFFFFFu, missing);
    if (lane < kRows && sb * kRows + lane < blocks)
      a.nan_flags[(sb * kRows + lane) * F8 + ((g.first + f0) >> 3)] = (missing >> (2 * lane)) & 3u ? 1 : 0;
  }
}

// A candidate's ordinals: its warp's blocks and its lane's bytes in a row of
// them.  Bits 2 to 6 of a word's offset are zero, so the lane is merged by the
// operation that masks the offset and the warp-uniform base goes into the
// load's address: one integer operation a visit less than adding a pointer.
struct OrdRow {
  const unsigned char* warp;
  uint32_t lane4;
};
// The ordinal that a node word tests.
__device__ __forceinline__ uint32_t ord_at(const OrdRow& x, uint32_t w) {
  return ld_sm<unsigned short>(x.warp, (w & 0xFFFEu) | x.lane4);
}
// Heap index of the child that ordinal x takes below node i; a missing x
// (kOrdNan) becomes 0 where the word's flag sends it left.
template <bool NANP>
__device__ __forceinline__ uint32_t ord_child(uint32_t i, uint32_t w, uint32_t x) {
  if (NANP) x &= ~(w << 15);
  return __funnelshift_l(w - x * 65536u, i, 1);
}
// The same for a deep model's words, whose flag is at kOrdNan's bit.
__device__ __forceinline__ uint32_t deep_at(const OrdRow& x, uint32_t w) {
  return ld_sm<unsigned short>(x.warp, (w & 0x7FFEu) | x.lane4);
}
template <bool NANP>
__device__ __forceinline__ uint32_t deep_child(uint32_t i, uint32_t w, uint32_t x) {
  if (NANP) x &= ~(w & kOrdNan);
  return __funnelshift_l(w - x * 65536u, i, 1);
}

// A 32-byte block (one sector), kept in L2.
__device__ __forceinline__ void ldg_block(const uint4* ptr, unsigned long long pol, uint32_t (&b)[8]) {
  asm("ld.global.nc.L2::cache_hint.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
      : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7])
      : "l"(ptr), "l"(pol));
}

// Leaves of G consecutive trees at tb for one candidate.
template <int D, int G, bool NANP>
__device__ __forceinline__ void walk_ord(const unsigned char* tb, const OrdRow& xw, float* leaf) {
  constexpr uint32_t kTree = ord_tree_bytes(D);
  uint32_t j[G];
#pragma unroll
  for (int g = 0; g < G; ++g) j[g] = 1u;
#pragma unroll
  for (int l = 0; l < D; ++l) {
    uint32_t w[G], x[G];
#pragma unroll
    for (int g = 0; g < G; ++g) w[g] = ld_sm<uint32_t>(tb, g * kTree + j[g] * 4u);
#pragma unroll
    for (int g = 0; g < G; ++g) x[g] = ord_at(xw, w[g]);
#pragma unroll
    for (int g = 0; g < G; ++g) j[g] = ord_child<NANP>(j[g], w[g], x[g]);
  }
#pragma unroll
  for (int g = 0; g < G; ++g) leaf[g] = ld_sm<float>(tb, g * kTree + j[g] * 4u);
}

// Leaves of nt <= U trees (a multiple of 4), up to 8 trees in flight.
template <int D, int U, bool NANP>
__device__ __forceinline__ void walk_ord_unit(const unsigned char* tb, int nt, const OrdRow& xw, float* leaf) {
  constexpr uint32_t kTree = ord_tree_bytes(D);
#pragma unroll
  for (int t = 0; t < U; t += 8) {
    if (U >= 8 && nt >= t + 8)
      walk_ord<D, U >= 8 ? 8 : 4, NANP>(tb + t * kTree, xw, leaf + t);
    else if (nt > t)
      walk_ord<D, 4, NANP>(tb + t * kTree, xw, leaf + t);
  }
}

// Leaves of G consecutive trees of a deep model: H head levels and the exit
// from shared memory, then `rounds` blocks of three levels from global memory.
// Every walker runs every round -- some lane of a warp nearly always goes to
// the bottom, and a vote per round would tie the G walkers' loads together; a
// walker that has its leaf reads block 0, one line for all of them.  Bound: the
// L1 data pipe, about 23 wavefronts a warp and tree for the head and 38 for
// the tail (4,194,304 x 256, 1,000 trees of depth 12: 73 cycles a warp and tree
// on an SM, where the split table's 8-byte records took 94).
template <int H, int G, bool NANP>
__device__ __forceinline__ void walk_ord_deep(const unsigned char* tb, const OrdRow& xw, const uint4* tail,
                                              int rounds, float* leaf) {
  constexpr uint32_t kTree = ord_head_bytes(H);
  uint32_t j[G];
#pragma unroll
  for (int g = 0; g < G; ++g) j[g] = 1u;
#pragma unroll
  for (int l = 0; l < H; ++l) {
    uint32_t w[G], x[G];
#pragma unroll
    for (int g = 0; g < G; ++g) w[g] = ld_sm<uint32_t>(tb, g * kTree + j[g] * 4u);
#pragma unroll
    for (int g = 0; g < G; ++g) x[g] = deep_at(xw, w[g]);
#pragma unroll
    for (int g = 0; g < G; ++g) j[g] = deep_child<NANP>(j[g], w[g], x[g]);
  }
  uint32_t val[G], at[G];
  bool live[G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    // exit j - 2^H of the tree: 8 bytes at (4 << H) + 8 (j - 2^H)
    const uint2 e = ld_sm<uint2>(tb, g * kTree + j[g] * 8u - (4u << H));
    live[g] = !(e.y & kOrdExitLeaf);
    val[g] = e.x;
    const uint32_t w = live[g] ? e.x : 0u;  // a leaf's bits are no index
    at[g] = live[g] ? e.y + (deep_child<NANP>(0u, w, deep_at(xw, w)) & 1u) : 0u;
  }
  const unsigned long long keep = policy_evict_last();
  for (int s = 0; s < rounds; ++s) {
    uint32_t b[G][8], i[G], w[G];
#pragma unroll
    for (int g = 0; g < G; ++g) ldg_block(tail + 2ull * at[g], keep, b[g]);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      i[g] = 1u;
      w[g] = b[g][1];
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      uint32_t x[G];
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const bool is_leaf = ((b[g][0] >> i[g]) & (1u << (kOrdBlockBits - 1))) != 0u;
        if (is_leaf && live[g]) val[g] = w[g];
        live[g] = live[g] && !is_leaf;
        w[g] = is_leaf ? 0u : w[g];
        x[g] = deep_at(xw, w[g]);
      }
#pragma unroll
      for (int g = 0; g < G; ++g) {
        i[g] = deep_child<NANP>(i[g], w[g], x[g]);
        if (l == 0) w[g] = (i[g] & 1u) ? b[g][3] : b[g][2];
        if (l == 1) {
          const uint32_t lo = (i[g] & 1u) ? b[g][5] : b[g][4], hi = (i[g] & 1u) ? b[g][7] : b[g][6];
          w[g] = (i[g] & 2u) ? hi : lo;
        }
      }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) at[g] = live[g] ? (b[g][0] & ((1u << kOrdBlockBits) - 1u)) + i[g] - 8u : 0u;
  }
#pragma unroll
  for (int g = 0; g < G; ++g) leaf[g] = __uint_as_float(val[g]);
}

// Leaves of nt <= U trees (a multiple of 4) of a deep model.
template <int H, int U, int G, bool NANP>
__device__ __forceinline__ void walk_deep_unit(const unsigned char* tb, int nt, const OrdRow& xw,
                                               const uint4* tail, int rounds, float* leaf) {
#pragma unroll
  for (int t = 0; t < U; t += G)
    if (nt > t) walk_ord_deep<H, G, NANP>(tb + t * ord_head_bytes(H), xw, tail, rounds, leaf + t);
}

// One tree group: trees [0, nt) of a chunk, leaves added in tree order.
template <int D, bool NANP>
__device__ __forceinline__ float walk_ord_sum(const unsigned char* tb, int nt, const OrdRow& xw, float acc) {
  constexpr uint32_t kTree = ord_tree_bytes(D);
  int t = 0;
  for (; t + 8 <= nt; t += 8) {
    float leaf[8];
    walk_ord<D, 8, NANP>(tb + static_cast<uint32_t>(t) * kTree, xw, leaf);
#pragma unroll
    for (int g = 0; g < 8; ++g) acc += leaf[g];
  }
  if (t < nt) {  // trees are padded to 4
    float leaf[4];
    walk_ord<D, 4, NANP>(tb + static_cast<uint32_t>(t) * kTree, xw, leaf);
#pragma unroll
    for (int g = 0; g < 4; ++g) acc += leaf[g];
  }
  return acc;
}

struct OrdSmem {
  size_t rows, sums, tbuf, bars, bytes;
};
// Q > 0: tree groups that hand the sums on (the candidates' running sums and a
// barrier per group and 32 candidates); 0: one group that keeps them.
__host__ __device__ inline OrdSmem ord_smem(int F, int TC, int Q, int nbuf, uint32_t chunk_bytes) {
  OrdSmem s;
  s.rows = static_cast<size_t>((F + 1) / 2) * TC * 4;  // a multiple of 128: TC is one of 32
  s.sums = s.rows + static_cast<size_t>(TC) * 4;
  s.tbuf = align_up(s.sums + (Q > 0 ? static_cast<size_t>(TC) * 4 : 0), 128);
  s.bars = s.tbuf + static_cast<size_t>(nbuf) * chunk_bytes;
  s.bytes = s.bars + 10 * 8 + static_cast<size_t>(TC / 32) * Q * 8;
  return s;
}

// The tile of a CTA in blocks of 32 candidates.  V pass: TC candidates each
// (the tile counts are scanned and scattered by tile).  P pass: the blocks of
// the survivors split evenly over whole waves of CTAs, as in cta_tile.
__device__ __forceinline__ void ord_tile(const TraverseArgs& a, long long count, int TC, long long* tile0, int* len) {
  if (!a.p_pass) {
    cta_tile(a, count, TC, tile0, len);
    return;
  }
  const uint32_t nb = (static_cast<uint32_t>(count) + 31u) >> 5, per = static_cast<uint32_t>(TC) >> 5;
  const uint32_t wave = a.p_wave > 0 ? static_cast<uint32_t>(a.p_wave) : gridDim.x;
  const uint32_t waves = (nb + per * wave - 1) / (per * wave);
  const uint32_t tiles = min(min(waves * wave, nb), gridDim.x);
  if (blockIdx.x >= tiles) {
    *tile0 = count;
    *len = 0;
    return;
  }
  const uint32_t lo = split_start(nb, tiles, blockIdx.x), hi = split_start(nb, tiles, blockIdx.x + 1);
  *tile0 = static_cast<long long>(lo) * 32;
  *len = static_cast<int>(min(static_cast<long long>(hi) * 32, count) - *tile0);
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrive on an mbarrier; returns the arrivals that were still pending before.
__device__ __forceinline__ uint32_t mbar_arrive_pending(uint32_t bar) {
  uint32_t pending;
  asm volatile(
      "{\n\t.reg .b64 st;\n\t"
      "mbarrier.arrive.shared::cta.b64 st, [%1];\n\t"
      "mbarrier.pending_count.b64 %0, st;\n\t}"
      : "=r"(pending)
      : "r"(bar)
      : "memory");
  return pending;
}

// One CTA = a tile of TC candidates and Q groups of TC threads: the tile's
// ordinals arrive in one bulk copy, the trees in chunks through nbuf buffers
// (a warp arrives on the buffer's second barrier when it is done with it, and
// the last one to arrive refills it).  The groups take units of U trees in
// turn (U = 0: one group, the sum stays in its register).  With Q > 1 a
// candidate's sum goes from group to group: a warp walks its unit, waits for the
// sum of the trees before it, adds its leaves in tree order and hands the sum on
// -- the same sequential fp32 sum as one walker.
// A warp issues an instruction every other cycle at best, so the groups
// multiply the warps where a tile's candidates alone leave an SM too few.
// Bound: shared-memory wavefronts (one per ordinal gather, one to 3.4 per node
// gather) and issue.
// DEEP: a deep model's heads (D head levels) and tail.
template <int D, int U, int DEEP = 0>
__global__ void __launch_bounds__(kOrdMaxCta, 1) k_walk_ord(const __grid_constant__ TraverseArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int last_issued[4];  // latest chunk copied into each buffer
  __shared__ unsigned ord_failed;
  constexpr bool kGroups = U > 0;
  const int Q = kGroups ? a.groups : 1, TC = blockDim.x / Q, tid = threadIdx.x, lane = tid & 31;
  const int cols = TC >> 5, q = (tid >> 5) / cols, col = (tid >> 5) - q * cols;  // warp-uniform
  const int F2 = (a.F + 1) >> 1;
  if (a.p_pass || a.stream) pdl_wait();
  if (a.stream && *reinterpret_cast<volatile const unsigned*>(&a.stream->done)) return;
  const long long count = a.p_pass ? static_cast<long long>(a.state->survivors) : a.n;
  long long tile0;
  int rows_here;
  ord_tile(a, count, TC, &tile0, &rows_here);
  if (rows_here <= 0) return;  // whole CTA, before any copy is issued

  constexpr uint32_t kTree = DEEP ? ord_head_bytes(D) : ord_tree_bytes(D);
  const uint32_t chunk_bytes = static_cast<uint32_t>(a.chunk_trees) * kTree;
  const OrdSmem L = ord_smem(a.F, TC, kGroups ? Q : 0, a.nbuf, chunk_bytes);
  uint32_t* rowidx = reinterpret_cast<uint32_t*>(smem + L.rows);
  float* sums = reinterpret_cast<float*>(smem + L.sums);
  unsigned char* tbuf = smem + L.tbuf;
  // [0, nbuf) chunk buffers full, [4] the tile, [5] never completed
  // (self-test), [6, 6 + nbuf) chunk buffers empty, then the sums' barriers
  unsigned long long* bars = reinterpret_cast<unsigned long long*>(smem + L.bars);
  const int n_chunks = (a.n_trees + a.chunk_trees - 1) / a.chunk_trees;
  const int live_cols = (rows_here + 31) >> 5;  // columns that hold candidates
  const bool stall = static_cast<int>(blockIdx.x) == a.stall_cta;
  if (tid == 0) {
    for (int b = 0; b < 6; ++b) mbar_init(smem_u32(&bars[b]), 1);
    for (int b = 0; b < 4; ++b) {
      mbar_init(smem_u32(&bars[6 + b]), static_cast<uint32_t>(live_cols * Q));
      last_issued[b] = b < a.nbuf && b < n_chunks ? b : -1;
    }
    if (kGroups)
      for (int b = 0; b < cols * Q; ++b) mbar_init(smem_u32(&bars[10 + b]), 1);
    fence_mbar_init();
  }
  __syncthreads();
  auto issue = [&](int ch, int b) {
    const int first = ch * a.chunk_trees;
    const uint32_t bytes = static_cast<uint32_t>(min(a.chunk_trees, a.n_trees - first)) * kTree;
    const uint32_t bar = smem_u32(&bars[b]);
    mbar_expect_tx(bar, bytes);
    bulk_copy_g2s(smem_u32(tbuf + static_cast<size_t>(b) * chunk_bytes), a.table + static_cast<size_t>(first) * kTree,
                  bytes, bar);
  };
  if (tid == 0)
    for (int ch = 0; ch < a.nbuf && ch < n_chunks; ++ch) issue(ch, ch);  // tables are static
  if (!a.p_pass && !a.stream) pdl_wait();
  if (tid == 0) {
    const uint32_t tile_bytes = static_cast<uint32_t>(live_cols) * static_cast<uint32_t>(F2) * 128u;
    mbar_expect_tx(smem_u32(&bars[4]), tile_bytes);
    bulk_copy_g2s(smem_u32(smem), a.ord + (tile0 >> 5) * F2 * 32, tile_bytes, smem_u32(&bars[4]));
    // in shared memory, not a register: needed at the end only, read while the
    // tile is on its way (a register held over the walk cost the deep kernel 5 %)
    ord_failed = *reinterpret_cast<const volatile unsigned*>(&a.state->ord_failed);
  }
  if (a.p_pass && tid < rows_here) rowidx[tid] = a.rows[tile0 + tid];
  bool nan = false;
  if (col < live_cols) {
    const unsigned char* fl = a.nan_flags + ((tile0 >> 5) + col) * a.nan_groups;
    for (int g = lane; g < a.nan_groups; g += 32) nan |= fl[g] != 0;
  }
  nan = __any_sync(0xFFFFFFFFu, nan);
  float acc = 0.0f;
  bool timed_out = false;
  if (col < live_cols) {
    timed_out = !__all_sync(0xFFFFFFFFu, mbar_wait_bounded(smem_u32(&bars[4]), 0u));
    const OrdRow xw{smem + static_cast<uint32_t>(__shfl_sync(0xFFFFFFFFu, col, 0)) * static_cast<uint32_t>(F2) * 128u,
                    static_cast<uint32_t>(lane) * 4u};  // the shuffle makes the base warp-uniform to the compiler
    const uint32_t turn = smem_u32(&bars[10 + col * Q + q]);
    const uint32_t next_turn = smem_u32(&bars[10 + col * Q + (q + 1 == Q ? 0 : q + 1)]);
    float* sum = sums + col * 32 + lane;
    uint32_t turns = q == 0 ? 0u : 1u;  // waits done or due; group 0's first unit waits for nobody
    for (int ch = 0, b = 0, ph = 0; ch < n_chunks && !timed_out; ++ch) {
      const bool ok = stall && ch == 0 ? mbar_wait_bounded_ns(smem_u32(&bars[5]), 0u, a.stall_ns)
                                       : mbar_wait_bounded(smem_u32(&bars[b]), static_cast<uint32_t>(ph));
      if (!__all_sync(0xFFFFFFFFu, ok)) {
        timed_out = true;
        break;
      }
      const unsigned char* tb = tbuf + static_cast<uint32_t>(b) * chunk_bytes;
      const int nt = min(a.chunk_trees, a.n_trees - ch * a.chunk_trees);
      if constexpr (!kGroups) {
        acc = nan ? walk_ord_sum<D, true>(tb, nt, xw, acc) : walk_ord_sum<D, false>(tb, nt, xw, acc);
      } else {
        for (int t = q * U; t < nt; t += Q * U) {
          float leaf[U];
          const int here = min(U, nt - t);
          if constexpr (DEEP > 0) {
            const unsigned char* tt = tb + static_cast<uint32_t>(t) * kTree;
            const uint4* tail = reinterpret_cast<const uint4*>(a.tail);
            if (nan)
              walk_deep_unit<D, U, DEEP, true>(tt, here, xw, tail, a.max_depth, leaf);
            else
              walk_deep_unit<D, U, DEEP, false>(tt, here, xw, tail, a.max_depth, leaf);
          } else if (nan)
            walk_ord_unit<D, U, true>(tb + static_cast<uint32_t>(t) * kTree, here, xw, leaf);
          else
            walk_ord_unit<D, U, false>(tb + static_cast<uint32_t>(t) * kTree, here, xw, leaf);
          if ((ch | t) != 0) {  // the first unit starts from 0
            if (!__all_sync(0xFFFFFFFFu, mbar_wait_bounded(turn, (turns - 1u) & 1u))) {
              timed_out = true;
              break;
            }
            acc = *sum;
          }
#pragma unroll
          for (int g = 0; g < U; g += 4)
            if (g < here) {
              acc += leaf[g];
              acc += leaf[g + 1];
              acc += leaf[g + 2];
              acc += leaf[g + 3];
            }
          ++turns;
          *sum = acc;
          __syncwarp();
          if (lane == 0) mbar_arrive(next_turn);
        }
      }
      __syncwarp();
      if (lane == 0 && !timed_out && ch + a.nbuf < n_chunks && mbar_arrive_pending(smem_u32(&bars[6 + b])) == 1u) {
        mbar_try_wait(smem_u32(&bars[6 + b]), static_cast<uint32_t>(ph));  // complete: every warp is out
        last_issued[b] = ch + a.nbuf;
        issue(ch + a.nbuf, b);
      }
      if (++b == a.nbuf) {
        b = 0;
        ph ^= 1;
      }
    }
  }
  if (__syncthreads_or(timed_out || (tid == 0 && ord_failed != 0u))) {
    if (tid == 0) {
      // every copy in flight lands before the CTA's shared memory is released
      // (bounded waits), then the timeout is reported
      mbar_wait_bounded(smem_u32(&bars[4]), 0u);
      for (int b = 0; b < a.nbuf; ++b)
        if (last_issued[b] >= 0)
          mbar_wait_bounded(smem_u32(&bars[b]), static_cast<uint32_t>(last_issued[b] / a.nbuf) & 1u);
      atomicOr(a.err, kErrWaitTimeout);
    }
    acc = -INFINITY;  // the tile's bookkeeping still completes, none of it valid
    __syncthreads();
  } else if (kGroups && tid < TC) {
    acc = sums[tid];
  }
  pdl_trigger();
  finish_tile(a, rowidx, tile0, rows_here, count, acc, TC);
}

template <int U>
FullKernelPtr ord_kernel_for(int d) {
  switch (d) {
    case 1: return k_walk_ord<1, U>;
    case 2: return k_walk_ord<2, U>;
    case 3: return k_walk_ord<3, U>;
    case 4: return k_walk_ord<4, U>;
    case 5: return k_walk_ord<5, U>;
    case 6: return k_walk_ord<6, U>;
    case 7: return k_walk_ord<7, U>;
    case 8: return k_walk_ord<8, U>;
    case 9: return k_walk_ord<9, U>;
    case 10: return k_walk_ord<10, U>;
    default: return nullptr;
  }
}

// Trees of a unit: 16 where every group gets one of each full chunk, else
// fewer (the hand-over of the sums costs 16 / U as much).
int ord_unit(int chunk, int groups) {
  if (groups == 1) return 0;
  return chunk % (16 * groups) == 0 ? 16 : chunk % (8 * groups) == 0 ? 8 : chunk % (4 * groups) == 0 ? 4 : -1;
}
FullKernelPtr ord_kernel(int d, int unit) {
  return unit == 0 ? ord_kernel_for<0>(d) : unit == 4 ? ord_kernel_for<4>(d) : unit == 8 ? ord_kernel_for<8>(d)
                                                                                         : ord_kernel_for<16>(d);
}

}  // namespace

cudaError_t launch_ordinals(const OrdTable& t, OrdArgs a, long long n_max, int sms, cudaStream_t st) {
  if (n_max <= 0) return cudaSuccess;
  a.groups = t.groups;
  a.features = t.features;
  a.image = t.image;
  a.n_groups = t.n_groups;
  const size_t smem = std::max<size_t>(16, t.max_bytes);
  // one wave of CTAs, spread over the groups by their features
  int chunks = 0;
  for (int g = 0; g < t.n_groups; ++g) chunks += t.chunks[g];
  const bool wide = a.vec4 && n_max / 128 * chunks >= static_cast<long long>(sms) * (kOrdThreads / 32);
  const int rows = !a.vec4 ? 32 : wide ? 128 : 64;  // of a warp at a time
  const long long supers = (n_max + rows - 1) / rows;
  const int spare = std::max(0, sms - t.n_groups);  // one CTA of 32 warps an SM
  a.first_cta[0] = 0;
  for (int g = 0; g < t.n_groups; ++g) {
    const long long ctas = std::min(supers * t.chunks[g], 1 + static_cast<long long>(spare) * t.chunks[g] / chunks);
    a.first_cta[g + 1] = static_cast<unsigned short>(a.first_cta[g] + ctas);
  }
  auto pick = [&](auto narrow_k, auto wide_k) { return wide ? wide_k : narrow_k; };
  auto k = a.vec4 ? (t.round_half ? pick(k_ordinals<true, true, 4>, k_ordinals<true, true, 8>)
                                  : pick(k_ordinals<true, false, 4>, k_ordinals<true, false, 8>))
                  : (t.round_half ? k_ordinals<false, true, 8> : k_ordinals<false, false, 8>);
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(k), smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k, dim3(a.first_cta[t.n_groups]), dim3(kOrdThreads), smem, st, a);
}

// Shape of the ordinal walk over a deep model: a warp's tree waits on its tail
// loads, so the shape that puts the most warps on the busiest SM's candidates,
// then the largest tile (each tile streams every head).  Measured V passes of
// 4,194,304 x 256, 1,000 trees of depth 12: 33.3 ms with 256 candidates x 4
// groups, 34.5 with 192 x 4, 37.9 with 256 x 2, 38.3 with 128 x 2 twice an SM.
ScreenShape plan_ord_deep(int F, const OrdTable& t, long long n_eff, int sms, int optin) {
  ScreenShape best{};
  if (sms < 1) sms = 1;
  if (n_eff < 1) n_eff = 1;
  const uint32_t tb = ord_head_bytes(kOrdHead);
  double best_cost = 1e300;
  for (int tc = 32; tc <= 512; tc += 32) {
    for (int q : {1, 2, 3, 4, 6, 8, 12, 16}) {
      if (tc * q > kOrdMaxCta) continue;
      for (int ch = 128; ch >= 8; ch -= 8) {
        if (ch % (kOrdDeepUnit * q) != 0) continue;
        for (int nb : {2, 3}) {
          const size_t smem = ord_smem(F, tc, q, nb, static_cast<uint32_t>(ch) * tb).bytes;
          if (smem + kStaticSmem > static_cast<size_t>(optin)) continue;
          const long long tiles = (n_eff + tc - 1) / tc;
          const long long tiles_sm = (tiles + sms - 1) / sms;
          const long long fit =
              std::min<long long>({static_cast<long long>(kSmPerSm / (smem + kStaticSmem + kCtaReserve)),
                                   2048 / (tc * q), 65536 / (tc * q * 64)});
          if (fit < 1) continue;
          const long long res = std::min(fit, tiles_sm);
          const double warps = static_cast<double>(res) * tc * q / 32;
          const double tree = 45.0 + 400.0 / warps + tb / 128.0 / (tc / 32.0) * 2.0;
          const double chunks = std::ceil(static_cast<double>(t.n_trees) / ch);
          const double cost = static_cast<double>(tiles_sm) * (tc / 32.0 * t.n_trees * tree + chunks * 500.0 / (res * res) +
                                                               (res == 1 ? 6000.0 : 2000.0 / res)) +
                              40.0 * nb;
          if (cost < best_cost) {
            best_cost = cost;
            best.threads = tc;
            best.smem = smem;
            best.chunk_trees = ch;
            best.nbuf = nb;
            best.group = kOrdDeepFlight;
            best.lanes = q;
            best.resident = static_cast<int>(res);
            best.p_grid = sms * static_cast<int>(res);
          }
        }
      }
    }
  }
  if (best.threads) best = cap_residency(best, optin);
  return best;
}

// Candidates per CTA, tree groups, trees per chunk and buffers of the ordinal
// walk: the shape with the least estimated cycles of the busiest SM.  Fitted
// to sweeps on GB300 (65,536 x 64 and 1,048,576 x 128, depth 8; 16,700,000 x
// 96, depth 10): a warp visit costs 2.6 cycles of the shared-memory pipe, more
// with few warps, and its share of the chunk's copy into shared memory.  Tree
// groups pay where a tile's candidates leave an SM few warps (65,536 x 64, P
// pass of 7 warps' candidates: 58.0 / 50.5 / 47.5 us with 1 / 2 / 4 groups)
// and cost 5 % or more where they do not (1,048,576 x 128, V pass of 16 warps:
// 1.53 ms with 1 group, 1.59 with 2).  A chunk's hand-off stalls its warps
// together, and a tile's start about 6,000 cycles: another resident CTA hides
// both.
ScreenShape plan_ord(int F, const OrdTable& t, int depth, long long n_eff, int sms, int optin) {
  if (t.rounds > 0) return plan_ord_deep(F, t, n_eff, sms, optin);
  ScreenShape best{};
  if (sms < 1) sms = 1;
  if (n_eff < 1) n_eff = 1;
  const uint32_t tb = ord_tree_bytes(depth);
  const int trees8 = (t.n_trees + 7) / 8 * 8;
  double best_cost = 1e300;
  for (int tc = 32; tc <= 768; tc += 32) {
    for (int q : {1, 2, 4, 8, 16}) {
      if (tc * q > kOrdMaxCta) continue;
      for (int ch = 128; ch >= 8; ch -= 8) {
        if (ch > std::max(trees8, 4 * q) && ch != 8) continue;
        const int unit = ord_unit(ch, q);
        if (unit < 0) continue;
        for (int nb : {2, 3}) {
          const size_t smem = ord_smem(F, tc, q > 1 ? q : 0, nb, static_cast<uint32_t>(ch) * tb).bytes;
          if (smem + kStaticSmem > static_cast<size_t>(optin)) continue;
          const long long tiles = (n_eff + tc - 1) / tc;
          const long long tiles_sm = (tiles + sms - 1) / sms;
          const long long fit =
              std::min<long long>({static_cast<long long>(kSmPerSm / (smem + kStaticSmem + kCtaReserve)),
                                   2048 / (tc * q), 65536 / (tc * q * 64)});
          if (fit < 1) continue;
          const long long res = std::min(fit, tiles_sm);
          const double warps = static_cast<double>(res) * tc * q / 32;
          const double visit = 2.6 + 30.0 / (warps * warps) + tb / 128.0 / (tc / 32.0) / depth +
                               (unit ? 0.15 + 1.6 / unit : 0.0);
          const double chunks = std::ceil(static_cast<double>(t.n_trees) / ch);
          const double cost = static_cast<double>(tiles_sm) *
                                  (tc / 32.0 * t.n_trees * depth * visit + chunks * (400.0 + 4000.0 / warps) / (res * res) +
                                   (res == 1 ? 6000.0 : 2000.0 / res)) +
                              40.0 * nb;
          if (cost < best_cost) {
            best_cost = cost;
            best.threads = tc;
            best.smem = smem;
            best.chunk_trees = ch;
            best.nbuf = nb;
            best.group = 8;
            best.lanes = q;
            best.resident = static_cast<int>(res);
            best.p_grid = sms * static_cast<int>(res);
          }
        }
      }
    }
  }
  if (best.threads) best = cap_residency(best, optin);
  return best;
}

cudaError_t launch_walk_ord(int depth, const TraverseArgs& args, const ScreenShape& shape, long long n_tiles,
                            cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  TraverseArgs a = args;
  a.groups = shape.lanes;
  long long ctas = n_tiles;
  if (args.p_pass && shape.p_grid > 0) {
    a.p_wave = shape.p_grid;
    ctas = (n_tiles + shape.p_grid - 1) / shape.p_grid * shape.p_grid;
  }
  FullKernelPtr k = depth > kMaxFullDepth ? k_walk_ord<kOrdHead, kOrdDeepUnit, kOrdDeepFlight>
                                          : ord_kernel(depth, ord_unit(shape.chunk_trees, shape.lanes));
  if (k == nullptr) return cudaErrorInvalidValue;
  cudaError_t e =
      allow_smem(reinterpret_cast<const void*>(k), shape.smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k, dim3(static_cast<unsigned>(ctas)), dim3(shape.threads * shape.lanes), shape.smem, st, a);
}

}  // namespace mlt
