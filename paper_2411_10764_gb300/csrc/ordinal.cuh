// Ordinal form of a model: every threshold replaced by its place among the
// model's distinct thresholds of that feature, and every candidate feature by
// the number of those thresholds it is not below.
//
// x >= t_i  <=>  #{distinct t <= x} > i, so a comparison of two small
// integers decides exactly what the fp32 comparison decides: the walk takes
// the same path and adds the same fp32 leaves in the same order.  A node then
// fits one 4-byte word (fp32 tables: 4-byte threshold + 2-byte meta, two
// loads) and a feature fits 2 bytes, so a visit costs two shared-memory loads
// instead of three and an SM holds twice the candidates.
//
// Feature ordinals (k_ordinals writes them, the walk reads them): blocks of
// 32 candidates, each block [ceil(F/2)][32] 4-byte words; word (q, lane) holds
// features 2q (low half) and 2q + 1 (high half) of candidate `lane`.  A warp
// gathering 32 different features of its 32 candidates hits 32 different
// banks, and a tile of blocks is one contiguous copy.  A missing value is
// kOrdNan.
//
// Node word: ordinal i (15 bits) << 16 | byte offset of the feature in a block
// ((f >> 1) * 128 + (f & 1) * 2) | NaN-goes-left flag (bit 0; bit 15 in a deep
// model).  With x the feature's ordinal, the sign of word - (x << 16) is the
// branch: set iff x > i (the low 16 bits of the word never reach the sign).
// kOrdNan << 16 is the sign bit, so a missing x goes right; the flag clears it
// to 0, which goes left.
//
// Tree: 2^(D+1) words, node j (1-based heap index) at word j, the leaf of
// child index c (2^D <= c) as an fp32 at word c; word 0 is unused.  Trees are
// padded with zero trees (leaves +0) to a multiple of kOrdTreePad.
//
// Deep models (depth > kMaxFullDepth): the first H = kOrdHead levels of a tree
// are such a heap, streamed through shared memory; then come 2^H exits of 8
// bytes: a leaf {fp32, kOrdExitLeaf}, or the level-H split {word, index of the
// block of its left child; the right child's follows}.  The rest of a tree
// stays in global memory as 32-byte blocks of three levels (one sector, one
// load): word 0 = index of the first of 8 child blocks | leaf flags of nodes
// 1 .. 7 << kOrdBlockBits, words 1 .. 7 = a 3-level heap of node words or fp32
// leaves.  A path that leaves the head takes one load per three levels, where
// 8-byte records took one per level.
//
// Search of a feature's ordinal: its distinct thresholds in ascending order,
// padded with NaN (never <= x), and a lookup table of buckets: lut[b] =
// thresholds in the buckets below b (2 bytes).  The bucket of x is taken from
// the bits of the positive float max(x, lo) + (c - lo), which never decrease
// with x: above c they follow x's logarithm, below it x itself, and c is
// chosen per feature to spread its thresholds.  A bucket holds few
// thresholds, so two to four compares finish what a binary search over all of
// them takes ten or more for; a compare past the bucket's end meets a larger
// threshold or the padding and changes nothing.
#pragma once

#include <vector>

#include "mlt.h"
#include "mlt_internal.cuh"

namespace mlt {

__host__ __device__ constexpr uint32_t ord_tree_bytes(int D) { return 8u << D; }
__host__ __device__ constexpr uint32_t ord_head_bytes(int H) { return 12u << H; }
__host__ __device__ constexpr uint32_t ord_offset(uint32_t f) { return (f >> 1) * 128u + (f & 1u) * 2u; }
constexpr int kOrdDeepMaxF = 512;  // offsets below bit 15

struct OrdArgs {
  const float* feats;      // [n][F]
  int F;
  int vec4;                // rows 16-byte aligned, F % 4 == 0
  long long n;             // rows (when count is null)
  const uint32_t* rows;    // P pass: row of candidate i (null: i)
  const unsigned* count;   // P pass: candidates (device)
  const StreamState* stream;
  const OrdGroup* groups;
  const OrdFeature* features;
  const unsigned char* image;
  uint32_t* out;           // [blocks][ceil(F/2)][32]
  unsigned char* nan_flags;  // [blocks][ceil(F/8)]: a missing value among 8 features
  unsigned* err;
  unsigned* failed;        // SelectState::ord_failed
  unsigned long long stall_ns;  // self-test: CTA 0 waits this long on a barrier nothing completes (0: no)
  int n_groups;
  unsigned short first_cta[kOrdMaxGroups + 1];  // CTAs [first_cta[g], first_cta[g + 1]) take group g
};

// ordinal_pack.cu: the ordinal form of a validated ensemble, described by t
// (offsets into `out`; multiples of 128).  round_half: thresholds, leaves and
// features rounded to binary16.  False (and `out` empty) when a feature has too many distinct thresholds (or one of -inf).
bool pack_ordinal(const mlt_node* nodes, int n_trees, int depth, int F, bool round_half,
                  std::vector<unsigned char>& out, OrdTable& t);
// ordinal.cu
cudaError_t launch_ordinals(const OrdTable& t, OrdArgs a, long long n_max, int sms, cudaStream_t st);
ScreenShape plan_ord(int F, const OrdTable& t, int depth, long long n_eff, int sms, int optin);
cudaError_t launch_walk_ord(int depth, const TraverseArgs& args, const ScreenShape& shape, long long n_tiles,
                            cudaStream_t st);

}  // namespace mlt
