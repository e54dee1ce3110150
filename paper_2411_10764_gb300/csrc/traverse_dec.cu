// Tree-walk kernels that build each candidate's features on chip from its
// index (mixed-radix knob decode + feature program) instead of reading a
// stored feature matrix, and the materialising decoder of mlt_decode_knobs.
// ML^2Tuner Sec. 2: the explorer enumerates the search space of
// configurations; Appendix A.2: the knobs are tiling sizes and virtual-thread
// counts; Table 5: derived (hidden) features.
#include <algorithm>

#include "mlt.h"
#include "walk.cuh"

namespace mlt {
namespace {

using namespace walk;

using CompactDecKernel = void (*)(TraverseArgs, DecodeParams);

CompactDecKernel compact_dec_kernel(int group, int lanes) {
  if (group == 8) {
    switch (lanes) {
      case 1: return k_traverse_compact_dec<8, 1>;
      case 2: return k_traverse_compact_dec<8, 2>;
      case 4: return k_traverse_compact_dec<8, 4>;
      case 8: return k_traverse_compact_dec<8, 8>;
    }
  } else if (group == 4) {
    switch (lanes) {
      case 1: return k_traverse_compact_dec<4, 1>;
      case 2: return k_traverse_compact_dec<4, 2>;
      case 4: return k_traverse_compact_dec<4, 4>;
      case 8: return k_traverse_compact_dec<4, 8>;
    }
  }
  return nullptr;
}

// Knob values and features of a tile of candidates (a thread each) in shared
// memory, one column of `stride` floats per slot (knobs first), then written
// out as rows.  The program sits beside them as 16-byte records {opcode,
// operand columns, constant}: one broadcast read an operation, the next one's
// in flight meanwhile, where fields read from the parameter bank by a running
// index and knob values in local memory took longer.  The stride is 1 modulo
// 32: the 32 lanes of a column access hit 32 banks, and so do 8 groups of 4
// columns x 4 candidates, the shape in which a warp stores four 128-byte row
// pieces.  Bound: issue and branch latency of about 45 instructions an
// operation at the warps that shared memory allows; several candidates a
// thread were slower (fewer warps: 1.16 ms with 2, 1.45 with 4, 0.95 with 1 for
// 4,194,304 candidates x 96 features; 1.29 before).
__host__ __device__ constexpr size_t program_offset(int slots, int stride) {
  return (static_cast<size_t>(slots) * stride * 4 + 15) / 16 * 16;
}
__global__ void __launch_bounds__(256)
    k_decode_rows(const __grid_constant__ DecodeParams d, long long n, int stride, int vec4, uint8_t* out_knobs,
                  float* out_feats, const StreamState* ss) {
  extern __shared__ __align__(128) unsigned char smem[];
  float* xs = reinterpret_cast<float*>(smem);
  const int T = blockDim.x, tid = threadIdx.x, F = d.F, nk = d.n_knobs;
  const long long tile0 = static_cast<long long>(blockIdx.x) * T;
  const int rows_here = static_cast<int>(min(static_cast<long long>(T), n - tile0));
  int4* prog = reinterpret_cast<int4*>(smem + program_offset(F + nk, stride));
  if (out_feats != nullptr)
    for (int f = tid; f < F; f += T) prog[f] = make_int4(d.op[f], d.a[f], d.b[f], __float_as_int(d.c[f]));
  pdl_wait();
  pdl_trigger();
  if (ss && *reinterpret_cast<volatile const unsigned*>(&ss->done)) return;
  if (tid < rows_here) {
    const long long idx = d.index_list ? d.index_list[tile0 + tid] : d.first_index + tile0 + tid;
    uint8_t* kn = out_knobs != nullptr ? out_knobs + (tile0 + tid) * nk : nullptr;
    const bool pack = kn != nullptr && nk == 8 && (reinterpret_cast<uintptr_t>(kn) & 7u) == 0;  // one 8-byte store
    unsigned long long packed = 0;
    unsigned long long rem = static_cast<unsigned long long>(idx);
    for (int j = 0; j < nk; ++j) {
      const uint32_t radix = static_cast<uint32_t>(d.radix[j]);
      uint32_t digit;
      if ((rem >> 32) == 0) {  // a 64-bit division is a long subroutine
        const uint32_t q = static_cast<uint32_t>(rem) / radix;
        digit = static_cast<uint32_t>(rem) - q * radix;
        rem = q;
      } else {
        const unsigned long long q = rem / radix;
        digit = static_cast<uint32_t>(rem - q * radix);
        rem = q;
      }
      xs[j * stride + tid] = d.opts[d.opt_off[j] + static_cast<int>(digit)];
      if (pack)
        packed |= static_cast<unsigned long long>(digit) << (8 * j);
      else if (kn)
        kn[j] = static_cast<uint8_t>(digit);
    }
    if (pack) *reinterpret_cast<unsigned long long*>(kn) = packed;
  } else {
    for (int j = 0; j < nk; ++j) xs[j * stride + tid] = 1.0f;
  }
  if (out_feats == nullptr) return;
  __syncthreads();
  const float* mine = xs + tid;
  float* col = xs + nk * stride + tid;
  int4 next = prog[0];
  for (int f = 0; f < F; ++f, col += stride) {
    const int4 o = next;
    next = prog[min(f + 1, F - 1)];
    const float A = o.y < 0 ? __int_as_float(o.w) : mine[o.y * stride];
    const float B = o.z < 0 ? __int_as_float(o.w) : mine[o.z * stride];
    float x;
    if (o.x >= MLT_OP_DIV && o.x <= MLT_OP_REM) {  // one copy of the division
      const float q = __fdiv_rn(A, B);
      x = o.x == MLT_OP_DIV       ? q
          : o.x == MLT_OP_CEILDIV ? ceilf(q)
                                  : __fsub_rn(A, __fmul_rn(B, floorf(q)));
    } else {
      switch (o.x) {
        case MLT_OP_COPY: x = A; break;
        case MLT_OP_ILOG2: x = ilog2_exact(A); break;
        case MLT_OP_ADD: x = __fadd_rn(A, B); break;
        case MLT_OP_SUB: x = __fsub_rn(A, B); break;
        case MLT_OP_MUL: x = __fmul_rn(A, B); break;
        case MLT_OP_MIN: x = (B < A) ? B : A; break;
        case MLT_OP_MAX: x = (B > A) ? B : A; break;
        case MLT_OP_GT: x = (A > B) ? 1.0f : 0.0f; break;
        default: x = (A == B) ? 1.0f : 0.0f; break;
      }
    }
    *col = x;
  }
  __syncthreads();
  const float* feats = xs + nk * stride;
  float* dst = out_feats + tile0 * F;
  const int lane = tid & 31, warp = tid >> 5, warps = T >> 5;
  if (vec4) {
    const int F4 = F >> 2, q0 = lane >> 2;
    for (int r0 = warp * 4; r0 < rows_here; r0 += warps * 4) {
      const int row = r0 + (lane & 3);
      if (row >= rows_here) continue;
      for (int q = q0; q < F4; q += 8) {
        const float* src = feats + 4 * q * stride + row;
        *reinterpret_cast<float4*>(dst + static_cast<long long>(row) * F + 4 * q) =
            make_float4(src[0], src[stride], src[2 * stride], src[3 * stride]);
      }
    }
  } else {
    // element v = r * F + f of the tile's rows, v = tid, tid + T, ...: (r, f)
    // advance by (T / F, T % F) with a carry, no division per step
    const int dr = T / F, df = T - dr * F;
    int r = tid / F, f = tid - r * F;
    for (int v = tid; v < rows_here * F; v += T) {
      dst[v] = feats[f * stride + r];
      r += dr;
      f += df;
      if (f >= F) {
        f -= F;
        ++r;
      }
    }
  }
}

}  // namespace

FullDecKernelPtr full_dec_kernel_q1(int depth, int group) { return full_dec_kernel_q<1>(depth, group); }

FullDecKernelPtr full_dec_kernel(int depth, int group, int q) {
  switch (q) {
    case 0: return full_dec_kernel_sf(depth, group);
    case 1: return full_dec_kernel_q1(depth, group);
    case 2: return full_dec_kernel_q2(depth, group);
    case 4: return full_dec_kernel_q4(depth, group);
    default: return nullptr;
  }
}

cudaError_t launch_traverse_dec(const DeviceModel& m, const TraverseArgs& args, const DecodeParams& dec,
                                const ScreenShape& shape, long long n_tiles, cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  // full-table P pass: whole waves of CTAs, the survivors split evenly over
  // them on the device (CTAs without rows exit at once)
  TraverseArgs a = args;
  long long ctas = n_tiles;
  if (m.kind == kTableHalf) return cudaErrorInvalidValue;  // half tables need stored features
  if (args.p_pass && (m.kind == kTableFull || m.kind == kTableSplit) && shape.p_grid > 0) {
    a.p_wave = shape.p_grid;
    ctas = (n_tiles + shape.p_grid - 1) / shape.p_grid * shape.p_grid;
  }
  const dim3 grid(static_cast<unsigned>(ctas));
  if (m.kind == kTableFull || m.kind == kTableSplit) {
    const int q = shape.sync_free ? 0 : shape.lanes;
    FullDecKernelPtr k = m.kind == kTableSplit ? split_dec_kernel(m.head_levels, shape.group, q)
                                               : full_dec_kernel(m.depth, shape.group, q);
    if (k == nullptr) return cudaErrorInvalidValue;
    cudaError_t e = allow_smem(reinterpret_cast<const void*>(k), shape.smem);
    if (e != cudaSuccess) return e;
    e = launch_pdl(k, grid, dim3(shape.threads * shape.lanes), shape.smem, st, a, dec);
    if (e != cudaSuccess) return e;
  } else {
    CompactDecKernel k = compact_dec_kernel(shape.group, shape.lanes);
    if (k == nullptr) return cudaErrorInvalidValue;
    cudaError_t e = allow_smem(reinterpret_cast<const void*>(k), shape.smem);
    if (e != cudaSuccess) return e;
    e = launch_pdl(k, grid, dim3(shape.threads * shape.lanes), shape.smem, st, a, dec);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t launch_decode_rows(const DecodeParams& dec, long long n, uint8_t* out_knobs, float* out_feats,
                               cudaStream_t st, const StreamState* ss) {
  if (n <= 0) return cudaSuccess;
  // the tile that keeps the most warps on an SM; no wider than the batch needs
  // to reach every SM
  int sms = 1, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int slots = dec.F + dec.n_knobs;
  auto smem_of = [&](int tile) { return program_offset(slots, tile + 1) + static_cast<size_t>(dec.F) * 16; };
  int tile = 32, best = 0;
  for (int t : {256, 192, 128, 96, 64, 32}) {
    const int held = static_cast<int>(std::min<size_t>(228 * 1024 / (smem_of(t) + 1024), 2048 / t)) * t;
    if (smem_of(t) > 224 * 1024 || (t > 32 && static_cast<long long>(t) * sms > n)) continue;
    if (held > best) {
      best = held;
      tile = t;
    }
  }
  const size_t smem = smem_of(tile);
  auto k = k_decode_rows;
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(k), smem);
  if (e != cudaSuccess) return e;
  const int vec4 = (dec.F & 3) == 0 && (reinterpret_cast<uintptr_t>(out_feats) & 15u) == 0 ? 1 : 0;
  return launch_pdl(k, dim3(static_cast<unsigned>((n + tile - 1) / tile)), dim3(tile), smem, st, dec, n, tile + 1,
                    vec4, out_knobs, out_feats, ss);
}

}  // namespace mlt
