// fp32 path of grass_project_grad: Gc[j,c] = rho_j * sum_t dY[t,idx_j] X[t,c]
// (Section 3.1 of the GRASS paper) with fp32 FMA on the CUDA cores.
//
// Used when the caller asks for "fp32 everywhere": tensor-core TF32 would drop
// 13 mantissa bits of every product, so this path keeps full fp32 products.
//
// Bound by the FMA pipes (74.4 TFLOP/s).  A CTA owns a (16 TM) x (16 TM) output tile, a thread TM x TM
// of it, in packed pairs of columns (fma.rn.f32x2: half the issue slots, the same two roundings).
// Tokens come 16 at a time through a three-stage cp.async ring: 16 bytes a copy for X and a dense
// dY where their alignment allows it, else 4 bytes, which is also how the selected columns of dY are
// picked; out-of-range elements are zero-filled by the copy.  TM = 8 reads 16 floats of shared
// memory per 64 FMAs and thread; TM = 4 makes four times the tiles for outputs too small to fill
// the GPU otherwise.  Small problems are split over the tokens (gridDim.z slices, partials summed in
// slice order by the kernel that follows); results are bit-reproducible.
// 1024 x 1024, T = 2048: 292 us with 64 x 64 tiles and one synchronous stage, 104 now (41 TFLOP/s).
#pragma once

#include "common.cuh"

namespace grass {

constexpr int kSimtBT = 16, kSimtThreads = 256, kSimtStages = 3;
__host__ __device__ constexpr int simt_tile(int TM) { return 16 * TM; }
__host__ __device__ constexpr int simt_smem_bytes(int TM) {
  return kSimtStages * 2 * kSimtBT * simt_tile(TM) * static_cast<int>(sizeof(float));
}

// `bytes` of 4 (or 16) from global memory, zeros for the rest
__device__ __forceinline__ void cp_async_4(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_16(float* dst, const float* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void fma_pair(float2& d, float2 a, float2 b) {
  asm("{\n\t.reg .b64 x, y, z;\n\t"
      "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%0, %1};\n\t"
      "fma.rn.f32x2 z, x, y, z;\n\t"
      "mov.b64 {%0, %1}, z;\n\t}"
      : "+f"(d.x), "+f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
}

// avec / xvec: the dense dY / X may be copied 16 bytes at a time; ovec: so may the output.
template <int TM>
__global__ void __launch_bounds__(kSimtThreads, TM == 8 ? 2 : 4)
project_simt_kernel(const float* dY, int64_t lddy, const float* X, int64_t ldx,
                    int64_t Ttok, int64_t m, int64_t n, const int32_t* idx,
                    const float* rho, int r, float* Gc, int64_t ldgc,
                    int64_t tokens_per_split, int64_t split_stride, bool avec, bool xvec, bool ovec,
                    int* status) {
  constexpr int B = simt_tile(TM), BT = kSimtBT, Q = TM / 4;
  constexpr int ROWS = kSimtThreads / B;             // tokens covered by one 4-byte copy a thread
  constexpr int ROWS4 = kSimtThreads / (B / 4);      // and by one 16-byte copy
  extern __shared__ __align__(16) float s_simt[];    // [stage][dY | X][token][column]
  const int tid = threadIdx.x;
  const int j0 = blockIdx.y * B;
  const int64_t c0 = static_cast<int64_t>(blockIdx.x) * B;
  grid_dep_wait();
  // the selected row whose column this thread copies
  int row = -1;
  if (!avec) {
    const int j = j0 + tid % B;
    if (j < r) {
      row = idx != nullptr ? idx[j] : j;
      if (row < 0 || row >= m) {
        if (tid < B) record_status(status, GRASS_ERR_INVALID_ARG, row);
        row = -1;
      }
    }
  }
  const int64_t t_lo = static_cast<int64_t>(blockIdx.z) * tokens_per_split;
  const int64_t t_hi = t_lo + tokens_per_split < Ttok ? t_lo + tokens_per_split : Ttok;
  const int steps = static_cast<int>((t_hi - t_lo + BT - 1) / BT);

  auto copy_stage = [&](int it) {
    float* sA = s_simt + (it % kSimtStages) * (2 * BT * B);
    float* sX = sA + BT * B;
    const int64_t t0 = t_lo + static_cast<int64_t>(it) * BT;
    if (avec) {
      const int col = (tid % (B / 4)) * 4;
      const int left = r - (j0 + col);
      const int bytes = left >= 4 ? 16 : left > 0 ? 4 * left : 0;
#pragma unroll
      for (int k = 0; k < BT; k += ROWS4) {
        const int tt = k + tid / (B / 4);
        const bool on = bytes > 0 && t0 + tt < t_hi;
        cp_async_16(sA + tt * B + col, on ? dY + (t0 + tt) * lddy + j0 + col : dY, on ? bytes : 0);
      }
    } else {
#pragma unroll
      for (int k = 0; k < BT; k += ROWS) {
        const int tt = k + tid / B;
        const bool on = row >= 0 && t0 + tt < t_hi;
        cp_async_4(sA + tt * B + tid % B, on ? dY + (t0 + tt) * lddy + row : dY, on ? 4 : 0);
      }
    }
    if (xvec) {
      const int col = (tid % (B / 4)) * 4;
      const int64_t left = n - (c0 + col);
      const int bytes = left >= 4 ? 16 : left > 0 ? 4 * static_cast<int>(left) : 0;
#pragma unroll
      for (int k = 0; k < BT; k += ROWS4) {
        const int tt = k + tid / (B / 4);
        const bool on = bytes > 0 && t0 + tt < t_hi;
        cp_async_16(sX + tt * B + col, on ? X + (t0 + tt) * ldx + c0 + col : X, on ? bytes : 0);
      }
    } else {
      const int64_t c = c0 + tid % B;
#pragma unroll
      for (int k = 0; k < BT; k += ROWS) {
        const int tt = k + tid / B;
        const bool on = c < n && t0 + tt < t_hi;
        cp_async_4(sX + tt * B + tid % B, on ? X + (t0 + tt) * ldx + c : X, on ? 4 : 0);
      }
    }
  };

  // thread (ty, tx) holds rows 4 ty .. + 3 (and 64 further on) by columns 4 tx .. + 3 (and 64 further on)
  const int ty = tid / 16, tx = tid % 16;
  float2 acc[TM][TM / 2];
#pragma unroll
  for (int a = 0; a < TM; ++a)
#pragma unroll
    for (int b = 0; b < TM / 2; ++b) acc[a][b] = make_float2(0.f, 0.f);

#pragma unroll
  for (int it = 0; it < kSimtStages - 1; ++it) {
    if (it < steps) copy_stage(it);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int it = 0; it < steps; ++it) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kSimtStages - 2) : "memory");
    __syncthreads();                 // stage `it` has landed; stage it - 1 has been read by all
    if (it + kSimtStages - 1 < steps) copy_stage(it + kSimtStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* sA = s_simt + (it % kSimtStages) * (2 * BT * B) + 4 * ty;
    const float* sX = s_simt + (it % kSimtStages) * (2 * BT * B) + BT * B + 4 * tx;
#pragma unroll
    for (int tt = 0; tt < BT; ++tt) {
      float a[TM];
      float2 b[TM / 2];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const float4 av = *reinterpret_cast<const float4*>(sA + tt * B + 64 * q);
        const float4 xv = *reinterpret_cast<const float4*>(sX + tt * B + 64 * q);
        a[4 * q] = av.x; a[4 * q + 1] = av.y; a[4 * q + 2] = av.z; a[4 * q + 3] = av.w;
        b[2 * q] = make_float2(xv.x, xv.y);
        b[2 * q + 1] = make_float2(xv.z, xv.w);
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int k = 0; k < TM / 2; ++k) fma_pair(acc[i][k], make_float2(a[i], a[i]), b[k]);
    }
  }
  grid_dep_launch();
  // with more than one slice the output is that slice's partial sum (rho applied later)
  Gc += static_cast<int64_t>(blockIdx.z) * split_stride;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int j = j0 + 4 * ty + (i / 4) * 64 + i % 4;
    if (j >= r) continue;
    const float s = (rho != nullptr && gridDim.z == 1) ? rho[j] : 1.f;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int64_t c = c0 + 4 * tx + 64 * q;
      const float4 v = make_float4(s * acc[i][2 * q].x, s * acc[i][2 * q].y, s * acc[i][2 * q + 1].x,
                                   s * acc[i][2 * q + 1].y);
      float* out = Gc + static_cast<int64_t>(j) * ldgc + c;
      if (ovec && c + 3 < n) {
        *reinterpret_cast<float4*>(out) = v;
      } else {
        if (c < n) out[0] = v.x;
        if (c + 1 < n) out[1] = v.y;
        if (c + 2 < n) out[2] = v.z;
        if (c + 3 < n) out[3] = v.w;
      }
    }
  }
}

}  // namespace grass
