// The network v_theta (2 -> 64 -> 64 -> 1, SiLU; Eq. 11, 37-39) on the
// fifth-generation tensor cores: v and grad v at many points, tile by tile.
//
// A CTA of four warpgroups (512 threads), one per SM; each warpgroup takes its
// own tiles of 128 points, thread t of the group owning point t of the tile
// (TMEM lane t), with its own operand buffer, mbarrier and TMEM columns, and
// synchronises on its own named barrier, so the groups' MMAs and SIMT work
// overlap.  Per tile:
//   layer 1 (FP32 SIMT)    a1 = W1 x + b1, h1 = SiLU(a1); SiLU'(a1) into TMEM
//   forward (tcgen05)      D = h1 W2^T              [128 x 64], TMEM
//   output  (FP32 SIMT)    a2 = D + b2, v = w3 . SiLU(a2) + b3,
//                          g2 = w3 * SiLU'(a2) = dv / da2
//   backward (tcgen05)     D = g2 W2                [128 x 64], TMEM
//   input gradient (SIMT)  grad v = W1^T (D * SiLU'(a1))
// h1 and g2 are the M x K operand (K-major, 128-byte swizzle), W2 and W2^T
// the N x K operands, staged once per CTA.  Every product is the 3xTF32 split
// (tc_sm103.cuh), so v and grad v carry FP32 rounding only.
//
// What bounds it: the SiLUs (two special-function operations and about ten
// instructions per unit, 128 units per point), which only enough warps keep
// flowing through a tile's chain of products.  So the operand goes through one
// 32-unit half buffer (hi and lo: 32 KB per group instead of 64): the half's
// MMA runs while the other half's units are computed in registers; SiLU'(a1)
// waits in TMEM instead of 64 registers; the units run in packed FP32 pairs.
// That makes 16 warps per SM instead of 8, at two thirds of the instructions
// (55 per point and warp lane instead of 82).  One GB300, 1.59e6 points: kernel
// 330 -> 190 us, the call with its kept scratch 525 -> 245 us; 1,000 points 211
// -> 48 us.  3xTF32 at N = 64 keeps the tensor pipe busy for about 115 us of it.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "pdds.h"
#include "pdds_internal.h"
#include "device_scratch.h"
#include "tc_sm103.cuh"

namespace pdds {
namespace {

constexpr int kH = 64;    // hidden width
constexpr int kTP = 128;  // points per tile = MMA M
constexpr int kOffW2 = 192, kOffB1 = 128, kOffB2 = 4288, kOffW3 = 4352, kOffB3 = 4416;

constexpr int kGroups = 4;   // warpgroups per CTA
constexpr int kHalf = kH / 2;  // units per operand buffer
constexpr unsigned kColsGroup = 128;  // TMEM per group: D (64 columns), SiLU'(a1) (64)

struct alignas(1024) EvalTcSmem {
  float B1[2][kH * kH];              // W2 as N = out x K = in, hi and lo parts
  float B2[2][kH * kH];              // W2^T as N = in x K = out
  float A[kGroups][2][kTP * kHalf];  // per group: half of h1 or g2 (M = point x K = unit)
  float w1x[kH], w1y[kH], b1[kH], b2[kH], w3[kH];
  float b3;
  unsigned long long mbar[kGroups];
  unsigned tmem;
};
constexpr size_t kEvalTcSmemBytes = sizeof(EvalTcSmem) + 1024;  // + alignment slack

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }

// 1 / (1 + e^-a) from the hardware exponential and reciprocal (a few ulp; 0
// when e^-a overflows; where e^-a would be denormal the sum is 1 either way)
__device__ __forceinline__ float2 logistic2(float2 a) {
  const float2 t = mul2(a, f2(-1.4426950408889634f, -1.4426950408889634f));
  float ex, ey, rx, ry;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ex) : "f"(t.x));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(ey) : "f"(t.y));
  const float2 y = add2(f2(ex, ey), f2(1.0f, 1.0f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rx) : "f"(y.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(ry) : "f"(y.y));
  return f2(rx, ry);
}
// SiLU'(a) = sg (1 + a (1 - sg)) from the logistic sg
__device__ __forceinline__ float2 dsilu2(float2 a, float2 sg) {
  const float2 m = add2(f2(1.0f, 1.0f), f2(-sg.x, -sg.y));
  return mul2(sg, fma2(a, m, f2(1.0f, 1.0f)));
}
__device__ __forceinline__ void group_sync(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(kTP) : "memory");
}

// Units 4c .. 4c + 3 of this point's half into the operand buffers, split.
__device__ __forceinline__ void put_split(float* hi_base, float* lo_base, int off_bytes, float2 v,
                                          float2 w) {
  const float4 h = make_float4(tc::tf32_hi(v.x), tc::tf32_hi(v.y), tc::tf32_hi(w.x), tc::tf32_hi(w.y));
  const float2 l0 = add2(v, f2(-h.x, -h.y)), l1 = add2(w, f2(-h.z, -h.w));
  *reinterpret_cast<float4*>(reinterpret_cast<char*>(hi_base) + off_bytes) = h;
  *reinterpret_cast<float4*>(reinterpret_cast<char*>(lo_base) + off_bytes) =
      make_float4(l0.x, l0.y, l1.x, l1.y);
}

// D (TMEM, 64 columns at d) [+]= A B^T over the 32 units of half `hf` with the
// 3xTF32 split: 3 x 4 K-steps.
__device__ __forceinline__ void mma_half(unsigned d, unsigned a_hi, unsigned a_lo, unsigned b_hi,
                                         unsigned b_lo, int hf) {
  constexpr uint32_t idesc = tc::idesc_tf32(kTP, kH);
#pragma unroll
  for (int pr = 0; pr < 3; ++pr) {  // hi hi, hi lo, lo hi
    const unsigned a = pr == 2 ? a_lo : a_hi, b = (pr == 1 ? b_lo : b_hi) + hf * kH * 128;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
      tc::mma_tf32(d, tc::sdesc_k128(a + kk * 32), tc::sdesc_k128(b + kk * 32), idesc,
                   hf > 0 || pr > 0 || kk > 0);
  }
}

__global__ void __launch_bounds__(kGroups * kTP, 1)
    mlp_eval_tc_kernel(const float* __restrict__ theta, const float* __restrict__ xy, int64_t npts,
                       float* __restrict__ v, float* __restrict__ gxy, int* __restrict__ err) {
  extern __shared__ unsigned char eval_raw[];
  EvalTcSmem& S = *reinterpret_cast<EvalTcSmem*>(
      (reinterpret_cast<uintptr_t>(eval_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int tid = threadIdx.x, warp = tid >> 5;
  const int g = tid / kTP, t = tid % kTP;  // warpgroup, point of the tile
  // the network, staged once: W2 and W2^T split into their TF32 hi / lo parts
  for (int i = tid; i < kH * kH; i += kGroups * kTP) {
    const float w = theta[kOffW2 + i], wh = tc::tf32_hi(w);
    const int o = i / kH, u = i % kH;
    const int ob = tc::swz_offset(o, u, kH), ot = tc::swz_offset(u, o, kH);
    *reinterpret_cast<float*>(reinterpret_cast<char*>(S.B1[0]) + ob) = wh;
    *reinterpret_cast<float*>(reinterpret_cast<char*>(S.B1[1]) + ob) = w - wh;
    *reinterpret_cast<float*>(reinterpret_cast<char*>(S.B2[0]) + ot) = wh;
    *reinterpret_cast<float*>(reinterpret_cast<char*>(S.B2[1]) + ot) = w - wh;
  }
  if (tid < kH) {
    S.w1x[tid] = theta[2 * tid];
    S.w1y[tid] = theta[2 * tid + 1];
    S.b1[tid] = theta[kOffB1 + tid];
    S.b2[tid] = theta[kOffB2 + tid];
    S.w3[tid] = theta[kOffW3 + tid];
  }
  if (tid == 0) {
    S.b3 = theta[kOffB3];
    for (int q = 0; q < kGroups; ++q) tc::mbar_init(&S.mbar[q]);
  }
  if (warp == 0) tc::tmem_alloc(&S.tmem, kColsGroup * kGroups);
  tc::fence_async_smem();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  // group g: TMEM columns [128 g, 128 g + 128); its warps read lanes 32 (warp % 4) ..
  const unsigned tm = S.tmem + kColsGroup * g, tm_s1 = tm + kH;
  const unsigned lane = (unsigned)((warp & 3) * 32) << 16;
  float* const A0 = S.A[g][0];
  float* const A1 = S.A[g][1];
  unsigned long long* const mbar = &S.mbar[g];
  unsigned phase = 0;
  bool ok = true;
  // The operand half in the buffers is complete: its product, by one thread.
  auto issue = [&](const float (&B)[2][kH * kH], int hf) {
    tc::fence_async_smem();
    tc::fence_before();
    group_sync(g);
    if (t == 0) {
      tc::fence_after();
      mma_half(tm, tc::smem_addr(A0), tc::smem_addr(A1), tc::smem_addr(B[0]), tc::smem_addr(B[1]), hf);
      tc::commit(mbar);
    }
  };
  auto wait = [&] {
    ok = tc::mbar_wait(mbar, phase, 2000000000ull) && ok;
    phase ^= 1u;
    tc::fence_after();
  };
  const int64_t stride = (int64_t)kGroups * gridDim.x * kTP;
  int64_t p = ((int64_t)g * gridDim.x + blockIdx.x) * kTP + t;
  auto point = [&](int64_t q) { return q < npts ? f2(xy[2 * q], xy[2 * q + 1]) : f2(0.f, 0.f); };
  float2 next = point(p);  // one tile ahead
  for (; p - t < npts; p += stride) {
    const bool valid = p < npts;
    const float x = next.x, y = next.y;
    next = point(p + stride);
    // layer 1, 16 units from u0 on: h into h[], SiLU' into TMEM
    auto layer1 = [&](int u0, float2* h) {
      float s1[16];
#pragma unroll
      for (int j = 0; j < 16; j += 2) {
        const int u = u0 + j;
        const float2 a = fma2(ld2(&S.w1x[u]), f2(x, x), fma2(ld2(&S.w1y[u]), f2(y, y), ld2(&S.b1[u])));
        const float2 sg = logistic2(a);
        h[j / 2] = mul2(a, sg);
        const float2 d = dsilu2(a, sg);
        s1[j] = d.x;
        s1[j + 1] = d.y;
      }
      tc::tmem_st16(tm_s1 + lane + u0, s1);
    };
    auto put16 = [&](int c0, const float2* h) {  // chunks c0 .. c0 + 3 of the half
#pragma unroll
      for (int c = 0; c < 4; ++c)
        put_split(A0, A1, tc::swz_chunk(t, c0 + c, kTP), h[2 * c], h[2 * c + 1]);
    };
    float2 h[16];
    layer1(0, h);
    put16(0, h);
    layer1(16, h);
    put16(4, h);
    issue(S.B1, 0);
    layer1(kHalf, h);
    layer1(kHalf + 16, h + 8);
    wait();
    put16(0, h);
    put16(4, h + 8);
    tc::st_wait();
    issue(S.B1, 1);
    wait();
    // a2 -> v and g2 = w3 SiLU'(a2), 32 outputs from o0 on
    float2 vs = f2(S.b3, 0.f);
    auto output = [&](int o0, float (&d)[32], float2* gg) {
#pragma unroll
      for (int j = 0; j < 32; j += 2) {
        const int o = o0 + j;
        const float2 a = add2(f2(d[j], d[j + 1]), ld2(&S.b2[o]));
        const float2 w = ld2(&S.w3[o]);
        const float2 sg = logistic2(a);
        vs = fma2(w, mul2(a, sg), vs);
        gg[j / 2] = mul2(w, dsilu2(a, sg));
      }
    };
    float d[32];
    tc::tmem_ld32(tm + lane, d);
    output(0, d, h);
    put16(0, h);
    put16(4, h + 8);
    tc::tmem_ld32(tm + lane + kHalf, d);  // before the backward product takes D's place
    issue(S.B2, 0);
    output(kHalf, d, h);
    wait();
    put16(0, h);
    put16(4, h + 8);
    issue(S.B2, 1);
    wait();
    // grad v = W1^T (dh1 * SiLU'(a1))
    float2 gx = f2(0.f, 0.f), gy = f2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float dh[16], s1[16];
      tc::tmem_ld16x2(tm + lane + 16 * q, tm_s1 + lane + 16 * q, dh, s1);
#pragma unroll
      for (int j = 0; j < 16; j += 2) {
        const int u = 16 * q + j;
        const float2 da = mul2(f2(dh[j], dh[j + 1]), f2(s1[j], s1[j + 1]));
        gx = fma2(da, ld2(&S.w1x[u]), gx);
        gy = fma2(da, ld2(&S.w1y[u]), gy);
      }
    }
    if (valid) {
      if (v) v[p] = vs.x + vs.y;
      gxy[2 * p] = gx.x + gx.y;
      gxy[2 * p + 1] = gy.x + gy.y;
    }
    // (the next product into D follows the group's next barrier, so every
    // thread has read its columns by then)
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after();
    tc::tmem_dealloc(S.tmem, kColsGroup * kGroups);
  }
  if (!ok && t == 0) atomicExch(err, (int)PDDS_ETIMEOUT);
}

}  // namespace
}  // namespace pdds

using namespace pdds;

extern "C" pdds_status pdds_mlp_eval_tc(const float* theta, const float* xy, int64_t npts, float* v,
                                        float* grad_xy, void* cuda_stream) {
  if (!theta || !xy || !grad_xy || npts < 1) {
    set_global_error("mlp_eval_tc: NULL pointer or npts < 1");
    return PDDS_EINVAL;
  }
  (void)cudaGetLastError();
  cudaStream_t s = (cudaStream_t)cuda_stream;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int* d_err = nullptr;
  DeviceScratch scratch;
  if (e == cudaSuccess) e = scratch.get(sizeof(int));
  d_err = static_cast<int*>(scratch.ptr());
  if (e == cudaSuccess) e = cudaMemsetAsync(d_err, 0, sizeof(int), s);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_eval_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kEvalTcSmemBytes);
  if (e == cudaSuccess) {
    const int64_t tiles = (npts + kTP - 1) / kTP;
    // a tile per SM first, then a second group's, and so on
    const int grid = (int)std::min<int64_t>(tiles, sms);
    mlp_eval_tc_kernel<<<grid, kGroups * kTP, kEvalTcSmemBytes, s>>>(theta, xy, npts, v, grad_xy,
                                                                      d_err);
    e = cudaGetLastError();
  }
  int herr = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost, s);
  // also after a failure: the buffer goes back only when nothing uses it
  const cudaError_t done = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = done;
  if (e != cudaSuccess) {
    set_global_error(std::string("mlp_eval_tc: ") + cudaGetErrorString(e));
    return PDDS_ECUDA;
  }
  if (herr != 0) {
    set_global_error("mlp_eval_tc: a tensor-core wait ran out (results incomplete)");
    return PDDS_ETIMEOUT;
  }
  return PDDS_OK;
}
