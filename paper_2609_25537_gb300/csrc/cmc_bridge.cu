// MemoryBridge output (Section 2.2, the norm-calibrated tanh equation): the
// decoder-ready CMEs from the output x of the MemoryBridge MLP,
//   m_hat = LayerNorm(x)  (mean and biased variance over the H_d features,
//                          eps, per-feature gamma and beta: PyTorch's default
//                          LayerNorm, as the hyperparameter appendix states)
//   m     = nu tanh(m_hat) min(1, 2 nu / ||nu tanh(m_hat)||_2)
// so that every CME's norm is at most 2 nu.  The MLP's two matrix products
// are plain library GEMMs and stay with the caller; this is the row-wise
// epilogue that turns their output into the bank the Tier-1 scoring reads.
//
// A row stays in the registers of the CTA that takes it (bridge_epilogue_kernel,
// below); the three row reductions (sum, squared deviations, squared norm of
// nu tanh) meet in a fixed tree.
// tanh(z) is evaluated as 1 - 2 / (1 + e^{2z}) with the hardware base-2
// exponential (ex2.approx, relative error ~2^-22) and a fast division:
// absolute error below 1e-6, saturating correctly to +-1.
// HBM-bound: 8 * H_d bytes per row.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "cmc_internal.cuh"

namespace cmc {

constexpr int kBridgeMaxD = 16384;

// tanh(z) = 1 - 2 / (1 + 2^(2 z log2 e)).
__device__ __forceinline__ float tanh_ex2(float z) {
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(e) : "f"(z * 2.8853900817779268f));
  return 1.f - __fdividef(2.f, 1.f + e);
}

// One CTA of NT threads per row, V float4s of it in each thread's registers; 64
// registers a thread, 1,024 / NT CTAs per SM, grid-stride over the rows.  Each
// reduction takes one barrier (its own partials array, summed by every thread
// in the same order).  Before the grid dependency wait a CTA asks L2 to prefetch
// its first row, so that under programmatic dependent launch the row streams in
// while the kernel before drains (a prefetch is a hint: L2 stays coherent with
// that kernel's writes to x), and, where that helps, at the start of each row the
// next one.
//
// Bound by HBM above a few thousand rows, by latency below.  With gamma or beta
// (kKept) their values are requested with the first row and kept for the CTA's
// later rows: requested where they are used, behind two reductions, they were
// one more trip to L2 per row (1,024 rows of 4,096: 11.8 us a call against 8.3
// without gamma and beta; now 9.4 and 7.7).  That takes 2 V more float4s, hence 256
// threads for rows of up to 4,096 features where a row alone takes 128 (V <= 8);
// longer rows take 512.
//
// kRead requests them, if there are any, where they are used.  That leaves room for
// more rows to an SM: eight of up to 4,096 features, for many rows (see
// bridge_many_rows), and two of over 8,192 (1,024 threads that kept them: 300 rows
// of 8,196 9.2 us a call, now 8.1; 8,000 157.7 and 116.8, plain 148.7 and 104.1; 8,000
// of 16,384 229 and 196, but 300 of those 13.3 and 13.8).
enum { kPlain, kKept, kRead };

template <int NT, int V, int MODE, bool AHEAD>
__global__ void __launch_bounds__(NT, 1024 / NT)
bridge_epilogue_kernel(const float* x, const float* __restrict__ gamma,
                       const float* __restrict__ beta, long long rows, int D, float eps, float nu,
                       float* out) {
  constexpr int NW = NT / 32;
  constexpr bool kKeep = MODE == kKept;
  __shared__ float red[3][NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // D * 4 bytes of a 16-byte aligned row (D a multiple of 4): the bulk
  // prefetch's alignment and size rules hold
  auto prefetch = [&](long long r) {
    if (tid == 0 && r < rows)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(x + r * D),
                   "r"(static_cast<unsigned int>(D) * 4u)
                   : "memory");
  };
  prefetch(blockIdx.x);
  pdl_wait();
  pdl_trigger();
  const int D4 = D >> 2;
  auto block_sum = [&](float v, float* part) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane == 0) part[warp] = v;
    __syncthreads();
    if (NW <= 8) {
      float t = part[0];
#pragma unroll
      for (int w = 1; w < NW; ++w) t += part[w];
      return t;
    }
    float t = lane < NW ? part[lane] : 0.f;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    return t;
  };
  float4 gv[kKeep ? V : 1], bv[kKeep ? V : 1];
  for (long long r = blockIdx.x; r < rows; r += gridDim.x) {
    float4 cur[V];
    const float4* src = reinterpret_cast<const float4*>(x + r * D);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const int i = tid + e * NT;
      cur[e] = i < D4 ? __ldcs(src + i) : make_float4(0.f, 0.f, 0.f, 0.f);  // coherent: x may be out
    }
    if (kKeep && r == blockIdx.x) {
#pragma unroll
      for (int e = 0; e < (kKeep ? V : 1); ++e) {
        const int i = tid + e * NT;
        gv[e] = (gamma && i < D4) ? __ldg(reinterpret_cast<const float4*>(gamma) + i)
                                  : make_float4(1.f, 1.f, 1.f, 1.f);
        bv[e] = (beta && i < D4) ? __ldg(reinterpret_cast<const float4*>(beta) + i)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    if (AHEAD) prefetch(r + gridDim.x);
    float s = 0.f;
#pragma unroll
    for (int e = 0; e < V; ++e) s += (cur[e].x + cur[e].y) + (cur[e].z + cur[e].w);
    const float mean = block_sum(s, red[0]) / static_cast<float>(D);
    float q = 0.f;
#pragma unroll
    for (int e = 0; e < V; ++e) {
      if (tid + e * NT < D4) {
        const float a = cur[e].x - mean, b = cur[e].y - mean, c = cur[e].z - mean, d = cur[e].w - mean;
        q += (a * a + b * b) + (c * c + d * d);
      }
    }
    const float var = block_sum(q, red[1]) / static_cast<float>(D);
    const float rstd = 1.0f / sqrtf(var + eps);
    float n2 = 0.f;
#pragma unroll
    for (int e = 0; e < V; ++e) {
      if (tid + e * NT < D4) {
        float4 g = make_float4(1.f, 1.f, 1.f, 1.f), b = make_float4(0.f, 0.f, 0.f, 0.f);
        if (kKeep) {
          g = gv[kKeep ? e : 0];
          b = bv[kKeep ? e : 0];
        } else if (MODE == kRead) {
          if (gamma) g = __ldg(reinterpret_cast<const float4*>(gamma) + tid + e * NT);
          if (beta) b = __ldg(reinterpret_cast<const float4*>(beta) + tid + e * NT);
        }
        float4& t = cur[e];
        t.x = nu * tanh_ex2(fmaf(g.x, (t.x - mean) * rstd, b.x));
        t.y = nu * tanh_ex2(fmaf(g.y, (t.y - mean) * rstd, b.y));
        t.z = nu * tanh_ex2(fmaf(g.z, (t.z - mean) * rstd, b.z));
        t.w = nu * tanh_ex2(fmaf(g.w, (t.w - mean) * rstd, b.w));
        n2 += (t.x * t.x + t.y * t.y) + (t.z * t.z + t.w * t.w);
      }
    }
    const float norm = sqrtf(block_sum(n2, red[2]));
    const float f = (norm > 2.f * nu) ? (2.f * nu) / norm : 1.f;
    float4* orow = reinterpret_cast<float4*>(out + r * D);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const int i = tid + e * NT;
      if (i < D4) orow[i] = make_float4(cur[e].x * f, cur[e].y * f, cur[e].z * f, cur[e].w * f);
    }
    __syncthreads();  // red is rewritten by the next row of this CTA
  }
}

// Whether `rows` rows are so many that the kRead variant is the faster one (for
// widths of 1,537 to 4,096 features).  Kept gamma and beta leave four rows to an SM,
// and threads without work where the width is no multiple of 1,024; with many rows
// an SM that costs more than the trip to L2, the earlier the fewer threads work.
// us a call, kept / read: 30,000 rows of 2,560 118.8 / 103.8, 32,000 of 3,328 162.0 /
// 140.8, 10,000 of 2,052 41.3 / 36.6, but 5,000 of 3,072 23.8 / 26.2 and 32,000 of
// 4,096 178.0 / 179.9.  Plain rows, whose loads are the same in both, gain 1 to 3 %
// at some widths (the cause is not known): 32,000 of 4,096 173.4 / 171.5, of 3,840
// 161.6 / 158.0, of 2,048 (with the next row's prefetch) 90.5 / 87.9, but 5,000 of
// 4,096 28.6 / 28.9.
static bool bridge_many_rows(long long rows, int D4, bool affine) {
  const long long per_sm = rows / sm_count();
  if (D4 > 512) {
    if (!affine) return D4 > 704 && per_sm > 50;
    const int V = (D4 + 255) / 256;
    return D4 < 1020 && per_sm > 120 * D4 / (256 * V) - 62;  // 18 to 58
  }
  return affine ? D4 <= 416 && per_sm > 100 : D4 > 480 && per_sm > 80;
}

template <int NT, int V, int MODE, bool AHEAD>
static int launch_bridge(const float* x, const float* gamma, const float* beta, long long rows, int D,
                         float eps, float nu, float* out, cudaStream_t s) {
  const long long cap = static_cast<long long>(sm_count()) * (1024 / NT);
  const long long grid = rows < cap ? rows : cap;
  return launch_pdl(bridge_epilogue_kernel<NT, V, MODE, AHEAD>, dim3(static_cast<unsigned>(grid)), dim3(NT), 0,
                    s, x, gamma, beta, rows, D, eps, nu, out);
}

}  // namespace cmc

extern "C" {

int cmc_bridge_epilogue(const float* x, const float* gamma, const float* beta, int64_t rows, int D,
                        float eps, float nu, float* out, void* stream) {
  using namespace cmc;
  if (rows < 1 || D < 4 || D > kBridgeMaxD || (D & 3)) return CMC_ERR_SHAPE;
  if (!(eps > 0.f) || !(nu > 0.f) || !isfinite(eps) || !isfinite(nu)) return CMC_ERR_RANGE;
  if (!x || !out) return CMC_ERR_NULL;
  if (!aligned16(x) || !aligned16(out) || (gamma && !aligned16(gamma)) || (beta && !aligned16(beta)))
    return CMC_ERR_ALIGN;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int D4 = D / 4;
  const long long R = static_cast<long long>(rows);
  const bool affine = gamma || beta;
  // NT threads; V float4s a thread.  The next row's prefetch: eight CTAs of 128 threads
  // with 8 to 16 KB of row each keep HBM busy by themselves; there it only
  // competes (8,000 rows of 4,096: 49.9 us with it, 46.4 without; 3,000 of 2,048:
  // 21.9 and 24.5 for two calls).
#define CMC_BRIDGE_CASE(NT, V, MODE, AHEAD) \
  case V: return launch_bridge<NT, V, MODE, AHEAD>(x, gamma, beta, R, D, eps, nu, out, s);
  if (D4 > 384 && D4 <= 1024 && bridge_many_rows(R, D4, affine)) {
    switch ((D4 + 127) / 128) {
      CMC_BRIDGE_CASE(128, 4, kRead, true)
      CMC_BRIDGE_CASE(128, 5, kRead, false) CMC_BRIDGE_CASE(128, 6, kRead, false)
      CMC_BRIDGE_CASE(128, 7, kRead, false) CMC_BRIDGE_CASE(128, 8, kRead, false)
    }
  } else if (D4 <= 1024 && !affine) {
    switch ((D4 + 127) / 128) {
      CMC_BRIDGE_CASE(128, 1, kPlain, true) CMC_BRIDGE_CASE(128, 2, kPlain, true)
      CMC_BRIDGE_CASE(128, 3, kPlain, true) CMC_BRIDGE_CASE(128, 4, kPlain, true)
      CMC_BRIDGE_CASE(128, 5, kPlain, false) CMC_BRIDGE_CASE(128, 6, kPlain, false)
      CMC_BRIDGE_CASE(128, 7, kPlain, false) CMC_BRIDGE_CASE(128, 8, kPlain, false)
    }
  } else if (D4 <= 512) {
    switch ((D4 + 127) / 128) {
      CMC_BRIDGE_CASE(128, 1, kKept, true) CMC_BRIDGE_CASE(128, 2, kKept, true)
      CMC_BRIDGE_CASE(128, 3, kKept, true) CMC_BRIDGE_CASE(128, 4, kKept, true)
    }
  } else if (D4 <= 1024) {
    switch ((D4 + 255) / 256) {
      CMC_BRIDGE_CASE(256, 3, kKept, true) CMC_BRIDGE_CASE(256, 4, kKept, true)
    }
  } else if (D4 <= 2048 && !affine) {
    switch ((D4 + 511) / 512) {
      CMC_BRIDGE_CASE(512, 3, kPlain, true) CMC_BRIDGE_CASE(512, 4, kPlain, true)
    }
  } else if (D4 <= 2048) {
    switch ((D4 + 511) / 512) {
      CMC_BRIDGE_CASE(512, 3, kKept, true) CMC_BRIDGE_CASE(512, 4, kKept, true)
    }
  } else if (!affine) {
    switch ((D4 + 511) / 512) {
      CMC_BRIDGE_CASE(512, 5, kPlain, true) CMC_BRIDGE_CASE(512, 6, kPlain, true)
      CMC_BRIDGE_CASE(512, 7, kPlain, true) CMC_BRIDGE_CASE(512, 8, kPlain, true)
    }
  } else {
    switch ((D4 + 511) / 512) {
      CMC_BRIDGE_CASE(512, 5, kRead, true) CMC_BRIDGE_CASE(512, 6, kRead, true)
      CMC_BRIDGE_CASE(512, 7, kRead, true) CMC_BRIDGE_CASE(512, 8, kRead, true)
    }
  }
#undef CMC_BRIDGE_CASE
  return CMC_ERR_SHAPE;  // not reached: the cases cover 4 <= D <= kBridgeMaxD
}

}  // extern "C"
