// fst_small32.cuh -- FP32 projection of one pair per CTA for 2^10 <= M <= 2^14 (device only).
//
// The whole projection of a pair in one launch, as small_body of fst_kernels.cuh, restructured:
//   * T = M/16 threads keep 16 values each in registers; M = 16^a R0 (R0 = 1, 2, 4, 8).  Forward:
//     radix 16 (its upper half inputs are the zero padding), radix 16, ..., radix R0 last, so the
//     spectrum product and the inverse's first radix-R0 stage happen on the same registers;
//     inverse: radix R0, radix 16, ..., the last one forming only the rows that hold output.
//     One shared-memory exchange per stage; every stage twiddle is one table entry.
//   * the rank-r correction reads half of S_T (s_l(N-1-n) = (-1)^l s_l(n)): S_T^T y with 16-byte
//     row pieces (rpad / 4 threads per row), S_T a sample by sample from the K-major copy of S_T,
//     whose columns are coalesced along the samples.
// Bound: FP32 issue and the S_T reads from L2 (both copies of the half, once per pair).
// Measured, 999 signals of N = 3001, r = 25: 273 -> 65 us.
#pragma once
#include "fst_fast.cuh"

namespace fst {

__host__ __device__ constexpr size_t sm_smem(int log2M, int rpad) {
  return (size_t)padded_size(1 << log2M) * 8 + 2 * (size_t)rpad * 4 + 16;
}
__global__ void k_tw_small(Tw<double> tw, int log2M, float2 *dst) {
  const int total = sm_words(log2M), n16 = sm_n16(log2M);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    int i = 0, ns = sm_r0(log2M), o = 0;
    while (i < n16 && e >= o + 16 * ns) {
      o += 16 * ns;
      ns *= 16;
      ++i;
    }
    double2 w;
    if (i < n16) w = tw.root<false>((uint64_t)((e - o) / ns) * (uint64_t)((e - o) % ns), (log2M & 3) + 4 * i + 4);
    else {
      const int mr = (1 << log2M) / sm_r0(log2M);
      w = tw.root<false>((uint64_t)((e - o) / mr + 1) * (uint64_t)((e - o) % mr), log2M);
    }
    dst[e] = make_float2((float)w.x, (float)w.y);
  }
}

// word w < 4 of the antisymmetric bits, by selects (a run-time index would put the plan in local memory)
__device__ __forceinline__ unsigned sm_odd(const SmallPlan &p, int w) {
  return w < 2 ? (w == 0 ? p.odd[0] : p.odd[1]) : (w == 2 ? p.odd[2] : p.odd[3]);
}
// LD: n -> float2 of the pair (n < N); SV: (n, value)
template <int LM, typename LD, typename SV>
__device__ __forceinline__ void small32_body(const SmallPlan &p, const float2 *twB, bool corr, LD load, SV store) {
  constexpr int M = 1 << LM, T = M / 16, R0 = sm_r0(LM), N16 = sm_n16(LM), PER = 16 / R0;
  extern __shared__ __align__(16) float2 sbuf[];
  float2 *coef = sbuf + ((padded_size(M) + 1) & ~1);   // (re, im) of a, [rpad]
  const int j = threadIdx.x, N = p.N, H = (N + 1) / 2;
  float2 x[16];
  if (!corr) {
#pragma unroll
    for (int t = 0; t < 8; ++t) x[t] = (j + T * t < N) ? load(j + T * t) : make_float2(0.f, 0.f);
  } else {
    // y in natural order in the first half of the buffer, partial sums in the second half
#pragma unroll
    for (int t = 0; t < 8; ++t) sbuf[j + T * t] = (j + T * t < N) ? load(j + T * t) : make_float2(0.f, 0.f);
    __syncthreads();
    const int tpr = p.rpad / 4, rpr = T / tpr, slot = j / tpr, jq = j % tpr;
    float *red = reinterpret_cast<float *>(sbuf + M / 2);   // [rpr][rpad][2], at most M/2 floats
    if (slot < rpr) {
      float2 A[4], B[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) A[c] = B[c] = make_float2(0.f, 0.f);
      const float4 *S4 = reinterpret_cast<const float4 *>(p.ST) + jq;
#pragma unroll 8
      for (int n = slot; n < H; n += rpr) {
        const float4 s = __ldg(S4 + (int64_t)n * tpr);
        const float2 v = sbuf[n];
        float2 u = sbuf[N - 1 - n];
        if (N - 1 - n == n) u = make_float2(0.f, 0.f);
        const float sc[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          A[c].x = fmaf(sc[c], v.x, A[c].x);
          A[c].y = fmaf(sc[c], v.y, A[c].y);
          B[c].x = fmaf(sc[c], u.x, B[c].x);
          B[c].y = fmaf(sc[c], u.y, B[c].y);
        }
      }
      const unsigned odd = sm_odd(p, (4 * jq) >> 5) >> ((4 * jq) & 31);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float2 s = ((odd >> c) & 1u) ? csub(A[c], B[c]) : cadd(A[c], B[c]);
        reinterpret_cast<float2 *>(red)[slot * p.rpad + 4 * jq + c] = s;
      }
    }
    __syncthreads();
    // sums in a fixed order: part q of value o adds slots q, q + parts, ...
    const int no = 2 * p.rpad, parts = T / no > 0 ? T / no : 1;
    float *red2 = red + M / 2;                               // [parts][no]
    for (int e = j; e < parts * no; e += T) {
      const int o = e % no, q = e / no;
      float s = 0.f;
      for (int i = q; i < rpr; i += parts) s += red[i * no + o];
      red2[e] = s;
    }
    __syncthreads();
    for (int o = j; o < no; o += T) {
      float s = 0.f;
      for (int q = 0; q < parts; ++q) s += red2[q * no + o];
      reinterpret_cast<float *>(coef)[o] = (o >> 1) < p.r ? __ldg(p.D + (o >> 1)) * s : 0.f;
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) x[t] = sbuf[j + T * t];
    __syncthreads();
  }

  // ---- forward -------------------------------------------------------------------------------
  dft_half_in<16>(x);
#pragma unroll
  for (int t = 0; t < 16; ++t) sbuf[pad(16 * j + t)] = x[t];
  __syncthreads();
#pragma unroll
  for (int s = 1; s < N16; ++s) {
    const int ns = 1 << (4 * s), k = j & (ns - 1);
#pragma unroll
    for (int t = 0; t < 16; ++t) x[t] = sbuf[pad(j + T * t)];
    tw_table16<true>(twB + (s == 1 ? 0 : 256), ns, k, false, x);
    Dft<float, 16, false>::run(x);
    if (R0 > 1 || s + 1 < N16) {
      __syncthreads();
#pragma unroll
      for (int t = 0; t < 16; ++t) sbuf[pad(((j - k) << 4) + k + ns * t)] = x[t];
      __syncthreads();
    }
  }
  if (R0 > 1) {
    const float2 *F = p.twS + sm_off(LM, N16);
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int jq = j + T * q;
#pragma unroll
      for (int t = 0; t < R0; ++t) {
        x[q * R0 + t] = sbuf[pad(jq + (M / R0) * t)];
        if (t > 0) x[q * R0 + t] = cmul(x[q * R0 + t], F[(t - 1) * (M / R0) + jq]);
      }
      RegDft<(R0 > 1 ? R0 : 2), false>::run(x + q * R0);
    }
  }
  // ---- spectrum, at the positions jq + (M / R0) t (R0 = 1: j + T t) ---------------------------
#pragma unroll
  for (int q = 0; q < PER; ++q)
#pragma unroll
    for (int t = 0; t < R0; ++t) {
      const int k = R0 > 1 ? j + T * q + (M / R0) * t : j + T * q;
      x[q * R0 + t] = cscale(x[q * R0 + t], __ldg(p.spec + k));
    }
  // ---- inverse -------------------------------------------------------------------------------
  __syncthreads();
  if (R0 > 1) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      RegDft<(R0 > 1 ? R0 : 2), true>::run(x + q * R0);
#pragma unroll
      for (int t = 0; t < R0; ++t) sbuf[pad(R0 * (j + T * q) + t)] = x[q * R0 + t];
    }
  } else {
    Dft<float, 16, true>::run(x);
#pragma unroll
    for (int t = 0; t < 16; ++t) sbuf[pad(16 * j + t)] = x[t];
  }
  __syncthreads();
  float2 o[8];
#pragma unroll
  for (int i = R0 > 1 ? 0 : 1; i < N16; ++i) {
    const int ns = R0 << (4 * i), k = j & (ns - 1);
#pragma unroll
    for (int t = 0; t < 16; ++t) x[t] = sbuf[pad(j + T * t)];
    tw_table16<true>(R0 > 1 ? p.twS + sm_off(LM, i) : twB + (i == 1 ? 0 : 256), ns, k, true, x);
    if (i + 1 < N16) {
      Dft<float, 16, true>::run(x);
      __syncthreads();
#pragma unroll
      for (int t = 0; t < 16; ++t) sbuf[pad(((j - k) << 4) + k + ns * t)] = x[t];
      __syncthreads();
    } else {
      idft_half_out<16>(x, o);
    }
  }
  if (corr) {
    // z(n) and z(N-1-n) for n < H, through shared memory to the threads that hold the samples
    __syncthreads();
    // (a thread's samples j + T q, q < 4, side by side: their loads overlap; H <= M/4 = 4 T)
    float2 zp[4], zm[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) zp[q] = zm[q] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int c = 0; c < p.r; ++c) {
      const float *col = p.STt + (int64_t)c * p.ld_t + j;
      const float2 w = coef[c];
      float s[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) s[q] = j + T * q < H ? __ldg(col + T * q) : 0.f;
      if ((sm_odd(p, c >> 5) >> (c & 31)) & 1u) {   // uniform
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          zm[q].x = fmaf(s[q], w.x, zm[q].x);
          zm[q].y = fmaf(s[q], w.y, zm[q].y);
        }
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          zp[q].x = fmaf(s[q], w.x, zp[q].x);
          zp[q].y = fmaf(s[q], w.y, zp[q].y);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int n = j + T * q;
      if (n < H) {
        sbuf[n] = cadd(zp[q], zm[q]);
        if (N - 1 - n != n) sbuf[N - 1 - n] = csub(zp[q], zm[q]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 8; ++t)
      if (j + T * t < N) o[t] = cadd(o[t], sbuf[j + T * t]);
  }
#pragma unroll
  for (int t = 0; t < 8; ++t)
    if (j + T * t < N) store(j + T * t, o[t]);
}

// grid: pairs; T threads; 1024 resident threads per SM, whose 64 registers each fill the register file
template <int LM>
__global__ void __launch_bounds__((1 << LM) / 16, 1024 / ((1 << LM) / 16)) k_small32(const ConvArgs<float> a,
                                                                                     const SmallPlan p) {
  const int64_t pl = blockIdx.x;
  small32_body<LM>(p, a.twB, a.mode == MODE_FULL && p.r > 0, [&](int n) { return load_pair(a, pl, n); },
                   [&](int n, float2 v) { store_pair(a, pl, n, v); });
}
template <int LM>
__global__ void __launch_bounds__((1 << LM) / 16, 1024 / ((1 << LM) / 16)) k_small32_ragged(const SmallDesc *d,
                                                                                            const float2 *twB, int cplx) {
  __shared__ SmallDesc q;
  if (threadIdx.x == 0) q = d[blockIdx.x];
  __syncthreads();
  if (cplx)
    small32_body<LM>(q.p, twB, q.p.r > 0, [&](int n) { return reinterpret_cast<const float2 *>(q.y)[n]; },
                     [&](int n, float2 v) { reinterpret_cast<float2 *>(q.out)[n] = v; });
  else
    small32_body<LM>(q.p, twB, q.p.r > 0, [&](int n) { return make_float2(q.y[n], 0.f); },
                     [&](int n, float2 v) { q.out[n] = v.x; });
}

}  // namespace fst
