// fst_lowrank.cuh -- FP32 kernels of the generated low-rank columns of T2^* y and T1 c (device only,
// N a power of two, N >= 128).
//
// Both sides are products with the same real columns of length N: Z_k(n), Z_k(N-1-n) (CF-ADI
// recurrence), the monomials u_n^i, and for T1 c the S_T columns.  Two things make them cheap:
//   * a column value is generated once per sample and block and used for every signal of the
//     block from shared memory (before, each group of 4 signals, or each vector, generated its own);
//   * the columns come in mirror pairs: Z_k(n) and Z_k(N-1-n), u_{N-1-n} = -u_n, s(N-1-n) = +-s(n).
//     With e = (Z_k(n) + Z_k(N-1-n)) and o = (Z_k(n) - Z_k(N-1-n)), n < H = N/2, sums over all samples
//     are sums over n < H of e (v(n) + v(N-1-n)) and of o (v(n) - v(N-1-n)): half the FMAs.
// Bound: FP32 FMA (packed, two results per instruction) next to the shared-memory reads.
#pragma once
#include "fst_fast.cuh"
#include "fst_coeffs.cuh"

namespace fst {

constexpr int LR_TN = 64;        // folded samples per tile
constexpr int LR_VC = 16;        // complex vector columns per block: real signals, or (signal, +-phase)
constexpr int LR_FLUSH = 8;      // tiles between two additions into the block's own sums in memory
constexpr int LR_VS = 2 * LR_VC + 4;

// column blocks, padded to 8: ZE [rH], PE [even powers], ZO [rH], PO [odd powers]
struct LrShape {
  int rH, DA, DB, nz, npe, npo;   // nz, npe, npo: padded sizes
  int cs;                         // floats per sample of the column tile
  int nvt, nct, ntile, kg;        // 8-wide vector tiles, column tiles, their product, sample groups
};
__host__ __device__ inline LrShape lr_shape(int rH, int DA, int DB, int vc) {
  LrShape s;
  s.rH = rH;
  s.DA = DA;
  s.DB = DB;
  const int D = DA > DB ? DA : DB;
  s.nz = (rH + 7) / 8 * 8;
  s.npe = ((D + 1) / 2 + 7) / 8 * 8;
  s.npo = (D / 2 + 7) / 8 * 8;
  s.cs = 2 * s.nz + s.npe + s.npo + 4;
  s.nvt = (2 * vc + 7) / 8;
  // column tiles: ZE PE ZO PO for the W' phase, PE PO for the W + W' phase
  s.nct = (2 * s.nz + 2 * (s.npe + s.npo)) / 8;
  s.ntile = s.nvt * s.nct;
  s.kg = s.ntile > 0 && s.ntile <= 256 ? 256 / s.ntile : 0;
  return s;
}
__host__ __device__ inline size_t lr_smem(const LrShape &s) {
  const size_t tile = 2 * (size_t)LR_TN * (s.cs + 4 * LR_VS), sums = (size_t)s.kg * s.ntile * 64;
  return (tile > sums ? tile : sums) * 4;
}

// (re, im) pair times a real, packed: acc += (c, c) * w
__device__ __forceinline__ void fma2(float2 &acc, float c, float2 w) { acc = __ffma2_rn(make_float2(c, c), w, acc); }

// ADI factor of step k at x: z_k = z_{k-1} sc (x - p_{k-1}) / (x + p_k)
__device__ __forceinline__ float lr_zstep(const float *zfirst, const float *zshift, int k, float x) {
  return __fdividef(zfirst[k] * (x - zshift[k - 1]), x + zshift[k]);
}

// ---------------------------------------------------------------------------
// raw low-rank sums of T2^* y, grid (nchunk, vector groups), 512 threads, dynamic lr_smem
//   a tile: 64 folded samples, two buffers.  The upper eight warps generate the next tile: four the
//   Z columns (one of the two mirror samples a thread, combined by a shuffle), four the powers and
//   the folded, phase-rotated vectors.  Meanwhile thread (column tile, vector tile, sample group)
//   of the lower eight accumulates 8 x 8 sums of the current one: per sample 4 16-byte loads feed
//   32 packed FMAs.  Named barriers 1, 2 (tile ready) and 3, 4 (buffer free) hand the buffers
//   over: each side arrives exactly as often as the other waits.  Every LR_FLUSH tiles the sums are added to the
//   block's own area of `scr`, which keeps the FP32 chains short; sample groups are added in order
//   at the end.  Same output layout as coef_lowrank_body.
// Measured, 16 real signals of N = 2^22, 38 + 38 + 31 columns: 3476 -> 770 us
// (960 with all warps generating, then multiplying).
// ---------------------------------------------------------------------------
// half of a named barrier of all 512 threads: wait for it, or only count towards it
__device__ __forceinline__ void lr_bar_sync(int id) {
  __syncwarp();
  asm volatile("bar.sync %0, 512;" ::"r"(id) : "memory");
}
__device__ __forceinline__ void lr_bar_arrive(int id) {
  __syncwarp();
  asm volatile("bar.arrive %0, 512;" ::"r"(id) : "memory");
}
__global__ void __launch_bounds__(512, 1) k_coef_gemm(const CoefArgs<float> a, int nchunk, float *scr) {
  extern __shared__ __align__(16) float lsm[];
  const int tid = threadIdx.x;
  const int64_t H = a.N / 2, nvc = a.cplx ? 2 * a.batch : a.batch;
  const int64_t c0 = (int64_t)blockIdx.y * LR_VC;
  const int vc = (int)(nvc - c0 < LR_VC ? nvc - c0 : LR_VC);
  const LrShape S = lr_shape(a.rH, a.DA, a.DB, vc);
  const int tile_f = LR_TN * (S.cs + 4 * LR_VS);   // floats of a buffer: columns, then PA, DA, PB, DB, each [LR_TN][LR_VS]
  const int64_t ntl = (H + LR_TN - 1) / LR_TN;
  const int64_t t0 = ntl * blockIdx.x / nchunk, t1 = ntl * (blockIdx.x + 1) / nchunk;
  // this thread's sums
  const int id = tid % S.ntile, kgi = tid / S.ntile, vt = id % S.nvt, ct = id / S.nvt;
  const bool gen = tid >= 256, on = !gen && kgi < S.kg;
  const int ne = (S.nz + S.npe) / 8, nA = ne + (S.nz + S.npo) / 8;
  const int cA = ct < nA ? ct * 8 : (ct - nA < S.npe / 8 ? S.nz + (ct - nA) * 8 : 2 * S.nz + S.npe + (ct - nA - S.npe / 8) * 8);
  const int vsel = ct < nA ? (ct < ne ? 0 : 1) : (ct - nA < S.npe / 8 ? 2 : 3);
  const float *cp = lsm + cA, *vp = lsm + LR_TN * S.cs + vsel * LR_TN * LR_VS + vt * 8;
  float2 acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[i][q] = make_float2(0.f, 0.f);
  float2 *own = reinterpret_cast<float2 *>(scr) + ((int64_t)blockIdx.y * nchunk + blockIdx.x) * 32 * 256 + tid;
  bool fresh = true;
  auto flush = [&]() {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float2 v = acc[i][q];
        if (!fresh) v = cadd(v, own[(i * 4 + q) * 256]);
        own[(i * 4 + q) * 256] = v;
        acc[i][q] = make_float2(0.f, 0.f);
      }
    fresh = false;
  };
  const float Nd = (float)a.N, cen = (float)(0.5 * (double)(a.N - 1)), invN = (float)(1.0 / (double)a.N);
  int since = 0;
  for (int64_t t = t0; t < t1; ++t) {
    const int buf = (int)((t - t0) & 1);
    if (gen) {
      if (t >= t0 + 2) lr_bar_sync(3 + buf);
      float *cols = lsm + buf * tile_f, *V = cols + LR_TN * S.cs;
      const int64_t n0 = t * LR_TN;
      if (tid < 384) {
        const int i = (tid - 256) >> 1, side = tid & 1;
        const int64_t n = n0 + i;
        const float xf = (float)n + 0.5f, x = side ? Nd - xf : xf;
        float *dst = cols + i * S.cs + (side ? S.nz + S.npe : 0);
        float z = __fdividef(a.zfirst[0], x + a.zshift[0]);
        for (int k0 = 0; k0 < S.nz; k0 += 4) {
          float v[4];
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const int k = k0 + kk;
            if (k > 0 && k < a.rH) z *= lr_zstep(a.zfirst, a.zshift, k, x);
            const float other = __shfl_xor_sync(0xffffffffu, z, 1);
            v[kk] = k < a.rH ? (side ? other - z : z + other) : 0.f;
          }
          *reinterpret_cast<float4 *>(dst + k0) = make_float4(v[0], v[1], v[2], v[3]);
        }
      } else {
        const int i = (tid - 384) & 63, g = (tid - 384) >> 6;
        const int64_t n = n0 + i, m = a.N - 1 - n;
        const bool in = n < H;
        const float2 z2 = make_float2(0.f, 0.f);
        // every load of the tile first: signals s = g + 2 q, q < LR_VC / 2
        float2 y1[LR_VC / 2], y2[LR_VC / 2];
#pragma unroll
        for (int q = 0; q < LR_VC / 2; ++q) {
          const int s = g + 2 * q;
          y1[q] = y2[q] = z2;
          if (in && s < vc) {
            if (!a.cplx) {
              const float *row = a.y + (c0 + s) * a.ld;
              y1[q].x = __ldg(row + n);
              y2[q].x = __ldg(row + m);
            } else {
              const float2 *row = reinterpret_cast<const float2 *>(a.y) + ((c0 + s) >> 1) * a.ld;
              y1[q] = __ldg(row + n);
              y2[q] = __ldg(row + m);
            }
          }
        }
        const float2 pa = in ? a.phA[n] : z2, pam = in ? a.phA[m] : z2, pb = in ? a.phB[n] : z2, pbm = in ? a.phB[m] : z2;
        const float u = ((float)n - cen) * invN, u2 = u * u;
        {
          float p = g ? u : 1.f;
          const int np = g ? S.npo : S.npe, D = (a.DA > a.DB ? a.DA : a.DB) - g;
          float *dst = cols + i * S.cs + (g ? 2 * S.nz + S.npe : S.nz);
          for (int k0 = 0; k0 < np; k0 += 4) {
            float v[4];
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              v[kk] = 2 * (k0 + kk) < D ? p : 0.f;
              p *= u2;
            }
            *reinterpret_cast<float4 *>(dst + k0) = make_float4(v[0], v[1], v[2], v[3]);
          }
        }
#pragma unroll
        for (int q = 0; q < LR_VC / 2; ++q) {
          const int s = g + 2 * q;
          if (s < 4 * S.nvt) {
            float2 an, am, bn, bm;
            if (!a.cplx) {
              an = cscale(pa, y1[q].x);
              am = cscale(pam, y2[q].x);
              bn = cscale(pb, y1[q].x);
              bm = cscale(pbm, y2[q].x);
            } else {
              const bool cj = ((c0 + s) & 1) != 0;
              an = cmul(cj ? cconj(pa) : pa, y1[q]);
              am = cmul(cj ? cconj(pam) : pam, y2[q]);
              bn = cmul(cj ? cconj(pb) : pb, y1[q]);
              bm = cmul(cj ? cconj(pbm) : pbm, y2[q]);
            }
            float2 *w = reinterpret_cast<float2 *>(V + i * LR_VS) + s;
            w[0] = cadd(an, am);
            w[LR_TN * LR_VS / 2] = csub(an, am);
            w[LR_TN * LR_VS] = cadd(bn, bm);
            w[3 * LR_TN * LR_VS / 2] = csub(bn, bm);
          }
        }
      }
      lr_bar_arrive(1 + buf);
    } else {
      lr_bar_sync(1 + buf);
      if (on) {
        const float *cb = cp + buf * tile_f, *vb = vp + buf * tile_f;
#pragma unroll 2
        for (int i = kgi; i < LR_TN; i += S.kg) {
          const float4 x0 = *reinterpret_cast<const float4 *>(cb + i * S.cs), x1 = *reinterpret_cast<const float4 *>(cb + i * S.cs + 4);
          const float4 w0 = *reinterpret_cast<const float4 *>(vb + i * LR_VS), w1 = *reinterpret_cast<const float4 *>(vb + i * LR_VS + 4);
          const float c[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
          const float2 w[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y), make_float2(w1.z, w1.w)};
#pragma unroll
          for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) fma2(acc[r][q], c[r], w[q]);
        }
      }
      if (t + 2 < t1) lr_bar_arrive(3 + buf);
      if (++since == LR_FLUSH) {
        flush();
        since = 0;
      }
    }
  }
  if (!gen && since) flush();
  __syncthreads();
  // sums of the sample groups in order: red[kg][tile][8 columns][8 floats]
  float *red = lsm;
  if (on && !fresh) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        reinterpret_cast<float2 *>(red)[((kgi * S.ntile + id) * 8 + i) * 4 + q] = own[(i * 4 + q) * 256];
  } else if (on) {
    for (int e = 0; e < 64; ++e) red[(kgi * S.ntile + id) * 64 + e] = 0.f;
  }
  __syncthreads();
  for (int e = tid; e < S.ntile * 64; e += 512) {
    float s = red[e];
    for (int q = 1; q < S.kg; ++q) s += red[q * S.ntile * 64 + e];
    red[e] = s;
  }
  __syncthreads();
  // column tile c8, column c of it, complex vector column s
  auto at = [&](int tile, int c, int s) {
    return reinterpret_cast<const float2 *>(red)[((tile * S.nvt + (s >> 2)) * 8 + c) * 4 + (s & 3)];
  };
  const int nq = a.rH + a.DA + a.DB;
  const int vbase[4] = {0, 2 * a.rH + a.DA, 4 * a.rH + 2 * a.DA, 4 * a.rH + 2 * a.DA + a.DB};
  for (int e = tid; e < vc * nq; e += 512) {
    const int s = e / nq, k = e % nq;
    const int64_t sig = a.cplx ? (c0 + s) >> 1 : c0 + s;
    const int var = a.cplx ? (int)((c0 + s) & 1) : 0;
    float2 *out = reinterpret_cast<float2 *>(a.part) + (sig * a.nchunks + blockIdx.x) * (int64_t)a.nraw;
    auto put = [&](int variant, int o, float2 v) {
      out[vbase[variant] + o] = v;
      if (!a.cplx) out[vbase[variant + 1] + o] = cconj(v);   // real signals: the other phase's sums
    };
    if (k < a.rH) {
      const float2 E = at(k >> 3, k & 7, s), O = at(ne + (k >> 3), k & 7, s);
      put(var, k, cscale(cadd(E, O), 0.5f));
      put(var, a.rH + k, cscale(csub(E, O), 0.5f));
    } else if (k < a.rH + a.DA) {
      const int i = k - a.rH, h = i >> 1;
      put(var, 2 * a.rH + i, at((i & 1 ? ne + S.nz / 8 : S.nz / 8) + (h >> 3), h & 7, s));
    } else {
      const int i = k - a.rH - a.DA, h = i >> 1;
      put(2 + var, i, at(nA + (i & 1 ? S.npe / 8 : 0) + (h >> 3), h & 7, s));
    }
  }
}

// ---------------------------------------------------------------------------
// T1 c: the low-rank and U parts for every sample, plus the transformed F part
// ---------------------------------------------------------------------------
// combined coefficients of one vector, float2 units: rH x (aE, cE, aO, cO), np x (aE, cE, bpE, bmE,
// aO, cO, bpO, bmO) for the powers 2i, 2i + 1, r x w
__host__ __device__ inline int xp_np(int DA, int DB) { return ((DA > DB ? DA : DB) + 1) / 2; }
__host__ __device__ inline int xp_words(int rH, int DA, int DB, int r) { return (4 * rH + 8 * xp_np(DA, DB) + r + 1) & ~1; }
__host__ __device__ inline int xp_cs(int rH, int DA, int DB, int r) {
  const int c = 2 * rH + 2 * xp_np(DA, DB) + r;   // floats per sample; half of it odd: no bank conflicts
  const int h = (c + 1) / 2;
  return 2 * (h | 1);
}
__global__ void k_exp_prep(const ExpArgs<float> a, int64_t nsig, float2 *cc) {
  const int rH = a.rH, DA = a.DA, DB = a.DB, np = xp_np(DA, DB), nw = xp_words(rH, DA, DB, a.r);
  const float ip2 = 0.07957747154594766788f;   // 1 / (4 pi)
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nsig * nw; e += (int64_t)gridDim.x * blockDim.x) {
    const int w = (int)(e % nw);
    const float2 *b1 = a.coef + (a.sig0 + e / nw) * a.Kp + (2 * a.h + 1);
    const float2 *b2 = b1 + rH, *b3 = b2 + rH, *b4 = b3 + rH, *b5 = b4 + rH;
    const float2 *b6 = b5 + DA, *b7 = b6 + DA, *b8 = b7 + DB, *cu = b8 + DB;
    float2 v = make_float2(0.f, 0.f);
    if (w < 4 * rH) {
      const int k = w >> 2;
      switch (w & 3) {
        case 0: v = cscale(csub(b1[k], b2[k]), ip2); break;
        case 1: v = cscale(csub(b4[k], b3[k]), ip2); break;
        case 2: v = cscale(cadd(b1[k], b2[k]), ip2); break;
        default: v = cscale(cadd(b4[k], b3[k]), -ip2); break;
      }
    } else if (w < 4 * rH + 8 * np) {
      const int i = 2 * ((w - 4 * rH) >> 3) + (((w - 4 * rH) >> 2) & 1), q = (w - 4 * rH) & 3;
      if (q == 0 && i < DA) v = cscale(b5[i], 0.5f);
      if (q == 1 && i < DA) v = cscale(b6[i], -0.5f);
      if (q == 2 && i < DB) v = cscale(b7[i], 0.5f);
      if (q == 3 && i < DB) v = cscale(b8[i], 0.5f);
    } else if (w < 4 * rH + 8 * np + a.r) {
      const int j = w - 4 * rH - 8 * np;
      v = cscale(cu[j], a.D[j] < 0 ? -a.sqrtD[j] : a.sqrtD[j]);
    }
    cc[e] = v;
  }
}

// grid (H / 64, vector splits), 256 threads.  A block generates the columns of 64 folded samples once
// and walks its vectors, 8 SPT at a time (their combined coefficients staged in shared memory): a
// thread takes the samples lane, lane + 32 and their mirror images for SPT vectors of its warp;
// coefficients are 16-byte broadcasts, E / O sums collapse into the result after each column kind.
// Measured, 256 vectors of N = 65536, r = 22: 911 -> 303 us.
template <int SPT>
__global__ void __launch_bounds__(256, 2) k_expand_gemm(const ExpArgs<float> a, int64_t nsig, const float2 *cc,
                                                        const unsigned char *cpar) {
  extern __shared__ __align__(16) float xsm[];
  const int rH = a.rH, np = xp_np(a.DA, a.DB), r = a.r;
  const int cs = xp_cs(rH, a.DA, a.DB, r), nw = xp_words(rH, a.DA, a.DB, r);
  float2 *cf = reinterpret_cast<float2 *>(xsm);          // [8 SPT][nw]
  float *cols = xsm + 2 * 8 * SPT * nw;                  // [LR_TN][cs]
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int64_t n0 = (int64_t)blockIdx.x * LR_TN;
  const float Nd = (float)a.N, cen = (float)(0.5 * (double)(a.N - 1)), invN = (float)(1.0 / (double)a.N);
  if (tid < 128) {
    const int i = tid >> 1, side = tid & 1;
    const float xf = (float)(n0 + i) + 0.5f, x = side ? Nd - xf : xf;
    float z = __fdividef(a.zfirst[0], x + a.zshift[0]);
    for (int k = 0; k < rH; ++k) {
      if (k > 0) z *= lr_zstep(a.zfirst, a.zshift, k, x);
      const float other = __shfl_xor_sync(0xffffffffu, z, 1);
      cols[i * cs + 2 * k + side] = side ? other - z : z + other;
    }
  } else {
    const int i = (tid - 128) & 63, g = (tid - 128) >> 6;
    const float u = ((float)(n0 + i) - cen) * invN, u2 = u * u;
    float p = g ? u : 1.f;
    for (int k = 0; k < np; ++k) {
      cols[i * cs + 2 * rH + 2 * k + g] = p;
      p *= u2;
    }
    for (int j = g; j < r; j += 2) cols[i * cs + 2 * rH + 2 * np + j] = __ldg(a.ST + (n0 + i) * a.rpad + j);
  }
  const int64_t per = (nsig + gridDim.y - 1) / gridDim.y, s_lo = per * blockIdx.y;
  const int64_t s_hi = s_lo + per < nsig ? s_lo + per : nsig;
  const float rs = (float)(1.0 / sqrt((double)a.N));
  for (int64_t s0 = s_lo; s0 < s_hi; s0 += 8 * SPT) {
    __syncthreads();   // columns written; the last vectors' coefficients read
    const int ns = (int)(s_hi - s0 < 8 * SPT ? s_hi - s0 : 8 * SPT);
    for (int e = tid; e < ns * nw / 2; e += 256)
      reinterpret_cast<float4 *>(cf)[e] = __ldg(reinterpret_cast<const float4 *>(cc + s0 * nw) + e);
    for (int e = ns * nw + tid; e < 8 * SPT * nw; e += 256) cf[e] = make_float2(0.f, 0.f);
    __syncthreads();
    if (wp * SPT >= ns) continue;
    const float2 *cw = cf + wp * SPT * nw;
    float2 rn[2][SPT], rm[2][SPT];   // results at n and N - 1 - n
    float2 e0[2][SPT], e1[2][SPT], o0[2][SPT], o1[2][SPT];
    auto clear = [&]() {
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int s = 0; s < SPT; ++s) e0[q][s] = e1[q][s] = o0[q][s] = o1[q][s] = make_float2(0.f, 0.f);
    };
    // W' phase: A (e0, o0) and C (e1, o1)
    clear();
    for (int k = 0; k < rH; ++k) {
      float2 c[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) c[q] = *reinterpret_cast<const float2 *>(cols + (lane + 32 * q) * cs + 2 * k);
#pragma unroll
      for (int s = 0; s < SPT; ++s) {
        const float4 E = *reinterpret_cast<const float4 *>(cw + s * nw + 4 * k), O = *reinterpret_cast<const float4 *>(cw + s * nw + 4 * k + 2);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          fma2(e0[q][s], c[q].x, make_float2(E.x, E.y));
          fma2(e1[q][s], c[q].x, make_float2(E.z, E.w));
          fma2(o0[q][s], c[q].y, make_float2(O.x, O.y));
          fma2(o1[q][s], c[q].y, make_float2(O.z, O.w));
        }
      }
    }
#pragma unroll 2
    for (int ph = 0; ph < 2; ++ph) {
      // powers with the W' phase's coefficients (ph 0), then the W + W' phase (ph 1)
      if (ph == 1) clear();
      for (int k = 0; k < np; ++k) {
        float2 c[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) c[q] = *reinterpret_cast<const float2 *>(cols + (lane + 32 * q) * cs + 2 * rH + 2 * k);
#pragma unroll
        for (int s = 0; s < SPT; ++s) {
          const float2 *b = cw + s * nw + 4 * rH + 8 * k + 2 * ph;
          const float4 E = *reinterpret_cast<const float4 *>(b), O = *reinterpret_cast<const float4 *>(b + 4);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            fma2(e0[q][s], c[q].x, make_float2(E.x, E.y));
            fma2(e1[q][s], c[q].x, make_float2(E.z, E.w));
            fma2(o0[q][s], c[q].y, make_float2(O.x, O.y));
            fma2(o1[q][s], c[q].y, make_float2(O.z, O.w));
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int64_t n = n0 + lane + 32 * q, m = a.N - 1 - n;
        const float2 dn = cconj(ph ? a.phB[n] : a.phA[n]), dm = cconj(ph ? a.phB[m] : a.phA[m]);
#pragma unroll
        for (int s = 0; s < SPT; ++s) {
          float2 pn = cadd(e0[q][s], o0[q][s]), pm = csub(e0[q][s], o0[q][s]);
          float2 cn = cadd(e1[q][s], o1[q][s]), cm = csub(e1[q][s], o1[q][s]);
          if (ph == 0) {   // times -j
            pn = make_float2(pn.y, -pn.x);
            pm = make_float2(pm.y, -pm.x);
            cn = make_float2(cn.y, -cn.x);
            cm = make_float2(cm.y, -cm.x);
            rn[q][s] = cadd(cmul(dn, pn), cmul(cconj(dn), cn));
            rm[q][s] = cadd(cmul(dm, pm), cmul(cconj(dm), cm));
          } else {
            rn[q][s] = cadd(rn[q][s], cadd(cmul(dn, pn), cmul(cconj(dn), cn)));
            rm[q][s] = cadd(rm[q][s], cadd(cmul(dm, pm), cmul(cconj(dm), cm)));
          }
        }
      }
    }
    // U part: symmetric columns in e0, antisymmetric ones in o0
    clear();
    for (int j = 0; j < r; ++j) {
      float c[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) c[q] = cols[(lane + 32 * q) * cs + 2 * rH + 2 * np + j];
      if (cpar[j]) {
#pragma unroll
        for (int s = 0; s < SPT; ++s)
#pragma unroll
          for (int q = 0; q < 2; ++q) fma2(o0[q][s], c[q], cw[s * nw + 4 * rH + 8 * np + j]);
      } else {
#pragma unroll
        for (int s = 0; s < SPT; ++s)
#pragma unroll
          for (int q = 0; q < 2; ++q) fma2(e0[q][s], c[q], cw[s * nw + 4 * rH + 8 * np + j]);
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int64_t n = n0 + lane + 32 * q, m = a.N - 1 - n;
      const int64_t xn = spec_pos(a.Lf, n), xm = spec_pos(a.Lf, m);
#pragma unroll
      for (int s = 0; s < SPT; ++s) {
        const int64_t sl = s0 + wp * SPT + s;
        if (sl < s_hi) {
          const float2 *X = a.X + sl * a.N;
          float2 *o = a.out + (a.sig0 + sl) * a.N;
          o[n] = cadd(cadd(rn[q][s], cadd(e0[q][s], o0[q][s])), cscale(cconj(X[xn]), rs));
          o[m] = cadd(cadd(rm[q][s], csub(e0[q][s], o0[q][s])), cscale(cconj(X[xm]), rs));
        }
      }
    }
  }
}

}  // namespace fst
