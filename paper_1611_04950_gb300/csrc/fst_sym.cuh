// fst_sym.cuh -- rank-r correction of an FP32 batch on the folded half of S_T (device only).
//
// Every Slepian vector is symmetric or antisymmetric, s_l(N-1-n) = (-1)^l s_l(n), so with H = ceil(N/2)
//   (S_T^T y)_j = sum_{n<H} s_j(n) (y(n) +- y(N-1-n))          (the middle sample of an odd N once)
//   (S_T a)(n) = z+ + z-,  (S_T a)(N-1-n) = z+ - z-,  z+- = sums over the (anti)symmetric columns
// which halves the FMAs and the S_T traffic of the unfolded forms.  Columns are read from the K-major
// copy S_T^T (rows of Npad floats, 16-byte aligned) in the order `cord`: symmetric ones first.
// A row is a real signal, or the real or imaginary part of a complex one (row / 2, row & 1).
#pragma once
#include "fst_fast.cuh"

namespace fst {

constexpr int SY_TN = 64, SY_LD = SY_TN + 4;
__host__ __device__ inline int sy_rows(int64_t rows) {   // rows per block of S_T^T y: 8, 16 or 32
  int b = 8;
  while (b < 32 && b < rows) b *= 2;
  return b;
}
__host__ __device__ inline int sy_tiles(int nE, int nO) { return (nE + 7) / 8 + (nO + 7) / 8; }
__host__ __device__ inline size_t sy_smem(int nE, int nO, int RB) {
  const int ct = sy_tiles(nE, nO), ntile = ct * (RB / 8), kg = ntile < 16 ? 16 : 256 / ntile;
  const size_t tile = (size_t)(2 * ct * 8 + 2 * RB) * SY_LD, sums = (size_t)kg * ntile * 64;
  return (tile > sums ? tile : sums) * 4;
}

// ---------------------------------------------------------------------------
// S_T^T y partials: grid (chunks, row groups of RB), 256 threads, dynamic sy_smem.  Per tile of 64
// folded samples the S columns (cp.async) and the folded rows y(n) + y(N-1-n), y(n) - y(N-1-n) lie in
// shared memory along the samples; the next tile's columns (second buffer) and rows (registers) are
// loaded while the current one is multiplied.  Thread (column tile, row tile, sample group) accumulates 8 x 8 sums,
// 16 16-byte loads per 256 FMAs (its columns and rows are ct + k nct and vt + k nvt: neighbouring
// threads read neighbouring 16-byte pieces).  Sample groups are added in fixed chains at the end; one partial
// per (row, chunk), the layout k_corr_reduce reads.
// QUAD: the four products of a step are added among themselves first, a quarter of the roundings at the
// size of the sum for a fifth FP32 instruction per four.  For chains of more than 64 products in blocks of 8
// rows, which wait for memory anyway: error of U2^* y against FP64 of one row of 2^21 samples 2.9e-7 -> 1.8e-7,
// of 8 rows 2.8e-7 -> 1.8e-7 (the 2048-sample blocks before this kernel 2.4e-7, 2.1e-7), same time; blocks of
// 32 rows would take 350 -> 487 us (64 complex signals of 2^20), and their errors are below those of the
// tensor cores' sums without it.
// Bound: FP32 FMA against the HBM reads of y and of half of S_T.  Measured (us, unfolded -> folded): 16 real
// signals of 2^22, r = 60: 366 -> 242; 64 complex ones of 2^20, r = 38: 246 (tcgen05, alone on the
// chip) -> 335, but the whole call 2075 -> 1997, since these blocks run beside the column passes.
// ---------------------------------------------------------------------------
template <bool CPLX, int RB, bool QUAD = false>
__global__ void __launch_bounds__(256, 2) k_sym_c(const ConvArgs<float> a, const int *cord, int nE, int nchunk) {
  extern __shared__ __align__(16) float ysm[];
  constexpr int nvt = RB / 8, RT = RB / 4;   // rows a thread loads (complex: RT / 2 signals)
  const int tid = threadIdx.x, nO = a.r - nE, tE = (nE + 7) / 8, tO = (nO + 7) / 8, nct = tE + tO;
  const int ntile = nct * nvt, kg = ntile < 16 ? 16 : 256 / ntile;
  float *S = ysm, *Vp = S + 2 * nct * 8 * SY_LD, *Vm = Vp + RB * SY_LD;
  const int64_t H = (a.N + 1) / 2, rows = CPLX ? 2 * a.batch : a.batch, row0 = (int64_t)blockIdx.y * RB;
  const int nr = (int)(rows - row0 < RB ? rows - row0 : RB);
  const int id = tid % ntile, kgi = tid / ntile, vt = id % nvt, ct = id / nvt;
  const bool on = kgi < kg;
  const int cst = (ct < tE ? tE : tO) * SY_LD;                // stride of this thread's columns
  const float *cp = S + (ct < tE ? ct : tE * 8 + (ct - tE)) * SY_LD;
  const float *vp = (ct < tE ? Vp : Vm) + vt * SY_LD;
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[i][q] = 0.f;
  const int64_t ntl = (H + SY_TN - 1) / SY_TN;
  const int64_t t0 = ntl * blockIdx.x / nchunk, t1 = ntl * (blockIdx.x + 1) / nchunk;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(S);
  const int i = tid & 63, r0 = tid >> 6;
  float u[RT], w[RT];
  auto fetch = [&](int64_t t, int buf) {
    const int64_t n0 = t * SY_TN, n = n0 + i, m = a.N - 1 - n;
    if (!CPLX) {
      const float *yn = a.y + (row0 + r0) * a.ld + n, *ym = a.y + (row0 + r0) * a.ld + m;
#pragma unroll
      for (int q = 0; q < RT; ++q) {
        const bool in = r0 + 4 * q < nr && n < H;
        u[q] = in ? __ldg(yn + 4 * q * a.ld) : 0.f;
        w[q] = in && m != n ? __ldg(ym + 4 * q * a.ld) : 0.f;
      }
    } else {
      const float2 *y2 = reinterpret_cast<const float2 *>(a.y) + ((row0 >> 1) + r0) * a.ld, z = make_float2(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < RT / 2; ++q) {
        const bool in = 2 * (r0 + 4 * q) < nr && n < H;
        const float2 x = in ? __ldg(y2 + 4 * q * a.ld + n) : z, v = in && m != n ? __ldg(y2 + 4 * q * a.ld + m) : z;
        u[2 * q] = x.x;
        u[2 * q + 1] = x.y;
        w[2 * q] = v.x;
        w[2 * q + 1] = v.y;
      }
    }
    const uint32_t sb = sbase + (uint32_t)(buf * nct * 8 * SY_LD * 4);
    for (int e = tid; e < nct * 8 * (SY_TN / 4); e += 256) {
      const int c = e / (SY_TN / 4), q = e % (SY_TN / 4);
      const bool odd = c >= tE * 8;
      const int o = odd ? c - tE * 8 + nE : c;               // position in cord (padding columns: zero)
      const bool ok = odd ? o < a.r : o < nE;
      cp_async16(sb + (uint32_t)((c * SY_LD + 4 * q) * 4),
                 ok ? a.STt + (int64_t)__ldg(cord + o) * a.tc_Npad + n0 + 4 * q : a.STt, ok ? 16 : 0);
    }
    cp_async_commit();
  };
  if (t0 < t1) fetch(t0, 0);
  for (int64_t t = t0; t < t1; ++t) {
    const int buf = (int)((t - t0) & 1);
    __syncthreads();   // the rows and the other column buffer are free
#pragma unroll
    for (int q = 0; q < RT; ++q) {
      const int row = CPLX ? 2 * (r0 + 4 * (q >> 1)) + (q & 1) : r0 + 4 * q;
      Vp[row * SY_LD + i] = u[q] + w[q];
      Vm[row * SY_LD + i] = u[q] - w[q];
    }
    cp_async_wait0();
    __syncthreads();
    if (t + 1 < t1) fetch(t + 1, buf ^ 1);
    if (on) {
      const float *cb = cp + buf * nct * 8 * SY_LD;
      for (int g = kgi; g < SY_TN / 4; g += kg) {
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = *reinterpret_cast<const float4 *>(vp + q * nvt * SY_LD + 4 * g);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float4 s = *reinterpret_cast<const float4 *>(cb + c * cst + 4 * g);
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (QUAD) acc[c][q] += fmaf(s.w, v[q].w, fmaf(s.z, v[q].z, fmaf(s.y, v[q].y, s.x * v[q].x)));
            else acc[c][q] = fmaf(s.w, v[q].w, fmaf(s.z, v[q].z, fmaf(s.y, v[q].y, fmaf(s.x, v[q].x, acc[c][q]))));
        }
      }
    }
  }
  __syncthreads();
  float *red = ysm;   // [kg][tile][8 columns][8 rows]
  if (on) {
#pragma unroll
    for (int c = 0; c < 8; ++c)
#pragma unroll
      for (int q = 0; q < 8; ++q) red[(kgi * ntile + id) * 64 + c * 8 + q] = acc[c][q];
  }
  __syncthreads();
  for (int e = tid; e < ntile * 64; e += 256) {
    const int tl = e >> 6, c = (e >> 3) & 7, q = e & 7, tct = tl / nvt, tvt = tl % nvt;
    const bool odd = tct >= tE;
    const int o = odd ? nE + (tct - tE) + c * tO : tct + c * tE;
    const int row = tvt + q * nvt;
    if ((odd ? o < a.r : o < nE) && row < nr) {
      // four chains, a quarter of the roundings in a row (32 rows have few groups: one chain, whose main
      // loop also compiles to the faster code, 350 instead of 367 us for 64 complex signals of 2^20)
      float sum = red[e];
      if (RB < 32) {
        float s[4] = {sum, 0.f, 0.f, 0.f};
        for (int k0 = 1; k0 < kg; k0 += 4) {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (k0 + i < kg) s[(i + 1) & 3] += red[(k0 + i) * ntile * 64 + e];
        }
        sum = (s[0] + s[1]) + (s[2] + s[3]);
      } else {
        for (int k = 1; k < kg; ++k) sum += red[k * ntile * 64 + e];
      }
      const int64_t rw = row0 + row;
      a.part[(((rw >> 1) * nchunk + blockIdx.x) * 2 + (rw & 1)) * a.rpad + __ldg(cord + o)] = sum;
    }
  }
}

// ---------------------------------------------------------------------------
// out += S_T a: grid (ceil(H / TN), row groups), 256 threads (64 where that leaves SMs idle).  A block takes 8 ng rows (ng = row groups
// of 8, a power of two up to 16) and TN = 4 threads / ng folded samples; thread (4 consecutive samples, 8
// rows) keeps z+ and z- of its samples and rows.  Per column one 16-byte load of S_T^T (coalesced; the
// row groups of a block share it through L1) and two 16-byte broadcasts of a feed 16 packed FMAs.
// VEC: 16-byte accesses of out (N, ld and the base allow them), else one by one.
// Bound: HBM (out read and written, half of S_T read).  Measured (us, unfolded -> folded):
// 64 complex signals of 2^20, r = 38: 628 -> 438; 16 real ones of 2^22, r = 60: 613 -> 287.
// ---------------------------------------------------------------------------
constexpr int SY_R = 8;   // rows per thread (4: 504 instead of 438 us, 351 instead of 287)
__host__ __device__ inline int sy_ng(int64_t rows) {
  int g = 1;
  while (g < 16 && (int64_t)g * SY_R < rows) g *= 2;
  return g;
}
template <bool VEC> __global__ void __launch_bounds__(256, 2) k_sym_z(const ConvArgs<float> a, const int *cord, int nE) {
  extern __shared__ __align__(16) float zsy[];   // a, [column in cord order][SY_R ng], then the column offsets
  const int64_t rows = a.cplx ? 2 * a.batch : a.batch, H = (a.N + 1) / 2;
  const int nthr = blockDim.x, ng = sy_ng(rows), RB = SY_R * ng, ns = nthr / ng;
  const int64_t row0 = (int64_t)blockIdx.y * RB;
  int *co = reinterpret_cast<int *>(zsy + a.r * RB);
  const int i = threadIdx.x % ns, g = threadIdx.x / ns;
  const int64_t n = ((int64_t)blockIdx.x * ns + i) * 4, m3 = a.N - 4 - n;   // m3: the mirror images of n + 3, ..., n
  const int nr = (int)(rows - row0 - SY_R * g < SY_R ? rows - row0 - SY_R * g : SY_R);
  const bool live = n < H && nr > 0;
  // row (or complex signal) q of this thread, in floats; both ends are on their way from memory while
  // the sums are formed
  const int64_t es = a.cplx ? 2 : 1;
  float *o0 = a.out + (a.cplx ? (row0 + SY_R * g) / 2 : row0 + SY_R * g) * a.ld * es;
  const int no = a.cplx ? (nr + 1) / 2 : nr;
  if (live) {
    for (int q = 0; q < no; ++q) {
      asm volatile("prefetch.global.L2 [%0];" ::"l"(o0 + q * a.ld * es + n * es));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(o0 + q * a.ld * es + (m3 > 0 ? m3 : 0) * es));
    }
  }
  for (int e = threadIdx.x; e < a.r; e += nthr) co[e] = __ldg(cord + e);
  for (int e = threadIdx.x; e < a.r * RB; e += nthr) {
    const int o = e / RB, q = e % RB;
    zsy[e] = row0 + q < rows ? a.acoef[(row0 + q) * a.rpad + __ldg(cord + o)] : 0.f;
  }
  __syncthreads();
  if (!live) return;
  float2 zp[4][SY_R / 2], zm[4][SY_R / 2];   // [sample][row pair]
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int q = 0; q < SY_R / 2; ++q) zp[s][q] = zm[s][q] = make_float2(0.f, 0.f);
  const float *st = a.STt + n, *as = zsy + SY_R * g;
  auto add = [&](int o, float2 (&z)[4][SY_R / 2]) {
    const float4 s = __ldg(reinterpret_cast<const float4 *>(st + (int64_t)co[o] * a.tc_Npad));
    const float4 w0 = *reinterpret_cast<const float4 *>(as + o * RB), w1 = *reinterpret_cast<const float4 *>(as + o * RB + 4);
    const float sv[4] = {s.x, s.y, s.z, s.w};
    const float2 w[SY_R / 2] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y), make_float2(w1.z, w1.w)};
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int q = 0; q < SY_R / 2; ++q) z[k][q] = __ffma2_rn(make_float2(sv[k], sv[k]), w[q], z[k][q]);
  };
#pragma unroll 8
  for (int o = 0; o < nE; ++o) add(o, zp);
#pragma unroll 8
  for (int o = nE; o < a.r; ++o) add(o, zm);
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int q = 0; q < SY_R / 2; ++q) {   // zp: at n + k, zm: at its mirror image
      const float2 p = cadd(zp[k][q], zm[k][q]);
      zm[k][q] = csub(zp[k][q], zm[k][q]);
      zp[k][q] = p;
    }
  auto vec4 = [](float *p) { return *reinterpret_cast<float4 *>(p); };
  if (VEC && n + 4 <= H && m3 >= n + 4) {
    // loads of four rows (two complex signals) before their stores
    if (!a.cplx) {
#pragma unroll
      for (int h = 0; h < SY_R / 4; ++h) {
        float4 v[4], w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (4 * h + q < nr) {
            v[q] = vec4(o0 + (4 * h + q) * a.ld + n);
            w[q] = vec4(o0 + (4 * h + q) * a.ld + m3);
          }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (4 * h + q < nr) {
            const int pr = 2 * h + (q >> 1);
            auto c = [&](float2 x) { return (q & 1) ? x.y : x.x; };
            v[q].x += c(zp[0][pr]); v[q].y += c(zp[1][pr]); v[q].z += c(zp[2][pr]); v[q].w += c(zp[3][pr]);
            w[q].x += c(zm[3][pr]); w[q].y += c(zm[2][pr]); w[q].z += c(zm[1][pr]); w[q].w += c(zm[0][pr]);
            *reinterpret_cast<float4 *>(o0 + (4 * h + q) * a.ld + n) = v[q];
            *reinterpret_cast<float4 *>(o0 + (4 * h + q) * a.ld + m3) = w[q];
          }
      }
    } else {
#pragma unroll
      for (int h = 0; h < SY_R / 4; ++h) {
        float4 v[2][2], w[2][2];
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (2 * h + q < no) {
            float *o = o0 + (2 * h + q) * a.ld * 2;
            v[q][0] = vec4(o + 2 * n);
            v[q][1] = vec4(o + 2 * n + 4);
            w[q][0] = vec4(o + 2 * m3);
            w[q][1] = vec4(o + 2 * m3 + 4);
          }
#pragma unroll
        for (int q = 0; q < 2; ++q)
          if (2 * h + q < no) {
            float *o = o0 + (2 * h + q) * a.ld * 2;
            const int pr = 2 * h + q;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              v[q][k].x += zp[2 * k][pr].x; v[q][k].y += zp[2 * k][pr].y;
              v[q][k].z += zp[2 * k + 1][pr].x; v[q][k].w += zp[2 * k + 1][pr].y;
              w[q][k].x += zm[3 - 2 * k][pr].x; w[q][k].y += zm[3 - 2 * k][pr].y;
              w[q][k].z += zm[2 - 2 * k][pr].x; w[q][k].w += zm[2 - 2 * k][pr].y;
              *reinterpret_cast<float4 *>(o + 2 * n + 4 * k) = v[q][k];
              *reinterpret_cast<float4 *>(o + 2 * m3 + 4 * k) = w[q][k];
            }
          }
      }
    }
    return;
  }
  // sample by sample: the loads of four rows (two complex signals) before their stores
  if (a.cplx) {
#pragma unroll
    for (int h = 0; h < SY_R / 4; ++h) {
      float2 v[2][4], w[2][4];
      auto sig = [&](int q) { return reinterpret_cast<float2 *>(o0) + q * a.ld; };
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (2 * h + q < no && n + k < H) {
            v[q][k] = sig(2 * h + q)[n + k];
            w[q][k] = sig(2 * h + q)[a.N - 1 - n - k];
          }
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (2 * h + q < no && n + k < H) {
            sig(2 * h + q)[n + k] = cadd(v[q][k], zp[k][2 * h + q]);
            if (a.N - 1 - n - k != n + k) sig(2 * h + q)[a.N - 1 - n - k] = cadd(w[q][k], zm[k][2 * h + q]);
          }
    }
    return;
  }
#pragma unroll
  for (int h = 0; h < SY_R / 4; ++h) {
    float v[4][4], w[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * h + q < nr)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (n + k < H) {
            v[q][k] = o0[(4 * h + q) * a.ld + n + k];
            w[q][k] = o0[(4 * h + q) * a.ld + a.N - 1 - n - k];
          }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (4 * h + q < nr)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (n + k < H) {
            const int pr = 2 * h + (q >> 1);
            const int64_t m = a.N - 1 - n - k;
            o0[(4 * h + q) * a.ld + n + k] = v[q][k] + ((q & 1) ? zp[k][pr].y : zp[k][pr].x);
            if (m != n + k) o0[(4 * h + q) * a.ld + m] = w[q][k] + ((q & 1) ? zm[k][pr].y : zm[k][pr].x);
          }
  }
}

}  // namespace fst
