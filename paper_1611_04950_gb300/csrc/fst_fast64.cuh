// fst_fast64.cuh -- FP64 projection kernels for 2^10 <= M <= 2^18 (device only).
//
// Same four-step decomposition as fst_kernels.cuh (n = n1 Q + n2, k = k1 + P k2), built for the
// FP64 unit of this part, which is the only bound here: an FP64 instruction holds its warp 64
// clocks, four warps per SM run side by side (1.7 lanes a clock per SM), everything else is
// hidden.  So what counts is the number of FP64 instructions and how evenly they spread over
// the SMs:
//   * radix-4 stages with 4 values per thread: as few FP64 instructions per level as radix 16
//     (7 per two levels and value) with four times the threads, so one short signal pair fills
//     64 SMs instead of one;
//   * stage twiddles are read from the table, not formed by products;
//   * the zero half of the padded columns (rows n1 >= P/2) costs nothing: the first radix-2 stage
//     of pass A is a copy, the last one of pass C forms only the rows that hold output;
//   * the rank-r correction runs outside the column passes on half of S_T: every Slepian vector
//     is symmetric or antisymmetric, s_l(N-1-n) = (-1)^l s_l(n), so the FMAs of S_T^T y and of
//     S_T a halve.
// Measured (us, before -> after): one pair of N = 4096 479 -> 40; 64 signals of N = 40000,
// r = 32, 1977 -> 1275.
#pragma once
#include "fst_kernels.cuh"

namespace fst {

struct F64Args {
  ConvArgs<double> a;
  int spec_log2P;     // the spectrum's own split: frequency k at [k mod P][k div P] (0: natural order)
  int log2NB;         // columns per tile of the column passes
  int log2RT;         // rows per block of the row pass
};

// One Stockham stage of radix R (2 or 4) at sub-length Ns = 2^ls over 2^lc transforms of length
// L = 2^ll in buf (element i of column c at (i << lc) + c), 2^(lc + ll) / R butterflies, up to PER
// per thread.  HALF (radix 2, last stage): only the first output of each butterfly is formed.
template <int R, bool INV, int PER, bool HALF>
__device__ __forceinline__ void f64_stage(double2 *buf, int ll, int ls, int lc, const Tw<double> &tw) {
  constexpr int LR = R == 4 ? 2 : 1;
  const int nthr = blockDim.x, nb = 1 << (lc + ll - LR), stride = 1 << (ll - LR);
  double2 v[PER][R];
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int b = threadIdx.x + q * nthr;
    if (b < nb) {
      const int c = b & ((1 << lc) - 1), j = b >> lc, k = j & ((1 << ls) - 1);
#pragma unroll
      for (int t = 0; t < R; ++t) v[q][t] = buf[((j + t * stride) << lc) + c];
      if (ls > 0) {
#pragma unroll
        for (int t = 1; t < R; ++t) v[q][t] = cmul(v[q][t], tw.root_s<INV>((uint32_t)(k * t), ls + LR));
      }
      if (HALF) v[q][0] = cadd(v[q][0], v[q][1]);
      else Dft<double, R, INV>::run(v[q]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < PER; ++q) {
    const int b = threadIdx.x + q * nthr;
    if (b < nb) {
      const int c = b & ((1 << lc) - 1), j = b >> lc, k = j & ((1 << ls) - 1);
      const int d0 = ((j >> ls) << (ls + LR)) + k;
      if (HALF) {
        buf[(d0 << lc) + c] = v[q][0];
      } else {
#pragma unroll
        for (int t = 0; t < R; ++t) buf[((d0 + (t << ls)) << lc) + c] = v[q][t];
      }
    }
  }
  __syncthreads();
}

// stages from sub-length 2^ls to 2^le (a radix-2 one first when their distance is odd)
template <bool INV, int PER>
__device__ __forceinline__ void f64_stages(double2 *buf, int ll, int ls, int le, int lc, const Tw<double> &tw) {
  if ((le - ls) & 1) {
    f64_stage<2, INV, 2 * PER, false>(buf, ll, ls, lc, tw);
    ++ls;
  }
  for (; ls < le; ls += 2) f64_stage<4, INV, PER, false>(buf, ll, ls, lc, tw);
}

// ---- pass A: a tile of NB columns of one pair, all P rows; blockDim.x = P NB / 4 ----------------
__global__ void __launch_bounds__(512) k_f64A(const F64Args f) {
  extern __shared__ __align__(16) double2 dsm[];
  const ConvArgs<double> &a = f.a;
  const int P = 1 << a.log2P, Q = 1 << a.log2Q, lc = f.log2NB, NB = 1 << lc;
  const int64_t pl = blockIdx.x >> (a.log2Q - lc), n2_0 = (int64_t)(blockIdx.x & ((Q >> lc) - 1)) << lc;
  // the first radix-2 stage: rows n1 >= P/2 are zero, so both outputs are the input itself
  for (int e = threadIdx.x; e < P / 2 * NB; e += blockDim.x) {
    const int j = e >> lc, c = e & (NB - 1);
    const int64_t n = (int64_t)j * Q + n2_0 + c;
    const double2 v = (j < a.Pnz && n < a.N) ? load_pair(a, pl, n) : make_double2(0.0, 0.0);
    dsm[((2 * j) << lc) + c] = v;
    dsm[((2 * j + 1) << lc) + c] = v;
  }
  __syncthreads();
  f64_stages<false, 1>(dsm, a.log2P, 1, a.log2P, lc, a.tw);
  double2 *dst = a.inter + (pl * P) * (int64_t)Q + n2_0;
  for (int e = threadIdx.x; e < P * NB; e += blockDim.x) {
    const int k1 = e >> lc, c = e & (NB - 1);
    const double2 v = dsm[e];
    dst[(int64_t)k1 * Q + c] =
        k1 == 0 ? v : cmul(v, a.tw.root_s<false>((uint32_t)((n2_0 + c) * k1) & ((1u << a.log2M) - 1), a.log2M));
  }
}

// ---- pass B for rows of up to 1024 points (longer ones: k_passB, whose 16 values per thread leave
// fewer barriers and already keep four warps per row): RT rows: forward DFT, spectrum, inverse DFT,
// twiddle; blockDim.x = RT Q / 4 ---------------------------------------------------------------------
__global__ void __launch_bounds__(512) k_f64B(const F64Args f) {
  extern __shared__ __align__(16) double2 dsm[];
  const ConvArgs<double> &a = f.a;
  const int P = 1 << a.log2P, Q = 1 << a.log2Q, lr = f.log2RT, RT = 1 << lr;
  const int64_t row0 = (int64_t)blockIdx.x << lr;   // row pl P + k1 of the launch group; RT divides P
  double2 *src = a.inter + row0 * Q;
  const int k1_0 = (int)(row0 & (P - 1));
  for (int e = threadIdx.x; e < RT * Q; e += blockDim.x) dsm[((e & (Q - 1)) << lr) + (e >> a.log2Q)] = src[e];
  __syncthreads();
  f64_stages<false, 1>(dsm, a.log2Q, 0, a.log2Q, lr, a.tw);
  for (int e = threadIdx.x; e < RT * Q; e += blockDim.x) {
    const int k = k1_0 + (e & (RT - 1)) + P * (e >> lr);
    const double s = __ldg(a.spec + ((k & ((1 << f.spec_log2P) - 1)) << (a.log2M - f.spec_log2P)) + (k >> f.spec_log2P));
    dsm[e] = cscale(dsm[e], s);
  }
  __syncthreads();
  f64_stages<true, 1>(dsm, a.log2Q, 0, a.log2Q, lr, a.tw);
  for (int e = threadIdx.x; e < RT * Q; e += blockDim.x) {
    const int n2 = e & (Q - 1), rr = e >> a.log2Q, k1 = k1_0 + rr;
    const double2 v = dsm[(n2 << lr) + rr];
    src[e] = k1 == 0 ? v : cmul(v, a.tw.root_s<true>((uint32_t)(n2 * k1) & ((1u << a.log2M) - 1), a.log2M));
  }
}

// ---- pass C: inverse DFTs of a tile's columns, rows n1 < P/2, first N samples; blockDim.x = P NB / 4
__global__ void __launch_bounds__(512) k_f64C(const F64Args f) {
  extern __shared__ __align__(16) double2 dsm[];
  const ConvArgs<double> &a = f.a;
  const int P = 1 << a.log2P, Q = 1 << a.log2Q, lc = f.log2NB, NB = 1 << lc;
  const int64_t pl = blockIdx.x >> (a.log2Q - lc), n2_0 = (int64_t)(blockIdx.x & ((Q >> lc) - 1)) << lc;
  const double2 *src = a.inter + (pl * P) * (int64_t)Q + n2_0;
  for (int e = threadIdx.x; e < P * NB; e += blockDim.x) dsm[e] = src[(int64_t)(e >> lc) * Q + (e & (NB - 1))];
  __syncthreads();
  f64_stages<true, 1>(dsm, a.log2P, 0, a.log2P - 1, lc, a.tw);
  f64_stage<2, true, 2, true>(dsm, a.log2P, a.log2P - 1, lc, a.tw);
  for (int e = threadIdx.x; e < P / 2 * NB; e += blockDim.x) {
    const int n1 = e >> lc;
    const int64_t n = (int64_t)n1 * Q + n2_0 + (e & (NB - 1));
    if (n1 < a.Pnz && n < a.N) store_pair(a, pl, n, dsm[e]);
  }
}

// ---- rank-r correction on the folded half of the samples, n < H = ceil(N/2) ---------------------
// A row is a real signal, or the real or imaginary part of a complex one (row / 2, row & 1); row b
// of the coefficients is row b of acoef ([pair][2][rpad]).  cpar[j] = 1: column j antisymmetric.
__device__ __forceinline__ int64_t f64_elem(const ConvArgs<double> &a, int64_t row, int64_t n) {
  return a.cplx ? 2 * ((row >> 1) * a.ld + n) + (row & 1) : row * a.ld + n;
}

// c partials: block (chunk of ch folded samples, RG rows), 256 threads.  Thread (slice, row, j) sums
// s_j(n) (y(n) +- y(N-1-n)) over the samples of its slice; the slices are added in order.  The folded
// rows and S_T rows pass through shared memory 32 samples at a time.  64 columns a round, and of the
// rows as many as 256 threads take; the number of slices goes by the rows of the whole call, so every
// row adds in the same order wherever it lies in its block.
// part: [chunk][row][rpad]
constexpr int F64_RG = 8, F64_SUB = 32, F64_JB = 64;
__global__ void __launch_bounds__(256) k_f64_corr(const ConvArgs<double> a, const unsigned char *cpar, int ch,
                                                  int64_t rows, double *part) {
  __shared__ double yp[F64_SUB][F64_RG], ym[F64_SUB][F64_RG], st[F64_SUB][F64_JB], red[256];
  const int64_t H = (a.N + 1) / 2, n0 = (int64_t)blockIdx.x * ch;
  const int64_t n1 = n0 + ch < H ? n0 + ch : H;
  const int64_t row0 = (int64_t)blockIdx.y * F64_RG;
  const int nr = (int)(rows - row0 < F64_RG ? rows - row0 : F64_RG);
  for (int j0 = 0; j0 < a.r; j0 += F64_JB) {
    const int nj = a.r - j0 < F64_JB ? a.r - j0 : F64_JB;
    const int rg = (int)(a.rows_all < F64_RG ? a.rows_all : F64_RG);
    const int rpr = rg * nj <= 256 ? rg : (rg + 1) / 2;   // rows a round
    const int no = rpr * nj, nsl = 256 / no;
    for (int q0 = 0; q0 < nr; q0 += rpr) {
      const int o = threadIdx.x % no, sl = threadIdx.x / no;
      const int rr = q0 + o / nj, j = o % nj;
      const bool on = sl < nsl && rr < nr, odd = on && cpar[j0 + j];
      double acc = 0.0;
      for (int64_t m0 = n0; m0 < n1; m0 += F64_SUB) {
        const int ns = (int)(n1 - m0 < F64_SUB ? n1 - m0 : F64_SUB);
        __syncthreads();
        for (int e = threadIdx.x; e < ns * nr; e += 256) {
          // real rows: samples along the threads; complex: the two parts of a sample side by side
          const int i = a.cplx ? (e / 2) % ns : e % ns, q = a.cplx ? 2 * (e / (2 * ns)) + (e & 1) : e / ns;
          const int64_t n = m0 + i, m = a.N - 1 - n;
          const double u = a.y[f64_elem(a, row0 + q, n)], w = m != n ? a.y[f64_elem(a, row0 + q, m)] : 0.0;
          yp[i][q] = u + w;
          ym[i][q] = u - w;
        }
        for (int e = threadIdx.x; e < ns * nj; e += 256) st[e / nj][e % nj] = __ldg(a.ST + (m0 + e / nj) * a.rpad + j0 + e % nj);
        __syncthreads();
        if (on)
          for (int i = sl; i < ns; i += nsl) acc = fma(st[i][j], odd ? ym[i][rr] : yp[i][rr], acc);
      }
      __syncthreads();
      red[threadIdx.x] = acc;
      __syncthreads();
      if (threadIdx.x < no && rr < nr) {
        double s = acc;
        for (int q = 1; q < nsl; ++q) s += red[q * no + threadIdx.x];
        part[((int64_t)blockIdx.x * rows + row0 + rr) * a.rpad + j0 + j] = s;
      }
    }
  }
}

// a[row][j] = D_j * (sum of the partials): a warp per (row, j), lanes over the chunks, fixed order
__global__ void __launch_bounds__(256) k_f64_reduce(const ConvArgs<double> a, int nchunk, int64_t rows,
                                                    const double *part, double *acoef) {
  const int64_t t = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (t >= rows * a.r) return;
  const int64_t row = t / a.r;
  const int j = (int)(t % a.r);
  double s = 0.0;
  for (int c = lane; c < nchunk; c += 32) s += part[((int64_t)c * rows + row) * a.rpad + j];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) acoef[row * a.rpad + j] = __ldg(a.D + j) * s;
}

// out(n), out(N-1-n) += S_T a: block of 64 folded samples x 4 rows, a thread per (sample, row):
// z+- over the (anti)symmetric columns, z(n) = z+ + z-, z(N-1-n) = z+ - z-
constexpr int F64_ZN = 64, F64_ZR = 4;
__global__ void __launch_bounds__(F64_ZN *F64_ZR) k_f64_z(const ConvArgs<double> a, const unsigned char *cpar,
                                                          int64_t rows, const double *acoef) {
  __shared__ double st[F64_ZN][F64_SUB + 1], as[F64_ZR][F64_SUB];
  const int64_t H = (a.N + 1) / 2, n0 = (int64_t)blockIdx.x * F64_ZN;
  const int64_t row0 = (int64_t)blockIdx.y * F64_ZR;
  const int i = threadIdx.x % F64_ZN, q = threadIdx.x / F64_ZN;
  const int64_t n = n0 + i, row = row0 + q;
  double zp = 0.0, zm = 0.0;
  for (int j0 = 0; j0 < a.r; j0 += F64_SUB) {
    const int nj = a.r - j0 < F64_SUB ? a.r - j0 : F64_SUB;
    __syncthreads();
    const int jl = threadIdx.x & 31, e0 = threadIdx.x >> 5;
    for (int e = e0; e < F64_ZN; e += F64_ZN * F64_ZR / 32)
      st[e][jl] = (n0 + e < H && jl < nj) ? __ldg(a.ST + (n0 + e) * a.rpad + j0 + jl) : 0.0;
    if (e0 < F64_ZR) as[e0][jl] = (row0 + e0 < rows && jl < nj) ? acoef[(row0 + e0) * a.rpad + j0 + jl] : 0.0;
    // the round's columns as bits, symmetric ones first (a choice of the sum inside one loop is
    // compiled into both FMAs: twice the FP64 time)
    const int lane = threadIdx.x & 31;
    const unsigned anti = __ballot_sync(0xffffffffu, lane < nj && cpar[j0 + lane]);
    const unsigned all = nj == 32 ? 0xffffffffu : (1u << nj) - 1u;
    __syncthreads();
    for (unsigned m = all & ~anti; m; m &= m - 1) zp = fma(st[i][__ffs(m) - 1], as[q][__ffs(m) - 1], zp);
    for (unsigned m = anti; m; m &= m - 1) zm = fma(st[i][__ffs(m) - 1], as[q][__ffs(m) - 1], zm);
  }
  if (n >= H || row >= rows) return;
  const int64_t m = a.N - 1 - n, en = f64_elem(a, row, n), em = f64_elem(a, row, m);
  a.out[en] += zp + zm;
  if (m != n) a.out[em] += zp - zm;
}

}  // namespace fst
