// fst_device.cu -- CUDA back-end of the fast Slepian projection library (sm_103a):
// the __global__ wrappers of the kernel bodies, the device Runner, and the
// host-buffer entry point with overlapped copies.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <string>
#include <vector>

#include "fst_internal.h"
#include "../../include/fst_testing.h"
#include "fst_fast.cuh"
#include "fst_big.cuh"
#include "fst_fast64.cuh"
#include "fst_small32.cuh"
#include "fst_lowrank.cuh"
#include "fst_sym.cuh"
#define FST_TC_KERNELS
#include "fst_tc.cuh"

namespace fst {

template <typename T> struct DevEx {
  using State = KState<T>;
  int nthr;
  int tid;
  State st;
  __device__ DevEx() : nthr(blockDim.x), tid(threadIdx.x) {}
  template <typename F> __device__ __forceinline__ void phase(F &&f) {
    f(tid, st);
    __syncthreads();
  }
};

struct NoState {
  int top;
};
struct DevExPlan {
  using State = NoState;
  int nthr;
  int tid;
  State st;
  __device__ DevExPlan() : nthr(blockDim.x), tid(threadIdx.x) {}
  template <typename F> __device__ __forceinline__ void phase(F &&f) {
    f(tid, st);
    __syncthreads();
  }
};

template <typename S> struct DevExS {
  using State = S;
  int nthr;
  int tid;
  State st;
  __device__ DevExS() : nthr(blockDim.x), tid(threadIdx.x) {}
  template <typename F> __device__ __forceinline__ void phase(F &&f) {
    f(tid, st);
    __syncthreads();
  }
};

// ---------------------------------------------------------------------------
// apply kernels
// ---------------------------------------------------------------------------

template <typename T> __global__ void __launch_bounds__(1024) k_small(const ConvArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int L = 1 << a.log2M;
  c2<T> *buf = reinterpret_cast<c2<T> *>(smem);
  T *red = reinterpret_cast<T *>(smem + padded_size(L) * sizeof(c2<T>));
  T *coef = red + ((blockDim.x + 31) / 32) * 128;
  DevEx<T> ex;
  small_body<T>(ex, a, (int64_t)blockIdx.x, buf, red, coef);
}

template <typename T>
__global__ void __launch_bounds__(1024) k_small_ragged(const RaggedDesc<T> *d, const ConvArgs<T> base) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int L = 1 << base.log2M;
  c2<T> *buf = reinterpret_cast<c2<T> *>(smem);
  T *red = reinterpret_cast<T *>(smem + padded_size(L) * sizeof(c2<T>));
  T *coef = red + ((blockDim.x + 31) / 32) * 128;
  const RaggedDesc<T> q = d[blockIdx.x];
  ConvArgs<T> a = base;
  a.y = q.y;
  a.out = q.out;
  a.ld = q.N;
  a.N = q.N;
  a.spec = q.spec;
  a.ST = q.ST;
  a.D = q.D;
  a.r = q.r;
  a.rpad = q.rpad;
  DevEx<T> ex;
  small_body<T>(ex, a, 0, buf, red, coef);
}

template <typename T> __global__ void __launch_bounds__(1024) k_passA(const ConvArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int P = 1 << a.log2P;
  const int ncols = a.G * a.NB;
  c2<T> *buf = reinterpret_cast<c2<T> *>(smem);
  T *red = reinterpret_cast<T *>(smem + padded_size(P * ncols) * sizeof(c2<T>));
  DevEx<T> ex;
  passA_body<T>(ex, a, (int64_t)blockIdx.x, (int64_t)blockIdx.y, buf, red);
}

template <typename T> __global__ void k_reduce(const ConvArgs<T> a) {
  reduce_body<T>(a, (int64_t)blockIdx.x, threadIdx.x, blockDim.x);
}

// (FP64 rows have at most 8192 points)
template <typename T> __global__ void __launch_bounds__(sizeof(T) == 8 ? 512 : 1024) k_passB(const ConvArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  c2<T> *buf = reinterpret_cast<c2<T> *>(smem);
  DevEx<T> ex;
  passB_body<T>(ex, a, (int64_t)blockIdx.y, (int)blockIdx.x, buf);
}

template <typename T> __global__ void __launch_bounds__(1024) k_passC(const ConvArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  c2<T> *buf = reinterpret_cast<c2<T> *>(smem);
  DevEx<T> ex;
  passC_body<T>(ex, a, (int64_t)blockIdx.x, (int64_t)blockIdx.y, buf);
}

// ---------------------------------------------------------------------------
// plan kernels
// ---------------------------------------------------------------------------

// One round of multisection: warp w of target t narrows the target's interval with the counts of
// the previous round (every warp of a target does so by itself; its first one keeps the result
// for the next round), then counts at its 32 points.  iv: [2][nt][lo, hi], cnt: [2][nt][32 warps],
// the halves alternate with the round.  The last call (eval = 0) only narrows.  Blocks of four
// warps: one on each sub-core's FP64 unit.
constexpr int BISECT_THREADS = 128;
__global__ void __launch_bounds__(BISECT_THREADS) k_bisect_round(const TargetDesc *td, int nt, int warps, int round, int eval,
                                                     const double *dcat, const double *e2cat, double *iv, int *cnt,
                                                     double *theta, int *flag) {
  const int gw = blockIdx.x * (BISECT_THREADS / 32) + (threadIdx.x >> 5);
  const int t = gw / warps, w = gw % warps, lane = threadIdx.x & 31, np = 32 * warps;
  if (t >= nt) return;
  const TargetDesc q = td[t];
  double lo = q.glo, hi = q.ghi;
  if (round > 0) {
    const double *ivp = iv + ((size_t)((round - 1) & 1) * nt + t) * 2;
    const int *cp = cnt + ((size_t)((round - 1) & 1) * nt + t) * np;
    int k = 0;
    for (int i = lane; i < np; i += 32) k += cp[i] <= q.target;
    k = __reduce_add_sync(0xffffffffu, k);
    lo = ivp[0];
    hi = ivp[1];
    bisect_narrow(&lo, &hi, k, np);
  }
  if (w == 0 && lane == 0) {
    double *ivn = iv + ((size_t)(round & 1) * nt + t) * 2;
    ivn[0] = lo;
    ivn[1] = hi;
    if (!eval) {
      theta[t] = 0.5 * (lo + hi);
      if (!bisect_converged(lo, hi, q.tol)) *flag = 1;
    }
  }
  if (eval)
    cnt[((size_t)(round & 1) * nt + t) * np + 32 * w + lane] =
        sturm_count(dcat + q.mat_off, e2cat + q.mat_off, q.n, bisect_point(lo, hi, 32 * w + lane, np), q.pivmin);
}

__global__ void k_bisect_many(const TargetDesc *td, int nt, const double *dcat, const double *e2cat, double *theta,
                              int *flag) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nt) return;
  const TargetDesc q = td[t];
  bisect1_body(dcat + q.mat_off, e2cat + q.mat_off, q.n, q.target, q.glo, q.ghi, q.pivmin, q.tol, theta + t, flag);
}
// `lanes` targets per one-warp block
__global__ void __launch_bounds__(32) k_fwdvec_many(const TargetDesc *td, int nt, int lanes, const double *dcat,
                                                    const double *ecat, const double *rcat, const double *theta,
                                                    double *z, double *w, int *ex, double *delta) {
  const int t = blockIdx.x * lanes + threadIdx.x;
  if ((int)threadIdx.x >= lanes || t >= nt) return;
  const TargetDesc q = td[t];
  fwdvec_body(dcat + q.mat_off, ecat + q.mat_off, rcat + q.mat_off, q.n, theta[t], z + q.x_off, w + q.x_off,
              ex + q.x_off / PLAN_B, delta + t);
}
__global__ void k_finalize_many(const TargetDesc *td, const double *z, const double *w, const int *bex,
                                const double *delta) {
  __shared__ double sh[2 * 256];
  DevExPlan ex;
  const TargetDesc q = td[blockIdx.x];
  finalize_body(ex, z + q.x_off, w + q.x_off, bex + q.x_off / PLAN_B, delta[blockIdx.x], q.n, q.parity, q.N, q.S, sh);
}

__global__ void k_dot(const double *a, const double *b, int64_t N, double *out) {
  __shared__ double sh[256];
  DevExPlan ex;
  const int64_t off = (int64_t)blockIdx.x * N;
  dot_body(ex, a + off, b + off, N, out + blockIdx.x, sh);
}

__global__ void k_sinc(double *c, int64_t N, int64_t M, double W) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < M; k += (int64_t)gridDim.x * blockDim.x)
    c[k] = sinc_embed_at(k, N, M, W);
}

__global__ void k_spec_store(const double2 *X, Layout L64, Layout L32, int64_t M, double scale, double *spec64,
                             float *spec32) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < M; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p64 = spec_pos(L64, k);
    const double v = X[p64].x * scale;
    spec64[p64] = v;
    spec32[spec_pos(L32, k)] = (float)v;
  }
}

__global__ void k_gather(const double *S, int64_t N, const int *sel, int r, int rpad, double *ST64, float *ST32) {
  const int64_t total = N * rpad;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t n = t / rpad;
    const int j = (int)(t % rpad);
    const double v = (j < r) ? S[(int64_t)sel[j] * N + n] : 0.0;
    ST64[t] = v;
    ST32[t] = (float)v;
  }
}

// ---- T1 c (fst_expand) ----
template <typename T> __global__ void k_exp_scatter(const ExpArgs<T> a, int64_t nsig, c2<T> *Xs) {
  const int64_t total = nsig * a.N;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x)
    exp_scatter_body<T>(a, t / a.N, t % a.N, Xs);
}
// block b of a signal row: samples b (EXP_E 256) + tid + i 256, i < EXP_E
template <typename T> __global__ void __launch_bounds__(256) k_expand(const ExpArgs<T> a, int64_t nsig) {
  const int64_t per = (a.N + EXP_E * 256 - 1) / (EXP_E * 256);
  for (int64_t bb = blockIdx.x; bb < nsig * per; bb += gridDim.x)
    exp_samples_body<T>(a, bb / per, (bb % per) * (EXP_E * 256) + threadIdx.x, 256);
}

// ---- fast coefficient vector kernels ----
template <typename T> __global__ void __launch_bounds__(COEF_THREADS) k_coef_lowrank(const CoefArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  DevExS<CState<T>> ex;
  coef_lowrank_body<T>(ex, a, (int64_t)blockIdx.y, (int)blockIdx.x, reinterpret_cast<T *>(smem));
}
template <typename T> __global__ void __launch_bounds__(COEF_THREADS) k_coef_st(const CoefArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  DevExS<CState<T>> ex;
  coef_st_body<T>(ex, a, (int64_t)blockIdx.y, (int)blockIdx.x, reinterpret_cast<T *>(smem));
}
template <typename T> __global__ void k_coef_reduce(const T *part, int nchunks, int nout, T *tot) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o < nout) coef_reduce_body<T>(part, nchunks, nout, (int64_t)blockIdx.y, o, tot);
}
template <typename T>
__global__ void k_coef_gather(const c2<T> *X, Layout Lf, int64_t N, int cplx, int64_t sig0, int64_t nsig, int64_t h,
                              c2<T> *out, int64_t Kp) {
  const int64_t nF = 2 * h + 1, total = nsig * nF;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = sig0 + t / nF, k = t % nF;
    const int64_t pl = cplx ? (s - sig0) : (s / 2 - sig0 / 2);
    coef_gather_body<T>(X, Lf, N, cplx, s, pl, h, k, out + s * Kp);
  }
}
// F^* y bins from the [k1][k2] transform of 4096-point rows (P >= 8): a block takes 32 columns k2 by
// up to 32 rows k1 of one pair (and, for real pairs, their mirror images: index N - k lies in row
// P - k1, column Q - 1 - k2, row 0: Q - k2), transposes them in shared memory and writes runs of
// consecutive bins.  Bound: memory; the plain gather reads 8 bytes per 32-byte sector.  Measured on
// 16 signals of N = 2^22, 2^21 bins each: 287 -> 136 us.
__global__ void __launch_bounds__(256) k_coef_gather_t(const float2 *X, int log2P, int log2Q, int cplx, int64_t sig0,
                                                       int64_t nsig, int64_t h, float2 *out, int64_t Kp) {
  __shared__ float2 ta[32][33], tb[32][33];   // [k2][k1] of the first and the second signal
  const int P = 1 << log2P, Q = 1 << log2Q, R = P < 32 ? P : 32;
  const int64_t N = (int64_t)P << log2Q, pl = blockIdx.y;
  const int k2_0 = (int)(blockIdx.x % (Q / 32)) * 32, k1_0 = (int)(blockIdx.x / (Q / 32)) * R;
  // indices k1_0 + P k2_0 .. of the tile: skip tiles without a bin in [0, h] or [N - h, N)
  const int64_t lo = k1_0 + (int64_t)P * k2_0, hi = k1_0 + R - 1 + (int64_t)P * (k2_0 + 31);
  if (lo > h && hi < N - h) return;
  const float2 *Xp = X + pl * N;
  const float s = (float)(1.0 / sqrt((double)N));
  for (int e = threadIdx.x; e < 32 * R; e += 256) {
    const int i = e % 32, q = e / 32, k1 = k1_0 + q, k2 = k2_0 + i;
    const float2 z = Xp[(int64_t)k1 * Q + k2];
    if (cplx) {
      ta[i][q] = cscale(z, s);
    } else {
      const int m1 = (P - k1) & (P - 1), m2 = (k1 ? Q - 1 - k2 : (Q - k2) & (Q - 1));
      const float2 zc = cconj(Xp[(int64_t)m1 * Q + m2]);
      ta[i][q] = cscale(cscale(cadd(z, zc), 0.5f), s);
      const float2 d = csub(z, zc);
      tb[i][q] = cscale(make_float2(0.5f * d.y, -0.5f * d.x), s);   // d / (2 j)
    }
  }
  __syncthreads();
  const int64_t sa = cplx ? sig0 + pl : sig0 + 2 * pl;
  for (int e = threadIdx.x; e < 32 * R; e += 256) {
    const int q = e % R, i = e / R;
    const int64_t k = k1_0 + q + (int64_t)P * (k2_0 + i);
    if (k > h && k < N - h) continue;
    const int64_t o = k <= h ? k + h : k - N + h;
    out[sa * Kp + o] = ta[i][q];
    if (!cplx && sa + 1 < sig0 + nsig) out[(sa + 1) * Kp + o] = tb[i][q];
  }
}
template <typename T>
__global__ void k_coef_mix(const CoefArgs<T> a, const T *tot, const T *totU, const T *CA, const T *CB, const T *sq,
                           c2<T> *out, int64_t Kp, int64_t nF) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t sig = blockIdx.y;
  const int nfin = 4 * a.rH + 2 * a.DA + 2 * a.DB + a.r;
  if (o >= nfin) return;
  out[sig * Kp + nF + o] =
      coef_mix_value<T>(a, tot + sig * (int64_t)a.nraw * 2, totU + sig * (int64_t)(a.r > 0 ? a.r : 1) * 2, CA, CB, sq, o, sig);
}

__global__ void k_split_tf32(const float *src, float2 *hl, int64_t n) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const float h = tf32_round(src[t]);
    hl[t] = make_float2(h, tf32_round(src[t] - h));
  }
}

__global__ void k_to_f32(const double *src, float *dst, int64_t n) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    dst[t] = (float)src[t];
}

// ---------------------------------------------------------------------------
// device runner
// ---------------------------------------------------------------------------

static fst_status cuda_fail(cudaError_t e, const char *what) {
  return fail(e == cudaErrorMemoryAllocation ? FST_ENOMEM : FST_ECUDA,
              std::string(what) + ": " + cudaGetErrorString(e));
}
#define CU(call, what)                                  \
  do {                                                  \
    cudaError_t _e = (call);                            \
    if (_e != cudaSuccess) return cuda_fail(_e, what);  \
  } while (0)
#define LAUNCHED(what) CU(cudaGetLastError(), what)
#define TRY(expr)                \
  do {                           \
    fst_status _s = (expr);      \
    if (_s != FST_OK) return _s; \
  } while (0)

static bool g_attr_done = false;
static fst_status set_attrs() {
  if (g_attr_done) return FST_OK;
  const int mx = 227 * 1024;
  CU(cudaFuncSetAttribute(k_small<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_small<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_small_ragged<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_small_ragged<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_passA<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_passA<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_passB<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_passB<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_passC<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_passC<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_c<false, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_c<false, 8, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_c<true, 8, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_c<false, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_c<false, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_c<true, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_c<true, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_c<true, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_z<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_sym_z<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_coef_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_expand_gemm<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_expand_gemm<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_expand_gemm<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_small32<13>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_smem(13, SM_RMAX)), "attr");
  CU(cudaFuncSetAttribute(k_small32<14>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_smem(14, SM_RMAX)), "attr");
  CU(cudaFuncSetAttribute(k_small32_ragged<13>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_smem(13, SM_RMAX)), "attr");
  CU(cudaFuncSetAttribute(k_small32_ragged<14>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_smem(14, SM_RMAX)), "attr");
  CU(cudaFuncSetAttribute(k_fastAw<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, fastw_smem(32)), "attr");
  CU(cudaFuncSetAttribute(k_fastAw<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, fastw_smem(16)), "attr");
  CU(cudaFuncSetAttribute(k_fastAw<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, fastw_smem(8)), "attr");
  CU(cudaFuncSetAttribute(k_corr_cc, cudaFuncAttributeMaxDynamicSharedMemorySize, cc_smem(64)), "attr");
  CU(cudaFuncSetAttribute(k_fastB8192, cudaFuncAttributeMaxDynamicSharedMemorySize, fastb8192_smem()), "attr");
  CU(cudaFuncSetAttribute(k_fastB4096_2s, cudaFuncAttributeMaxDynamicSharedMemorySize, fastb2s_smem()), "attr");
  CU(cudaFuncSetAttribute(k_rcorr_part, cudaFuncAttributeMaxDynamicSharedMemorySize, rcorr_smem()), "attr");
  CU(cudaFuncSetAttribute(k_colA<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(2)), "attr");
  CU(cudaFuncSetAttribute(k_colA<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(2)), "attr");
  CU(cudaFuncSetAttribute(k_colA<4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(4)), "attr");
  CU(cudaFuncSetAttribute(k_colA<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(4)), "attr");
  CU(cudaFuncSetAttribute(k_colA<8, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(8)), "attr");
  CU(cudaFuncSetAttribute(k_colA<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(8)), "attr");
  CU(cudaFuncSetAttribute(k_colA<16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(16)), "attr");
  CU(cudaFuncSetAttribute(k_colA<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(16)), "attr");
  CU(cudaFuncSetAttribute(k_colA<32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(32)), "attr");
  CU(cudaFuncSetAttribute(k_colA<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(32)), "attr");
  CU(cudaFuncSetAttribute(k_colC<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(2)), "attr");
  CU(cudaFuncSetAttribute(k_colC<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(4)), "attr");
  CU(cudaFuncSetAttribute(k_colC<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(8)), "attr");
  CU(cudaFuncSetAttribute(k_colC<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(16)), "attr");
  CU(cudaFuncSetAttribute(k_colC<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, big_smem_bytes(32)), "attr");
  CU(cudaFuncSetAttribute(k_corr_tc<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_corr_tc<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_corr_tc<96>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  CU(cudaFuncSetAttribute(k_corr_tc<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx), "attr");
  g_attr_done = true;
  return FST_OK;
}

// ---- launch accounting (fst_launch_count / fst_profile_*) --------------------
static long long g_launches = 0;
static int g_prof_on = 0;
struct ProfRec {
  const char *name;
  cudaEvent_t a, b;
  long long units;
};
static std::vector<ProfRec> g_prof;
static void prof_begin(cudaStream_t s, const char *name, long long units, cudaEvent_t *ea) {
  ++g_launches;
  *ea = nullptr;
  if (!g_prof_on) return;
  cudaEventCreate(ea);
  cudaEventRecord(*ea, s);
  ProfRec r{name, *ea, nullptr, units};
  g_prof.push_back(r);
}
static void prof_end(cudaStream_t s, cudaEvent_t ea) {
  if (!g_prof_on || !ea) return;
  cudaEvent_t eb;
  cudaEventCreate(&eb);
  cudaEventRecord(eb, s);
  g_prof.back().b = eb;
}
#define PROF(name, units, launch)            \
  do {                                       \
    cudaEvent_t _ea;                         \
    prof_begin(cur, name, (units), &_ea);    \
    launch;                                  \
    prof_end(cur, _ea);                      \
  } while (0)

#define PROF_S(stream, name, units, launch) \
  do {                                       \
    cudaEvent_t _ea;                         \
    prof_begin(stream, name, (units), &_ea); \
    launch;                                  \
    prof_end(stream, _ea);                   \
  } while (0)

bool profiling_enabled() { return g_prof_on != 0; }

// ---- TMA tensor maps (driver entry point, resolved once) --------------------
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    else
      cudaGetLastError();
  });
  return fn;
}

// 2-D FP32 tensor map: rows of `inner` elements `row_bytes` apart, box inner x outer
static fst_status encode_2d(CUtensorMap *m, const void *base, uint64_t inner, uint64_t outer, uint64_t row_bytes,
                            uint32_t box_inner, uint32_t box_outer, bool swizzle128) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc) return fail(FST_ECUDA, "cuTensorMapEncodeTiled not available");
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {row_bytes};
  const cuuint32_t box[2] = {box_inner, box_outer};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void *>(base), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE,
                         swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(FST_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return FST_OK;
}

// test hook (fst_test_tc_stall): the next g_tc_stall launches of the tcgen05 correction give
// up after g_tc_stall_limit_ns on a wait that nothing completes
static std::atomic<int> g_tc_stall{0};
static unsigned long long g_tc_stall_limit_ns = 20000000ull;
bool tc_stall_pending() { return g_tc_stall.load() > 0; }
bool tc_stall_take() {
  int v = g_tc_stall.load();
  while (v > 0)
    if (g_tc_stall.compare_exchange_weak(v, v - 1)) return true;
  return false;
}

// test hook (fst_test_alloc_fail): after g_alloc_after more device allocations the next g_alloc_fail
// ones report a full device
static std::atomic<int> g_alloc_fail{0}, g_alloc_after{0};
static bool alloc_fail_take() {
  if (g_alloc_fail.load() <= 0 || g_alloc_after.fetch_sub(1) > 0) return false;
  return g_alloc_fail.fetch_sub(1) > 0;
}

static inline int grid_for(int64_t n, int block) {
  int64_t g = (n + block - 1) / block;
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, 152 * 32));
}

struct DevRunner : Runner {
  cudaStream_t s = nullptr;     // caller's stream
  cudaStream_t cur = nullptr;   // stream the apply kernels go to (s, or a capture lane)
  cudaStream_t cap[3] = {nullptr, nullptr, nullptr};   // two lanes and the side lane
  cudaEvent_t fork = nullptr, join = nullptr, ev_mid = nullptr, ev_side = nullptr, join_side = nullptr;
  bool capturing = false;
  long long launches_at_begin = 0;
  int sms = 1;
  // raised by k_corr_tc when one of its waits timed out: a host-mapped word, so the host
  // reads it without a copy (fst_sync, and the next call on the plan)
  int *tc_err = nullptr;     // device address
  int *tc_err_h = nullptr;   // host address
  bool device() const override { return true; }
  int sm_count() const override { return sms; }
  void set_stream(void *st) override { s = (cudaStream_t)st; cur = s; }
  void *stream() const override { return (void *)s; }
  ~DevRunner() override {
    for (int i = 0; i < 3; ++i)
      if (cap[i]) cudaStreamDestroy(cap[i]);
    for (cudaEvent_t e : {fork, join, ev_mid, ev_side, join_side, t0, t1})
      if (e) cudaEventDestroy(e);
    for (cudaStream_t b : br)
      if (b) cudaStreamDestroy(b);
    for (cudaEvent_t e : br_ev)
      if (e) cudaEventDestroy(e);
    if (tc_err_h) cudaFreeHost(tc_err_h);
  }
  static constexpr int BRANCHES = 6;
  cudaStream_t br[BRANCHES] = {};
  cudaEvent_t br_ev[BRANCHES + 1] = {};
  bool br_on[BRANCHES] = {};
  fst_status branch(int k) override {
    cur = s;
    if (k < 0) return FST_OK;
    k %= BRANCHES;
    if (!br[k]) {
      CU(cudaStreamCreateWithFlags(&br[k], cudaStreamNonBlocking), "stream");
      CU(cudaEventCreateWithFlags(&br_ev[k], cudaEventDisableTiming), "event");
    }
    if (!br_ev[BRANCHES]) CU(cudaEventCreateWithFlags(&br_ev[BRANCHES], cudaEventDisableTiming), "event");
    if (!br_on[k]) {
      CU(cudaEventRecord(br_ev[BRANCHES], s), "event");
      CU(cudaStreamWaitEvent(br[k], br_ev[BRANCHES], 0), "wait");
      br_on[k] = true;
    }
    cur = br[k];
    return FST_OK;
  }
  fst_status branch_join() override {
    cur = s;
    for (int k = 0; k < BRANCHES; ++k)
      if (br_on[k]) {
        br_on[k] = false;
        CU(cudaEventRecord(br_ev[k], br[k]), "event");
        CU(cudaStreamWaitEvent(s, br_ev[k], 0), "wait");
      }
    return FST_OK;
  }
  cudaEvent_t t0 = nullptr, t1 = nullptr;
  fst_status timer(int phase, double *ms) override {
    if (!t0) {
      CU(cudaEventCreate(&t0), "event");
      CU(cudaEventCreate(&t1), "event");
    }
    if (phase == 0) {
      CU(cudaEventRecord(t0, cur), "event");
      return FST_OK;
    }
    CU(cudaEventRecord(t1, cur), "event");
    CU(cudaEventSynchronize(t1), "event sync");
    float f = 0.f;
    CU(cudaEventElapsedTime(&f, t0, t1), "elapsed");
    if (ms) *ms = f;
    return FST_OK;
  }
  fst_status device_status(bool sync) override {
    if (sync) CU(cudaStreamSynchronize(s), "cudaStreamSynchronize");
    if (tc_err_h && *(volatile int *)tc_err_h) {
      *(volatile int *)tc_err_h = 0;
      return fail(FST_ETIMEOUT, "a bounded wait of the tensor-core correction ran past its limit; the outputs "
                                "of that call are NaN");
    }
    return FST_OK;
  }

  int lanes() const override { return capturing ? 2 : 1; }
  void use_lane(int i) override { cur = capturing ? cap[i & 1] : s; }
  void lanes_join_first() override {
    if (!capturing) return;
    cudaEventRecord(ev_mid, cap[1]);
    cudaStreamWaitEvent(cap[0], ev_mid, 0);
  }
  void use_side() override { cur = capturing ? cap[2] : s; }
  void side_done() override {
    if (capturing) cudaEventRecord(ev_side, cap[2]);
  }
  void wait_side() override {
    if (capturing) cudaStreamWaitEvent(cur, ev_side, 0);
  }
  bool user_stream_capturing() override {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
      cudaGetLastError();
      return true;
    }
    return st != cudaStreamCaptureStatusNone;
  }
  bool graph_begin() override {
    if (!cap[0]) {
      for (int i = 0; i < 3; ++i)
        if (cudaStreamCreateWithFlags(&cap[i], cudaStreamNonBlocking) != cudaSuccess) { cudaGetLastError(); return false; }
      for (cudaEvent_t *e : {&fork, &join, &ev_mid, &ev_side, &join_side})
        if (cudaEventCreateWithFlags(e, cudaEventDisableTiming) != cudaSuccess) {
          cudaGetLastError();
          return false;
        }
    }
    if (set_attrs() != FST_OK) return false;
    if (cudaStreamBeginCapture(cap[0], cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    cudaEventRecord(fork, cap[0]);
    cudaStreamWaitEvent(cap[1], fork, 0);
    cudaStreamWaitEvent(cap[2], fork, 0);
    capturing = true;
    cur = cap[0];
    launches_at_begin = g_launches;
    return true;
  }
  fst_status graph_end(void **exec, long long *nodes) override {
    *exec = nullptr;
    cudaEventRecord(join, cap[1]);
    cudaStreamWaitEvent(cap[0], join, 0);
    cudaEventRecord(join_side, cap[2]);
    cudaStreamWaitEvent(cap[0], join_side, 0);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(cap[0], &g);
    capturing = false;
    cur = s;
    *nodes = g_launches - launches_at_begin;
    g_launches = launches_at_begin;   // captured, not yet run
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
    cudaGraphExec_t ex = nullptr;
    e = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
    *exec = (void *)ex;
    return FST_OK;
  }
  fst_status graph_launch(void *exec, long long nodes) override {
    CU(cudaGraphLaunch((cudaGraphExec_t)exec, s), "cudaGraphLaunch");
    g_launches += nodes;
    return FST_OK;
  }
  void graph_destroy(void *exec) override {
    if (exec) cudaGraphExecDestroy((cudaGraphExec_t)exec);
  }

  fst_status alloc(void **p, size_t bytes) override {
    *p = nullptr;
    const cudaError_t e = alloc_fail_take() ? cudaErrorMemoryAllocation : cudaMalloc(p, std::max<size_t>(bytes, 16));
    if (e == cudaSuccess) return FST_OK;
    cudaGetLastError();   // a caller that goes on without this memory must not find the error at its next launch
    return cuda_fail(e, "cudaMalloc");
  }
  void release(void *p) override {
    if (p) cudaFree(p);
  }
  fst_status h2d(void *dst, const void *src, size_t bytes) override {
    CU(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, s), "h2d");
    CU(cudaStreamSynchronize(s), "h2d sync");
    return FST_OK;
  }
  fst_status d2h(void *dst, const void *src, size_t bytes) override {
    CU(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s), "d2h");
    CU(cudaStreamSynchronize(s), "d2h sync");
    return FST_OK;
  }
  fst_status d2d(void *dst, const void *src, size_t bytes) override {
    CU(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, s), "d2d");
    return FST_OK;
  }
  fst_status zero(void *p, size_t bytes) override {
    CU(cudaMemsetAsync(p, 0, bytes, s), "memset");
    return FST_OK;
  }
  fst_status sync() override {
    CU(cudaStreamSynchronize(s), "sync");
    return FST_OK;
  }

  template <typename T> fst_status small_t(const ConvArgs<T> &a, const Layout &L) {
    if (set_attrs() != FST_OK) return FST_ECUDA;
    PROF(sizeof(T) == 4 ? "k_small<f32>" : "k_small<f64>", a.npairs,
         (k_small<T><<<(unsigned)a.npairs, L.nthr_small, L.smem_small, cur>>>(a)));
    LAUNCHED("k_small");
    return FST_OK;
  }
  template <typename T> fst_status passA_t(const ConvArgs<T> &a, const Layout &L) {
    if (set_attrs() != FST_OK) return FST_ECUDA;
    dim3 grid((unsigned)L.ntiles, (unsigned)((a.npairs + L.G - 1) / L.G));
    PROF(sizeof(T) == 4 ? "k_passA<f32>" : "k_passA<f64>", a.npairs, (k_passA<T><<<grid, L.nthr_A, L.smem_A, cur>>>(a)));
    LAUNCHED("k_passA");
    return FST_OK;
  }
  template <typename T> fst_status reduce_t(const ConvArgs<T> &a, const Layout &) {
    const int thr = std::min(1024, std::max(32, ((2 * a.r + 31) / 32) * 32));
    PROF(sizeof(T) == 4 ? "k_reduce<f32>" : "k_reduce<f64>", a.npairs, (k_reduce<T><<<(unsigned)a.npairs, thr, 0, cur>>>(a)));
    LAUNCHED("k_reduce");
    return FST_OK;
  }
  template <typename T> fst_status passB_t(const ConvArgs<T> &a, const Layout &L) {
    if (set_attrs() != FST_OK) return FST_ECUDA;
    dim3 grid((unsigned)(1u << L.log2P), (unsigned)a.npairs);
    PROF(sizeof(T) == 4 ? "k_passB<f32>" : "k_passB<f64>", a.npairs, (k_passB<T><<<grid, L.nthr_B, L.smem_B, cur>>>(a)));
    LAUNCHED("k_passB");
    return FST_OK;
  }
  template <typename T> fst_status passC_t(const ConvArgs<T> &a, const Layout &L) {
    if (set_attrs() != FST_OK) return FST_ECUDA;
    dim3 grid((unsigned)L.ntiles, (unsigned)((a.npairs + L.G - 1) / L.G));
    PROF(sizeof(T) == 4 ? "k_passC<f32>" : "k_passC<f64>", a.npairs, (k_passC<T><<<grid, L.nthr_C, L.smem_C, cur>>>(a)));
    LAUNCHED("k_passC");
    return FST_OK;
  }
  template <typename T>
  fst_status small_ragged_t(const RaggedDesc<T> *d, int count, const ConvArgs<T> &base, const Layout &L) {
    if (set_attrs() != FST_OK) return FST_ECUDA;
    PROF(sizeof(T) == 4 ? "k_small_ragged<f32>" : "k_small_ragged<f64>", count,
         (k_small_ragged<T><<<(unsigned)count, L.nthr_small, L.smem_small, cur>>>(d, base)));
    LAUNCHED("k_small_ragged");
    return FST_OK;
  }
  fst_status small_ragged(const RaggedDesc<float> *d, int count, const ConvArgs<float> &base,
                          const Layout &L) override { return small_ragged_t(d, count, base, L); }
  fst_status small_ragged(const RaggedDesc<double> *d, int count, const ConvArgs<double> &base,
                          const Layout &L) override { return small_ragged_t(d, count, base, L); }
  template <int LM> fst_status small32_t(const ConvArgs<float> &a) {
    TRY(set_attrs());
    SmallPlan p{a.spec, a.ST, a.STt, a.D, a.twS, a.tc_Npad, (int)a.N, a.r, a.rpad, {a.odd[0], a.odd[1], a.odd[2], a.odd[3]}};
    PROF("k_small32", a.npairs, (k_small32<LM><<<(unsigned)a.npairs, (1 << LM) / 16, sm_smem(LM, a.rpad), cur>>>(a, p)));
    LAUNCHED("k_small32");
    return FST_OK;
  }
  template <int LM>
  fst_status small32_ragged_t(const SmallDesc *d, int count, int rpad_max, const float2 *twB, int cplx) {
    TRY(set_attrs());
    PROF("k_small32_ragged", count,
         (k_small32_ragged<LM><<<(unsigned)count, (1 << LM) / 16, sm_smem(LM, rpad_max), cur>>>(d, twB, cplx)));
    LAUNCHED("k_small32_ragged");
    return FST_OK;
  }
  fst_status small32_prep(const Tw<double> &tw, int log2M, float2 *twS, const float *ST, int64_t N, int rpad, int r,
                          float *STs) override {
    if (sm_words(log2M) > 0) {
      k_tw_small<<<grid_for(sm_words(log2M), 256), 256, 0, s>>>(tw, log2M, twS);
      LAUNCHED("k_tw_small");
    }
    if (r > 0) {
      k_tc_prep<<<grid_for(r * N, 256), 256, 0, s>>>(ST, N, rpad, r, r, N, STs);
      LAUNCHED("k_tc_prep");
    }
    return FST_OK;
  }
  fst_status small32_ragged(const SmallDesc *d, int count, int log2M, int rpad_max, const float2 *twB,
                            int cplx) override {
    switch (log2M) {
      case 10: return small32_ragged_t<10>(d, count, rpad_max, twB, cplx);
      case 11: return small32_ragged_t<11>(d, count, rpad_max, twB, cplx);
      case 12: return small32_ragged_t<12>(d, count, rpad_max, twB, cplx);
      case 13: return small32_ragged_t<13>(d, count, rpad_max, twB, cplx);
      case 14: return small32_ragged_t<14>(d, count, rpad_max, twB, cplx);
      default: return fail(FST_EINVAL, "single-CTA transform length out of range");
    }
  }
  fst_status small(const ConvArgs<float> &a, const Layout &L) override {
    // the restructured kernel where its tables exist (M = 2^10 .. 2^14, r <= 128)
    if (a.twS && (a.mode == MODE_FULL || a.mode == MODE_CONV)) {
      switch (a.log2M) {
        case 10: return small32_t<10>(a);
        case 11: return small32_t<11>(a);
        case 12: return small32_t<12>(a);
        case 13: return small32_t<13>(a);
        case 14: return small32_t<14>(a);
        default: break;
      }
    }
    return small_t(a, L);
  }
  fst_status small(const ConvArgs<double> &a, const Layout &L) override { return small_t(a, L); }
  template <int P2> fst_status colA_t(const ConvArgs<float> &a, const Layout &L) {
    TRY(set_attrs());
    dim3 grid((unsigned)L.ntiles, (unsigned)a.npairs);
    if (a.mode == MODE_FORWARD) {
      PROF("k_colA_full", a.npairs, (k_colA<P2, true><<<grid, 256, big_smem_bytes(P2), cur>>>(a)));
      LAUNCHED("k_colA_full");
      return FST_OK;
    }
    PROF(P2 == 2 ? "k_colA<2>" : P2 == 4 ? "k_colA<4>" : P2 == 8 ? "k_colA<8>" : P2 == 16 ? "k_colA<16>" : "k_colA<32>",
         a.npairs, (k_colA<P2><<<grid, 256, big_smem_bytes(P2), cur>>>(a)));
    LAUNCHED("k_colA");
    return FST_OK;
  }
  template <int P2> fst_status colC_t(const ConvArgs<float> &a, const Layout &L) {
    TRY(set_attrs());
    dim3 grid((unsigned)L.ntiles, (unsigned)a.npairs);
    PROF(P2 == 2 ? "k_colC<2>" : P2 == 4 ? "k_colC<4>" : P2 == 8 ? "k_colC<8>" : P2 == 16 ? "k_colC<16>" : "k_colC<32>",
         a.npairs, (k_colC<P2><<<grid, 256, big_smem_bytes(P2), cur>>>(a)));
    LAUNCHED("k_colC");
    return FST_OK;
  }
  fst_status passA(const ConvArgs<float> &a, const Layout &L) override {
    if (L.big) {
      switch (L.P2) {
        case 2: return colA_t<2>(a, L);
        case 4: return colA_t<4>(a, L);
        case 8: return colA_t<8>(a, L);
        case 16: return colA_t<16>(a, L);
        case 32: return colA_t<32>(a, L);
        default: return fail(FST_EINVAL, "column pass width out of range");
      }
    }
    if (!L.fast) return passA_t(a, L);
    const int P = 1 << L.log2P;
    if (a.mode == MODE_FORWARD) {
      dim3 grid((unsigned)((1u << L.log2Q) / 256), (unsigned)a.npairs);
      if (P == 32) PROF("k_fastA_full", a.npairs, (k_fastA_full<32><<<grid, 256, 0, cur>>>(a)));
      else if (P == 16) PROF("k_fastA_full", a.npairs, (k_fastA_full<16><<<grid, 256, 0, cur>>>(a)));
      else PROF("k_fastA_full", a.npairs, (k_fastA_full<8><<<grid, 256, 0, cur>>>(a)));
      LAUNCHED("k_fastA_full");
      return FST_OK;
    }
    // no fused correction, real signals: 256-byte row loads when the rows allow float2 loads
    // (measured faster for real rows, slower for complex ones)
    const bool wide_ok = !a.rp && !a.cplx && (uintptr_t)a.y % 8 == 0 && a.ld % 2 == 0;
    if (a.mode != MODE_FULL && wide_ok) {
      TRY(set_attrs());
      const int64_t tiles = ((1 << L.log2Q) / FASTW_NB) * ((a.npairs + FASTW_G - 1) / FASTW_G);
      const unsigned grid = (unsigned)std::min<int64_t>(tiles, 3 * (int64_t)sms);
      if (P == 32) PROF("k_fastAw<32>", a.npairs, (k_fastAw<32><<<grid, FAST_THREADS, fastw_smem(32), cur>>>(a)));
      else if (P == 16) PROF("k_fastAw<16>", a.npairs, (k_fastAw<16><<<grid, FAST_THREADS, fastw_smem(16), cur>>>(a)));
      else PROF("k_fastAw<8>", a.npairs, (k_fastAw<8><<<grid, FAST_THREADS, fastw_smem(8), cur>>>(a)));
      LAUNCHED("k_fastAw");
      return FST_OK;
    }
    FastArgs f{a, a.ST_hl};
    dim3 grid((unsigned)L.ntiles, (unsigned)((a.npairs + FAST_G - 1) / FAST_G));
    if (P == 32) PROF("k_fastA<32>", a.npairs, (k_fastA<32><<<grid, FAST_THREADS, 0, cur>>>(f)));
    else if (P == 16) PROF("k_fastA<16>", a.npairs, (k_fastA<16><<<grid, FAST_THREADS, 0, cur>>>(f)));
    else PROF("k_fastA<8>", a.npairs, (k_fastA<8><<<grid, FAST_THREADS, 0, cur>>>(f)));
    LAUNCHED("k_fastA");
    return FST_OK;
  }
  fst_status passA(const ConvArgs<double> &a, const Layout &L) override { return passA_t(a, L); }
  fst_status reduce(const ConvArgs<float> &a, const Layout &L) override { return reduce_t(a, L); }
  fst_status reduce(const ConvArgs<double> &a, const Layout &L) override { return reduce_t(a, L); }
  fst_status passB(const ConvArgs<float> &a, const Layout &L) override {
    if (a.two_spec && !((L.fast || L.big) && L.log2Q == 12))
      return fail(FST_EINVAL, "two-spectrum row pass needs 4096-point rows");
    if ((L.fast || L.big) && L.log2Q == 13 && a.tw8) {
      TRY(set_attrs());
      dim3 grid((unsigned)(1u << L.log2P), (unsigned)a.npairs);
      PROF("k_fastB8192", a.npairs, (k_fastB8192<<<grid, 512, fastb8192_smem(), cur>>>(a, a.tw8)));
      LAUNCHED("k_fastB8192");
      return FST_OK;
    }
    if (!(L.fast || L.big) || L.log2Q != 12) return passB_t(a, L);
    if (a.two_spec) {
      if (!a.rp || a.cplx || a.mode != MODE_CONV)
        return fail(FST_EINVAL, "two-spectrum row pass needs real ragged slots");
      TRY(set_attrs());
      dim3 grid((unsigned)((1u << L.log2P) / 2 + 1), (unsigned)a.npairs);
      PROF("k_fastB4096_2s", a.npairs, (k_fastB4096_2s<<<grid, 256, fastb2s_smem(), cur>>>(a)));
      LAUNCHED("k_fastB4096_2s");
      return FST_OK;
    }
    dim3 grid((unsigned)(1u << L.log2P), (unsigned)a.npairs);
    PROF("k_fastB4096", a.npairs, (k_fastB4096<<<grid, 256, 0, cur>>>(a)));
    LAUNCHED("k_fastB4096");
    return FST_OK;
  }
  fst_status passB(const ConvArgs<double> &a, const Layout &L) override { return passB_t(a, L); }
  // Tile sizes: a block of 512 values (four warps, one per sub-core) once that makes two blocks per
  // SM; otherwise as small as 128 values (one warp), so that a single short signal spreads over
  // more SMs.  One pair of N = 4096: 39.7 us; with 512-value tiles 41.5.
  fst_status f64_passes(const ConvArgs<double> &a, int spec_log2P, int pass) override {
    TRY(set_attrs());
    F64Args f{a, spec_log2P, 0, 0};
    const int P = 1 << a.log2P, Q = 1 << a.log2Q;
    const int64_t vals = a.npairs << a.log2M;
    int tile = vals >= 512LL * 2 * sms ? 512 : 128;
    if (pass == 1 && a.log2Q >= 11 && spec_log2P == a.log2P) {
      dim3 grid((unsigned)P, (unsigned)a.npairs);
      PROF("k_passB<f64>", a.npairs, (k_passB<double><<<grid, Q / 16, padded_size(Q) * 16, cur>>>(a)));
      LAUNCHED("k_passB");
      return FST_OK;
    }
    auto lg = [](int v) { int l = 0; while ((2 << l) <= v) ++l; return l; };
    if (pass == 1) {
      f.log2RT = lg(std::max(1, std::min(P, tile / Q)));
      const int64_t blocks = (a.npairs * P) >> f.log2RT;
      PROF("k_f64B", a.npairs, (k_f64B<<<(unsigned)blocks, (Q << f.log2RT) / 4, ((size_t)Q << f.log2RT) * 16, cur>>>(f)));
      LAUNCHED("k_f64B");
      return FST_OK;
    }
    f.log2NB = lg(std::min(Q, tile / P));
    const int64_t blocks = a.npairs * (Q >> f.log2NB);
    const size_t smem = ((size_t)P << f.log2NB) * 16;
    if (pass == 0) PROF("k_f64A", a.npairs, (k_f64A<<<(unsigned)blocks, (P << f.log2NB) / 4, smem, cur>>>(f)));
    else PROF("k_f64C", a.npairs, (k_f64C<<<(unsigned)blocks, (P << f.log2NB) / 4, smem, cur>>>(f)));
    LAUNCHED("k_f64A/C");
    return FST_OK;
  }
  fst_status f64_corr(const ConvArgs<double> &a, const unsigned char *cpar, int64_t rows, int chunk, double *part,
                      double *acoef) override {
    const int64_t H = (a.N + 1) / 2;
    const int nchunk = (int)((H + chunk - 1) / chunk);
    const int64_t rg = (rows + F64_RG - 1) / F64_RG;
    if (rg > 65535 || (rows * a.r + 7) / 8 >= (1LL << 31)) return fail(FST_EINVAL, "batch too large for the FP64 correction");
    PROF("k_f64_corr", rows, (k_f64_corr<<<dim3((unsigned)nchunk, (unsigned)rg), 256, 0, cur>>>(a, cpar, chunk, rows, part)));
    LAUNCHED("k_f64_corr");
    PROF("k_f64_reduce", rows, (k_f64_reduce<<<(unsigned)((rows * a.r + 7) / 8), 256, 0, cur>>>(a, nchunk, rows, part, acoef)));
    LAUNCHED("k_f64_reduce");
    return FST_OK;
  }
  fst_status f64_z(const ConvArgs<double> &a, const unsigned char *cpar, int64_t rows, const double *acoef) override {
    const int64_t H = (a.N + 1) / 2;
    dim3 grid((unsigned)((H + F64_ZN - 1) / F64_ZN), (unsigned)((rows + F64_ZR - 1) / F64_ZR));
    PROF("k_f64_z", rows, (k_f64_z<<<grid, F64_ZN * F64_ZR, 0, cur>>>(a, cpar, rows, acoef)));
    LAUNCHED("k_f64_z");
    return FST_OK;
  }
  fst_status corr_c(const ConvArgs<float> &a) override {
    FastArgs f{a, a.ST_hl};
    dim3 grid((unsigned)((a.N + CORR_BLOCK - 1) / CORR_BLOCK), (unsigned)((a.npairs + FAST_G - 1) / FAST_G));
    PROF("k_corr_c", a.npairs, (k_corr_c<<<grid, FAST_THREADS, 0, cur>>>(f)));
    LAUNCHED("k_corr_c");
    return FST_OK;
  }
  fst_status tc_prep(const float *ST, int64_t N, int rpad, int r, int nB, int64_t Npad, float *STt) override {
    // plan time (never inside a stream capture): kernel attributes and the error word
    TRY(set_attrs());
    if (!tc_err_h) {
      CU(cudaHostAlloc((void **)&tc_err_h, sizeof(int), cudaHostAllocMapped), "cudaHostAlloc");
      *(volatile int *)tc_err_h = 0;
      CU(cudaHostGetDevicePointer((void **)&tc_err, tc_err_h, 0), "cudaHostGetDevicePointer");
    }
    k_tc_prep<<<grid_for((int64_t)nB * Npad, 256), 256, 0, s>>>(ST, N, rpad, r, nB, Npad, STt);
    LAUNCHED("k_tc_prep");
    return FST_OK;
  }
  fst_status corr_tc(const ConvArgs<float> &a) override {
    if (!tc_err) return fail(FST_EUNSUPPORTED, "tcgen05 correction used before its plan-time set-up");
    CUtensorMap mY, mS;
    // y in 128-byte swizzled boxes: 32 floats of 128 rows (real) or of 64 complex rows
    if (a.cplx)
      TRY(encode_2d(&mY, a.y, 2 * (uint64_t)a.N, (uint64_t)a.batch, (uint64_t)a.ld * 8, TC_KT, TC_M / 2, true));
    else
      TRY(encode_2d(&mY, a.y, (uint64_t)a.N, (uint64_t)a.batch, (uint64_t)a.ld * 4, TC_KT, TC_M, true));
    TRY(encode_2d(&mS, a.STt, (uint64_t)a.N, (uint64_t)a.tc_nB, (uint64_t)a.tc_Npad * 4, TC_KT, (uint32_t)a.tc_nB,
                  true));
    TcArgs t{};
    t.N = a.N;
    t.rows = a.batch;
    t.cplx = a.cplx;
    t.nB = a.tc_nB;
    t.r = a.r;
    t.rpad = a.rpad;
    t.ktiles = (int)((a.N + TC_KT - 1) / TC_KT);
    t.nks = tc_slices(a.N);
    const int64_t rb = a.cplx ? (a.batch + TC_M / 2 - 1) / (TC_M / 2) : (a.batch + TC_M - 1) / TC_M;
    if ((int64_t)t.nks * rb >= (1LL << 31)) return fail(FST_EINVAL, "batch too large for the tcgen05 correction");
    t.nitems = (int)(t.nks * rb);
    t.part = a.part;
    t.err = tc_err;
    t.timeout_ns = TC_TIMEOUT_NS;
    t.stall = 0;
    if (tc_stall_take()) {
      t.stall = 1;
      t.timeout_ns = g_tc_stall_limit_ns;
    }
    // persistent: one CTA per SM walks the items
    dim3 grid((unsigned)std::min<int64_t>(t.nitems, sms));
    const size_t smem = (size_t)tc_smem_bytes(t.nB);
    switch (t.nB) {
      case 32: PROF("k_corr_tc", a.npairs, (k_corr_tc<32><<<grid, TC_THREADS, smem, cur>>>(mY, mS, t))); break;
      case 64: PROF("k_corr_tc", a.npairs, (k_corr_tc<64><<<grid, TC_THREADS, smem, cur>>>(mY, mS, t))); break;
      case 96: PROF("k_corr_tc", a.npairs, (k_corr_tc<96><<<grid, TC_THREADS, smem, cur>>>(mY, mS, t))); break;
      case 128: PROF("k_corr_tc", a.npairs, (k_corr_tc<128><<<grid, TC_THREADS, smem, cur>>>(mY, mS, t))); break;
      default: return fail(FST_EINVAL, "tcgen05 correction width out of range");
    }
    LAUNCHED("k_corr_tc");
    return FST_OK;
  }
  fst_status rcorr(const RSig *sigs, int nsig, const RItem *items, int nitems, int cplx, float *part,
                   float *acoef) override {
    if (nitems <= 0) return FST_OK;
    TRY(set_attrs());
    PROF("k_rcorr_part", nitems, (k_rcorr_part<<<(unsigned)nitems, 256, rcorr_smem(), cur>>>(sigs, items, cplx, part)));
    LAUNCHED("k_rcorr_part");
    PROF("k_rcorr_reduce", nsig, (k_rcorr_reduce<<<(unsigned)nsig, 128, 0, cur>>>(sigs, part, acoef)));
    LAUNCHED("k_rcorr_reduce");
    return FST_OK;
  }
  fst_status rzadd(const RSig *sigs, const RItem *items, int nitems, int cplx, const float *acoef) override {
    if (nitems <= 0) return FST_OK;
    PROF("k_rzadd", nitems, (k_rzadd<<<(unsigned)nitems, 256, 0, cur>>>(sigs, items, cplx, acoef)));
    LAUNCHED("k_rzadd");
    return FST_OK;
  }
  // chunks of S_T^T y: about three blocks per SM in all (two are resident), at least a tile each, and
  // no more partials than the scratch of the other forms holds (CORR_BLOCK samples each)
  int sym_chunks(const ConvArgs<float> &a) override {
    const int64_t rows = a.rows_all;
    const int64_t groups = (rows + sy_rows(rows) - 1) / sy_rows(rows), tiles = ((a.N + 1) / 2 + SY_TN - 1) / SY_TN;
    if (groups > 65535 || a.N < 4 * SY_TN) return 0;
    const int64_t most = std::max<int64_t>((a.N + CORR_BLOCK - 1) / CORR_BLOCK, tc_slices(a.N));
    // ... and more where a thread would otherwise add more than 108 products in a row, as far as those
    // partials go: up to 64 columns that bound holds, above it the chains reach 16 tiles (192 products at
    // r = 76, 384 at most).  (At powers of two the resulting blocks are also whole waves of the 304 resident
    // ones: 16 rows of 2^22, 1214 chunks 240 us, 1024 chunks of 128 products 246.)
    const int ntile = sy_tiles(a.ncord, a.r - a.ncord) * (sy_rows(rows) / 8), kg = ntile < 16 ? 16 : 256 / ntile;
    const int64_t want = std::max<int64_t>(3 * (int64_t)sms / groups, (tiles * ((SY_TN / 4 + kg - 1) / kg) * 4 + 107) / 108);
    return (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(tiles, most), want));
  }
  fst_status sym_c(const ConvArgs<float> &a) override {
    TRY(set_attrs());
    const int64_t rows = a.cplx ? 2 * a.batch : a.batch;
    const int RB = sy_rows(a.rows_all);
    dim3 grid((unsigned)a.nkb, (unsigned)((rows + RB - 1) / RB));
    const size_t smem = sy_smem(a.ncord, a.r - a.ncord, RB);
    auto go = [&](auto kernel) { PROF("k_sym_c", a.npairs, (kernel<<<grid, 256, smem, cur>>>(a, a.cord, a.ncord, a.nkb))); };
    // products in a row per thread (sym_chunks)
    const int ntile = sy_tiles(a.ncord, a.r - a.ncord) * (RB / 8), kg = ntile < 16 ? 16 : 256 / ntile;
    const int64_t tiles = ((a.N + 1) / 2 + SY_TN - 1) / SY_TN;
    const bool quad = RB == 8 && (tiles + a.nkb - 1) / a.nkb * ((SY_TN / 4 + kg - 1) / kg) * 4 > 64;
    if (quad) go(a.cplx ? k_sym_c<true, 8, true> : k_sym_c<false, 8, true>);
    else if (a.cplx) go(RB == 8 ? k_sym_c<true, 8> : RB == 16 ? k_sym_c<true, 16> : k_sym_c<true, 32>);
    else go(RB == 8 ? k_sym_c<false, 8> : RB == 16 ? k_sym_c<false, 16> : k_sym_c<false, 32>);
    LAUNCHED("k_sym_c");
    return FST_OK;
  }
  fst_status sym_z(const ConvArgs<float> &a) override {
    TRY(set_attrs());
    const int64_t rows = a.cplx ? 2 * a.batch : a.batch, H = (a.N + 1) / 2;
    const int ng = sy_ng(rows);
    const int64_t rg = (rows + SY_R * ng - 1) / (SY_R * ng);
    // blocks of 64 threads where those of 256 would leave SMs idle (one row of N = 70001: 35 blocks)
    const int thr = (H * ng + 1023) / 1024 * rg < sms ? 64 : 256, ns = thr / ng;
    if (rg > 65535) return fail(FST_EINVAL, "batch too large for the correction pass");
    dim3 grid((unsigned)((H + 4 * ns - 1) / (4 * ns)), (unsigned)rg);
    const size_t smem = (size_t)a.r * (SY_R * ng + 1) * sizeof(float);
    const bool vec = a.N % 4 == 0 && ((uintptr_t)a.out % 16) == 0 && (a.ld * (a.cplx ? 8 : 4)) % 16 == 0;
    if (vec) PROF("k_sym_z", a.npairs, (k_sym_z<true><<<grid, thr, smem, cur>>>(a, a.cord, a.ncord)));
    else PROF("k_sym_z", a.npairs, (k_sym_z<false><<<grid, thr, smem, cur>>>(a, a.cord, a.ncord)));
    LAUNCHED("k_sym_z");
    return FST_OK;
  }
  fst_status corr_cc(const ConvArgs<float> &a) override {
    TRY(set_attrs());
    PROF("k_corr_cc", a.npairs,
         (k_corr_cc<<<(unsigned)((a.N + CORR_BLOCK - 1) / CORR_BLOCK), CC_THREADS, cc_smem(a.rpad), cur>>>(a)));
    LAUNCHED("k_corr_cc");
    return FST_OK;
  }
  fst_status corr_reduce(const ConvArgs<float> &a, const float *scale) override {
    dim3 grid((unsigned)a.npairs, (unsigned)((2 * a.r + 7) / 8));
    PROF("k_corr_reduce", a.npairs, (k_corr_reduce<<<grid, 256, 0, cur>>>(a, scale)));
    LAUNCHED("k_corr_reduce");
    return FST_OK;
  }
  fst_status corr_z(const ConvArgs<float> &a) override {
    FastArgs f{a, a.ST_hl};
    dim3 grid((unsigned)((a.N + CORR_ROWS - 1) / CORR_ROWS), (unsigned)((a.npairs + FAST_G - 1) / FAST_G));
    PROF("k_corr_z", a.npairs, (k_corr_z<<<grid, FAST_THREADS, 0, cur>>>(f)));
    LAUNCHED("k_corr_z");
    return FST_OK;
  }
  fst_status passC(const ConvArgs<float> &a, const Layout &L) override {
    if (L.big) {
      switch (L.P2) {
        case 2: return colC_t<2>(a, L);
        case 4: return colC_t<4>(a, L);
        case 8: return colC_t<8>(a, L);
        case 16: return colC_t<16>(a, L);
        case 32: return colC_t<32>(a, L);
        default: return fail(FST_EINVAL, "column pass width out of range");
      }
    }
    if (!L.fast) return passC_t(a, L);
    FastArgs f{a, a.ST_hl};
    dim3 grid((unsigned)L.ntiles, (unsigned)((a.npairs + FAST_G - 1) / FAST_G));
    const int P = 1 << L.log2P;
    if (P == 32) PROF("k_fastC<32>", a.npairs, (k_fastC<32><<<grid, FAST_THREADS, 0, cur>>>(f)));
    else if (P == 16) PROF("k_fastC<16>", a.npairs, (k_fastC<16><<<grid, FAST_THREADS, 0, cur>>>(f)));
    else PROF("k_fastC<8>", a.npairs, (k_fastC<8><<<grid, FAST_THREADS, 0, cur>>>(f)));
    LAUNCHED("k_fastC");
    return FST_OK;
  }
  fst_status passC(const ConvArgs<double> &a, const Layout &L) override { return passC_t(a, L); }

  fst_status bisect_ms_many(const TargetDesc *td, int nt, int warps, int rounds, const double *dcat,
                            const double *e2cat, double *iv, int *cnt, double *theta, int *flag) override {
    if (nt <= 0) return FST_OK;
    for (int r = 0; r <= rounds; ++r) {
      const int last = r == rounds;
      PROF_S(s, "k_bisect_round", nt, (k_bisect_round<<<(nt * warps * 32 + BISECT_THREADS - 1) / BISECT_THREADS, BISECT_THREADS, 0, s>>>(td, nt, warps, r, !last, dcat, e2cat, iv, cnt, theta, flag)));
      LAUNCHED("k_bisect_round");
    }
    return FST_OK;
  }
  fst_status bisect_many(const TargetDesc *td, int nt, const double *dcat, const double *e2cat, double *theta,
                         int *flag) override {
    // one warp per block: the targets spread over every SM (each one's FP64 pipe is the limit)
    PROF_S(s, "k_bisect_many", nt, (k_bisect_many<<<(nt + 31) / 32, 32, 0, s>>>(td, nt, dcat, e2cat, theta, flag)));
    LAUNCHED("k_bisect_many");
    return FST_OK;
  }
  fst_status fwdvec_many(const TargetDesc *td, int nt, const double *dcat, const double *ecat, const double *rcat,
                         const double *theta, double *z, double *w, int *ex, double *delta) override {
    // spread over the SMs: a warp's FP64 instruction takes its SM's pipe equally long with any
    // number of active lanes
    const int lanes = std::max(1, std::min(32, (nt + sms - 1) / sms));
    PROF_S(s, "k_fwdvec_many", nt, (k_fwdvec_many<<<(nt + lanes - 1) / lanes, 32, 0, s>>>(td, nt, lanes, dcat, ecat, rcat, theta, z, w, ex, delta)));
    LAUNCHED("k_fwdvec_many");
    return FST_OK;
  }
  fst_status finalize_many(const TargetDesc *td, int nt, const double *z, const double *w, const int *ex,
                           const double *delta) override {
    PROF_S(s, "k_finalize_many", nt, (k_finalize_many<<<nt, 256, 0, s>>>(td, z, w, ex, delta)));
    LAUNCHED("k_finalize_many");
    return FST_OK;
  }
  fst_status dot(const double *a, const double *b, int64_t N, int nvec, double *out) override {
    k_dot<<<nvec, 256, 0, s>>>(a, b, N, out);
    LAUNCHED("k_dot");
    return FST_OK;
  }
  fst_status sinc_embed(double *c, int64_t N, int64_t M, double W) override {
    k_sinc<<<grid_for(M, 256), 256, 0, s>>>(c, N, M, W);
    LAUNCHED("k_sinc");
    return FST_OK;
  }
  fst_status spec_store(const double2 *X, const Layout &L64, const Layout &L32, int64_t M, double scale,
                        double *spec64, float *spec32) override {
    k_spec_store<<<grid_for(M, 256), 256, 0, s>>>(X, L64, L32, M, scale, spec64, spec32);
    LAUNCHED("k_spec_store");
    return FST_OK;
  }
  fst_status gather_ST(const double *S, int64_t N, const int *sel, int r, int rpad, double *ST64,
                       float *ST32) override {
    k_gather<<<grid_for(N * rpad, 256), 256, 0, s>>>(S, N, sel, r, rpad, ST64, ST32);
    LAUNCHED("k_gather");
    return FST_OK;
  }
  template <typename T> fst_status coef_lowrank_t(const CoefArgs<T> &a) {
    const size_t smem = (size_t)COEF_RED_WORDS * sizeof(T);
    dim3 grid((unsigned)a.nchunks, (unsigned)a.batch);
    PROF("k_coef_lowrank", 0, (k_coef_lowrank<T><<<grid, COEF_THREADS, smem, cur>>>(a)));
    LAUNCHED("k_coef_lowrank");
    return FST_OK;
  }
  // one block per SM over the vector groups; two tile buffers in shared memory
  int lowrank_plan(int64_t N, int rH, int DA, int DB, int64_t nvc, size_t *scratch) override {
    const int64_t groups = (nvc + LR_VC - 1) / LR_VC, tiles = N / 2 / LR_TN;
    const LrShape sh = lr_shape(rH, DA, DB, (int)std::min<int64_t>(nvc, LR_VC));
    const LrShape s1 = lr_shape(rH, DA, DB, 1);
    if (N < 2 * LR_TN || groups > 65535 || sh.kg < 1 || s1.kg < 1 || std::max(lr_smem(sh), lr_smem(s1)) > 227 * 1024)
      return 0;
    const int64_t n = std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)sms / groups));
    *scratch = (size_t)(n * groups) * 64 * 256 * sizeof(float) + 256;
    return (int)n;
  }
  fst_status coef_gemm(const CoefArgs<float> &a, void *scratch) override {
    TRY(set_attrs());
    const int64_t nvc = a.cplx ? 2 * a.batch : a.batch;
    size_t smem = 0;
    for (int v : {(int)std::min<int64_t>(nvc, LR_VC), (int)(nvc % LR_VC)})
      if (v > 0) smem = std::max(smem, lr_smem(lr_shape(a.rH, a.DA, a.DB, v)));
    dim3 grid((unsigned)a.nchunks, (unsigned)((nvc + LR_VC - 1) / LR_VC));
    PROF("k_coef_gemm", 0, (k_coef_gemm<<<grid, 512, smem, cur>>>(a, a.nchunks, (float *)scratch)));
    LAUNCHED("k_coef_gemm");
    return FST_OK;
  }
  // vectors a thread: one, from 16 vectors two, from 32 four, but only as many as leave two blocks for
  // every SM, in number and in shared memory (more of them share the columns' loads, fewer spread the
  // batch).  us at N = 4096, eps = 1e-6, one / two / four: 64 vectors 35.0 / 34.9 / 41.1, 128 47.2 / 41.1 /
  // 43.1, 256 69.8 / 59.5 / 54.8; N = 128, 64 vectors 24.7 / 27.1 / 32.9; N = 32768, eps = 1e-10 (four: one
  // block per SM), 64 vectors 116 / 101 / 119
  int exp_spt(int64_t N, int rH, int DA, int DB, int r, int64_t nsig) const {
    const int64_t tiles = N / 2 / LR_TN;
    int spt = nsig >= 32 ? 4 : (nsig >= 16 ? 2 : 1);
    while (spt > 1 && (tiles * ((nsig + 4 * spt - 1) / (4 * spt)) <= 2 * sms ||
                       2 * exp_smem(rH, DA, DB, r, spt) > 226 * 1024))
      spt /= 2;
    return spt;
  }
  static size_t exp_smem(int rH, int DA, int DB, int r, int spt) {
    return (size_t)8 * spt * xp_words(rH, DA, DB, r) * 8 + (size_t)LR_TN * xp_cs(rH, DA, DB, r) * 4;
  }
  size_t expand_scratch(int64_t N, int rH, int DA, int DB, int r, int64_t nsig) override {
    // few short vectors with few columns: the generic kernel, one launch less (us, generic / shared columns:
    // N = 128, rH = 7, 64 vectors 20.6 / 22.6; N = 256, rH = 8, 16 20.6 / 22.6; N = 1024, rH = 7, 64 24.7 / 26.7;
    // but N = 256, rH = 8, 256 vectors 24.7 / 22.6; N = 1024, rH = 9, 64 28.8 / 26.7)
    if (N <= 1024 && rH <= 8 && nsig * rH <= 1024) return 0;
    if (N < 2 * LR_TN || exp_smem(rH, DA, DB, r, 4) > 227 * 1024) return 0;
    return (size_t)nsig * xp_words(rH, DA, DB, r) * 8 + 256;
  }
  fst_status expand_gemm(const ExpArgs<float> &a, int64_t nsig, void *scratch, const unsigned char *cpar) override {
    TRY(set_attrs());
    float2 *cc = (float2 *)scratch;
    const int nw = xp_words(a.rH, a.DA, a.DB, a.r), spt = exp_spt(a.N, a.rH, a.DA, a.DB, a.r, nsig);
    PROF("k_exp_prep", nsig, (k_exp_prep<<<grid_for(nsig * nw, 256), 256, 0, cur>>>(a, nsig, cc)));
    LAUNCHED("k_exp_prep");
    // vectors split until there are about four blocks per SM, in whole rounds of 8 spt vectors
    const int64_t tiles = a.N / 2 / LR_TN, rounds = (nsig + 8 * spt - 1) / (8 * spt);
    const int64_t split = std::max<int64_t>(1, std::min<int64_t>(rounds, 8 * (int64_t)sms / tiles));
    dim3 grid((unsigned)tiles, (unsigned)split);
    const size_t smem = exp_smem(a.rH, a.DA, a.DB, a.r, spt);
    if (spt == 4) PROF("k_expand_gemm", nsig, (k_expand_gemm<4><<<grid, 256, smem, cur>>>(a, nsig, cc, cpar)));
    else if (spt == 2) PROF("k_expand_gemm", nsig, (k_expand_gemm<2><<<grid, 256, smem, cur>>>(a, nsig, cc, cpar)));
    else PROF("k_expand_gemm", nsig, (k_expand_gemm<1><<<grid, 256, smem, cur>>>(a, nsig, cc, cpar)));
    LAUNCHED("k_expand_gemm");
    return FST_OK;
  }
  template <typename T> fst_status coef_st_t(const CoefArgs<T> &a) {
    const size_t smem = (COEF_THREADS / 32) * 128 * sizeof(T);
    dim3 grid((unsigned)a.nchunks, (unsigned)a.batch);
    PROF("k_coef_st", 0, (k_coef_st<T><<<grid, COEF_THREADS, smem, cur>>>(a)));
    LAUNCHED("k_coef_st");
    return FST_OK;
  }
  template <typename T> fst_status coef_reduce_t(const T *part, int nchunks, int nout, int64_t batch, T *tot) {
    dim3 grid((unsigned)((nout + 127) / 128), (unsigned)batch);
    PROF("k_coef_reduce", 0, (k_coef_reduce<T><<<grid, 128, 0, cur>>>(part, nchunks, nout, tot)));
    LAUNCHED("k_coef_reduce");
    return FST_OK;
  }
  template <typename T>
  fst_status coef_gather_t(const c2<T> *X, const Layout &Lf, int64_t N, int cplx, int64_t sig0, int64_t nsig,
                           int64_t h, c2<T> *out, int64_t Kp) {
    if (sizeof(T) == 4 && (Lf.fast || Lf.big)) {
      const int P = 1 << Lf.log2P;
      dim3 grid((unsigned)(((1u << Lf.log2Q) / 32) * (P / std::min(P, 32))), (unsigned)(cplx ? nsig : (nsig + 1) / 2));
      PROF("k_coef_gather_t", 0, (k_coef_gather_t<<<grid, 256, 0, cur>>>((const float2 *)X, Lf.log2P, Lf.log2Q, cplx, sig0, nsig, h, (float2 *)out, Kp)));
      LAUNCHED("k_coef_gather_t");
      return FST_OK;
    }
    PROF("k_coef_gather", 0, (k_coef_gather<T><<<grid_for(nsig * (2 * h + 1), 256), 256, 0, cur>>>(X, Lf, N, cplx, sig0, nsig, h, out, Kp)));
    LAUNCHED("k_coef_gather");
    return FST_OK;
  }
  template <typename T>
  fst_status coef_mix_t(const CoefArgs<T> &a, const T *tot, const T *totU, const T *CA, const T *CB, const T *sq,
                        c2<T> *out, int64_t Kp, int64_t nF) {
    const int nfin = 4 * a.rH + 2 * a.DA + 2 * a.DB + a.r;
    dim3 grid((unsigned)((nfin + 127) / 128), (unsigned)a.batch);
    PROF("k_coef_mix", 0, (k_coef_mix<T><<<grid, 128, 0, cur>>>(a, tot, totU, CA, CB, sq, out, Kp, nF)));
    LAUNCHED("k_coef_mix");
    return FST_OK;
  }
  template <typename T> fst_status exp_scatter_t(const ExpArgs<T> &a, int64_t nsig, c2<T> *Xs) {
    PROF("k_exp_scatter", nsig, (k_exp_scatter<T><<<grid_for(nsig * a.N, 256), 256, 0, cur>>>(a, nsig, Xs)));
    LAUNCHED("k_exp_scatter");
    return FST_OK;
  }
  template <typename T> fst_status expand_t(const ExpArgs<T> &a, int64_t nsig) {
    const int64_t blocks = nsig * ((a.N + EXP_E * 256 - 1) / (EXP_E * 256));
    PROF("k_expand", nsig, (k_expand<T><<<(unsigned)std::min<int64_t>(blocks, 152 * 64), 256, 0, cur>>>(a, nsig)));
    LAUNCHED("k_expand");
    return FST_OK;
  }
  fst_status exp_scatter(const ExpArgs<float> &a, int64_t nsig, float2 *Xs) override { return exp_scatter_t(a, nsig, Xs); }
  fst_status exp_scatter(const ExpArgs<double> &a, int64_t nsig, double2 *Xs) override { return exp_scatter_t(a, nsig, Xs); }
  fst_status expand(const ExpArgs<float> &a, int64_t nsig) override { return expand_t(a, nsig); }
  fst_status expand(const ExpArgs<double> &a, int64_t nsig) override { return expand_t(a, nsig); }
  fst_status coef_lowrank(const CoefArgs<float> &a) override { return coef_lowrank_t(a); }
  fst_status coef_lowrank(const CoefArgs<double> &a) override { return coef_lowrank_t(a); }
  fst_status coef_st(const CoefArgs<float> &a) override { return coef_st_t(a); }
  fst_status coef_st(const CoefArgs<double> &a) override { return coef_st_t(a); }
  fst_status coef_reduce(const float *part, int nchunks, int nout, int64_t batch, float *tot) override {
    return coef_reduce_t(part, nchunks, nout, batch, tot);
  }
  fst_status coef_reduce(const double *part, int nchunks, int nout, int64_t batch, double *tot) override {
    return coef_reduce_t(part, nchunks, nout, batch, tot);
  }
  fst_status coef_gather(const float2 *X, const Layout &Lf, int64_t N, int cplx, int64_t sig0, int64_t nsig,
                         int64_t h, float2 *out, int64_t Kp) override {
    return coef_gather_t<float>(X, Lf, N, cplx, sig0, nsig, h, out, Kp);
  }
  fst_status coef_gather(const double2 *X, const Layout &Lf, int64_t N, int cplx, int64_t sig0, int64_t nsig,
                         int64_t h, double2 *out, int64_t Kp) override {
    return coef_gather_t<double>(X, Lf, N, cplx, sig0, nsig, h, out, Kp);
  }
  fst_status coef_mix(const CoefArgs<float> &a, const float *tot, const float *totU, const float *CA, const float *CB,
                      const float *sq, float2 *out, int64_t Kp, int64_t nF) override {
    return coef_mix_t(a, tot, totU, CA, CB, sq, out, Kp, nF);
  }
  fst_status coef_mix(const CoefArgs<double> &a, const double *tot, const double *totU, const double *CA,
                      const double *CB, const double *sq, double2 *out, int64_t Kp, int64_t nF) override {
    return coef_mix_t(a, tot, totU, CA, CB, sq, out, Kp, nF);
  }

  fst_status split_tf32(const float *src, float2 *hl, int64_t n) override {
    k_split_tf32<<<grid_for(n, 256), 256, 0, s>>>(src, hl, n);
    LAUNCHED("k_split_tf32");
    return FST_OK;
  }
  fst_status to_f32(const double *src, float *dst, int64_t n) override {
    k_to_f32<<<grid_for(n, 256), 256, 0, s>>>(src, dst, n);
    LAUNCHED("k_to_f32");
    return FST_OK;
  }
};

Runner *make_dev_runner() {
  int n = 0;
  if (cudaGetDeviceCount(&n) != cudaSuccess || n < 1) {
    cudaGetLastError();
    return nullptr;
  }
  DevRunner *R = new DevRunner();
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&R->sms, cudaDevAttrMultiProcessorCount, dev);
  cudaGetLastError();
  if (R->sms < 1) R->sms = 1;
  return R;
}

}  // namespace fst

using namespace fst;

extern "C" long long fst_launch_count(void) { return g_launches; }

// ---------------------------------------------------------------------------
// fst_project_noalloc: fst_project for callers that cannot allocate device memory
// when they project (for example a process whose memory manager owns all device
// memory after start-up).  The four-step path's scratch (intermediate spectra,
// per-tile partial sums and the correction coefficients) lives in one fixed
// file-scope device array instead of the plan's on-demand workspace.  Every device
// that loads this library holds the array until the process exits.
// ---------------------------------------------------------------------------
#define FST_NOALLOC_SCRATCH_BYTES (128ull << 20)
static __device__ __align__(256) unsigned char g_noalloc_scratch[FST_NOALLOC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 128;
std::mutex g_scratch_mu;
void *g_scratch_addr[kMaxDevices] = {};
CUcontext g_scratch_ctx[kMaxDevices] = {};   // context the address was looked up in
// the calling thread's current context (the primary context of the current device,
// re-created after a device reset)
CUcontext current_context() {
  using Fn = CUresult (*)(CUcontext *);
  static Fn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 4000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (Fn)p;
    else
      cudaGetLastError();
  });
  CUcontext c = nullptr;
  if (!fn || fn(&c) != CUDA_SUCCESS) return nullptr;
  return c;
}
}  // namespace

extern "C" fst_status fst_project_noalloc(fst_plan_t p, const void *y, void *out, int64_t batch, int64_t ld,
                                          int dtype, void *stream) {
  if (!p) return fail(FST_EINVAL, "plan is NULL");
  if (!p->R->device()) return fail(FST_EINVAL, "fst_project_noalloc needs a device plan");
  int dev = 0;
  CU(cudaGetDevice(&dev), "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return fail(FST_EUNSUPPORTED, "device ordinal out of range");
  void *scratch = nullptr;
  {
    // set-up per device and context (with that device current): the host-side name of
    // the array is only a stand-in, its device address comes from the runtime; a new
    // context (after a device reset) gets the array at a new address
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    const CUcontext ctx = current_context();
    if (!g_scratch_addr[dev] || !ctx || g_scratch_ctx[dev] != ctx) {
      void *a = nullptr;
      CU(cudaGetSymbolAddress(&a, g_noalloc_scratch), "cudaGetSymbolAddress");
      g_scratch_addr[dev] = a;
      g_scratch_ctx[dev] = current_context();   // the runtime has made its context current
    }
    scratch = g_scratch_addr[dev];
  }
  p->R->set_stream(stream);
  // nothing in the scratch has to start at zero: every kernel writes the part it
  // later reads before reading it
  return run_apply_ws(p, y, out, batch, ld, dtype, true, scratch, (size_t)FST_NOALLOC_SCRATCH_BYTES);
}

extern "C" unsigned long long fst_noalloc_scratch_bytes(void) { return FST_NOALLOC_SCRATCH_BYTES; }

extern "C" fst_status fst_profile_enable(int on) {
  for (auto &r : g_prof) {
    if (r.a) cudaEventDestroy(r.a);
    if (r.b) cudaEventDestroy(r.b);
  }
  g_prof.clear();
  g_prof_on = on ? 1 : 0;
  return FST_OK;
}

extern "C" fst_status fst_profile_read(int i, const char **name, double *ms, long long *units) {
  if (i < 0 || i >= (int)g_prof.size()) return fail(FST_EINVAL, "profile index out of range");
  ProfRec &r = g_prof[i];
  float t = 0.f;
  if (r.a && r.b) {
    cudaError_t e = cudaEventSynchronize(r.b);
    if (e != cudaSuccess) return cuda_fail(e, "event sync");
    e = cudaEventElapsedTime(&t, r.a, r.b);
    if (e != cudaSuccess) return cuda_fail(e, "elapsed");
  }
  if (name) *name = r.name;
  if (ms) *ms = t;
  if (units) *units = r.units;
  return FST_OK;
}

extern "C" int fst_profile_count(void) { return (int)g_prof.size(); }

// ---------------------------------------------------------------------------
// host-buffer entry point: chunks of the batch go host -> device -> host on two
// copy streams while the previous / next chunk is projected on `stream`
// ---------------------------------------------------------------------------
namespace {
constexpr int HP_SLOTS = 4;   // chunks in flight: copy in, compute and copy out overlap freely
struct HostPipe {
  cudaStream_t cin = nullptr, cout = nullptr;
  cudaEvent_t in_done[HP_SLOTS] = {}, comp_done[HP_SLOTS] = {}, out_done[HP_SLOTS] = {};
  void *din[HP_SLOTS] = {}, *dout[HP_SLOTS] = {};
  size_t slot_bytes = 0;
  int dev = -1;
};
thread_local HostPipe *g_pipe = nullptr;
}  // namespace

extern "C" fst_status fst_project_host(fst_plan_t p, const void *y, void *out, int64_t batch, int dtype,
                                       void *stream) {
  if (!p) return fail(FST_EINVAL, "plan is NULL");
  if (batch < 0) return fail(FST_EINVAL, "batch < 0");
  if (batch == 0) return FST_OK;
  if (!y || !out) return fail(FST_EINVAL, "NULL signal pointer");
  if (!p->R->device()) return run_apply(p, y, out, batch, 0, dtype, true);
  size_t esz;
  switch (dtype) {
    case FST_F32: esz = 4; break;
    case FST_F64: esz = 8; break;
    case FST_C64: esz = 8; break;
    case FST_C128: esz = 16; break;
    default: return fail(FST_EINVAL, "unknown dtype");
  }
  const size_t sig_bytes = esz * (size_t)p->N;
  // chunk of the pipeline: FST_HOST_CHUNK_MB (default 64) MiB of signals
  const char *env = getenv("FST_HOST_CHUNK_MB");
  const int64_t chunk_mb = std::max<int64_t>(1, env ? atoll(env) : 64);
  int64_t per = std::max<int64_t>(2, (int64_t)(((size_t)chunk_mb << 20) / sig_bytes));
  per = (per / 2) * 2;
  per = std::min<int64_t>(per, ((batch + 1) / 2) * 2);
  const size_t slot = (size_t)per * sig_bytes;
  int dev = 0;
  CU(cudaGetDevice(&dev), "cudaGetDevice");
  if (!g_pipe || g_pipe->dev != dev || g_pipe->slot_bytes < slot) {
    if (g_pipe) {
      for (int i = 0; i < HP_SLOTS; ++i) {
        cudaFree(g_pipe->din[i]);
        cudaFree(g_pipe->dout[i]);
      }
    } else {
      g_pipe = new HostPipe();
    }
    if (!g_pipe->cin) {
      CU(cudaStreamCreateWithFlags(&g_pipe->cin, cudaStreamNonBlocking), "stream");
      CU(cudaStreamCreateWithFlags(&g_pipe->cout, cudaStreamNonBlocking), "stream");
      for (int i = 0; i < HP_SLOTS; ++i) {
        CU(cudaEventCreateWithFlags(&g_pipe->in_done[i], cudaEventDisableTiming), "event");
        CU(cudaEventCreateWithFlags(&g_pipe->comp_done[i], cudaEventDisableTiming), "event");
        CU(cudaEventCreateWithFlags(&g_pipe->out_done[i], cudaEventDisableTiming), "event");
      }
    }
    for (int i = 0; i < HP_SLOTS; ++i) {
      g_pipe->din[i] = g_pipe->dout[i] = nullptr;
      CU(cudaMalloc(&g_pipe->din[i], slot), "cudaMalloc");
      CU(cudaMalloc(&g_pipe->dout[i], slot), "cudaMalloc");
    }
    g_pipe->slot_bytes = slot;
    g_pipe->dev = dev;
  }
  HostPipe &hp = *g_pipe;
  cudaStream_t sc = (cudaStream_t)stream;
  p->R->set_stream(stream);
  // the copies must not start before earlier work on the compute stream is done
  CU(cudaEventRecord(hp.comp_done[0], sc), "event");
  CU(cudaStreamWaitEvent(hp.cin, hp.comp_done[0], 0), "wait");
  // chunk schedule: a short first chunk (compute starts after less copying), full chunks, and a
  // short last chunk (less copying after the last compute); every chunk but the last has an even
  // size, so real signals pair as in one call over the whole batch
  std::vector<int64_t> sizes;
  const int64_t small = std::max<int64_t>(2, (per / 4) / 2 * 2);
  if (per >= 8 && batch >= 2 * per + 2 * small) {
    const int64_t tail = small + (batch & 1);
    int64_t mid = batch - small - tail;
    sizes.push_back(small);
    while (mid > per) {
      sizes.push_back(per);
      mid -= per;
    }
    if (mid > 0) sizes.push_back(mid);
    sizes.push_back(tail);
  } else {
    for (int64_t b0 = 0; b0 < batch; b0 += per) sizes.push_back(std::min<int64_t>(per, batch - b0));
  }
  int64_t b0 = 0;
  for (size_t i = 0; i < sizes.size(); b0 += sizes[i], ++i) {
    const int k = (int)(i % HP_SLOTS);
    const int64_t nb = sizes[i];
    const size_t bytes = (size_t)nb * sig_bytes;
    if (i >= (size_t)HP_SLOTS) CU(cudaStreamWaitEvent(hp.cin, hp.out_done[k], 0), "wait");
    CU(cudaMemcpyAsync(hp.din[k], (const char *)y + b0 * sig_bytes, bytes, cudaMemcpyHostToDevice, hp.cin), "h2d");
    CU(cudaEventRecord(hp.in_done[k], hp.cin), "event");
    CU(cudaStreamWaitEvent(sc, hp.in_done[k], 0), "wait");
    fst_status s = run_apply(p, hp.din[k], hp.dout[k], nb, 0, dtype, true, batch);
    if (s != FST_OK) return s;
    CU(cudaEventRecord(hp.comp_done[k], sc), "event");
    CU(cudaStreamWaitEvent(hp.cout, hp.comp_done[k], 0), "wait");
    CU(cudaMemcpyAsync((char *)out + b0 * sig_bytes, hp.dout[k], bytes, cudaMemcpyDeviceToHost, hp.cout), "d2h");
    CU(cudaEventRecord(hp.out_done[k], hp.cout), "event");
  }
  CU(cudaStreamSynchronize(hp.cout), "sync");
  CU(cudaStreamSynchronize(sc), "sync");
  return p->R->device_status(false);
}

// ---------------------------------------------------------------------------
// fst_project_ragged: the first call with a given (plans, signals) signature runs
// directly (allocating what it needs), the second records the whole batch into a
// CUDA graph, later ones replay it.
// ---------------------------------------------------------------------------
namespace {
struct RaggedCtx {
  std::vector<const void *> sig;
  std::vector<fst_plan_t> plans;   // the batch's plans, in call order
  std::vector<uint64_t> gens;      // their workspace generations when the graph was recorded
  fst::RaggedState state;          // descriptor arrays and workspaces (cudaMalloc), launch choices
  cudaGraphExec_t exec = nullptr;
  long long nodes = 0;
  int seen = 0;
};
std::recursive_mutex g_ragged_mu;
std::vector<RaggedCtx *> g_ragged;
// frees a context after every launch that may still use it has finished
void free_ctx(RaggedCtx *c) {
  cudaDeviceSynchronize();
  if (c->exec) cudaGraphExecDestroy(c->exec);
  for (void *b : c->state.bufs) cudaFree(b);
  delete c;
}
bool ctx_current(const RaggedCtx *c) {
  for (size_t i = 0; i < c->plans.size(); ++i)
    if (c->plans[i]->ws_gen != c->gens[i]) return false;
  return true;
}
cudaStream_t g_ragged_cap = nullptr;
bool ragged_graphs_enabled() {
  const char *s = getenv("FST_GRAPHS");
  return !(s && s[0] == '0');
}
}  // namespace

extern "C" fst_status fst_project_ragged(const fst_plan_t *plans, const void *const *y, void *const *out,
                                         int64_t count, int dtype, void *stream) {
  if (count < 0 || (count > 0 && (!plans || !y || !out))) return fail(FST_EINVAL, "bad arguments");
  if (count == 0) return FST_OK;
  for (int64_t i = 0; i < count; ++i)
    if (!plans[i]) return fail(FST_EINVAL, "NULL plan");
  if (!plans[0]->R->device()) {
    RaggedState rs;
    fst_status st = run_ragged(plans, y, out, count, dtype, rs);
    for (void *b : rs.bufs) plans[0]->R->release(b);
    return st;
  }
  std::lock_guard<std::recursive_mutex> lk(g_ragged_mu);
  std::vector<const void *> sig;
  sig.reserve(3 * count + 1);
  sig.push_back((const void *)(intptr_t)dtype);
  for (int64_t i = 0; i < count; ++i) {
    sig.push_back(plans[i]);
    sig.push_back(y[i]);
    sig.push_back(out[i]);
  }
  RaggedCtx *ctx = nullptr;
  for (RaggedCtx *c : g_ragged)
    if (c->sig == sig) ctx = c;
  cudaStream_t us = (cudaStream_t)stream;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(us, &cs) != cudaSuccess) {
    cudaGetLastError();
    cs = cudaStreamCaptureStatusActive;
  }
  const bool graphs = ragged_graphs_enabled() && !profiling_enabled() && cs == cudaStreamCaptureStatusNone;
  if (ctx && ctx->exec && !ctx_current(ctx)) {
    // a plan's workspace moved since the recording: run directly, record again next time
    cudaDeviceSynchronize();
    cudaGraphExecDestroy(ctx->exec);
    ctx->exec = nullptr;
    ctx->seen = 0;
  }
  if (ctx && ctx->exec && graphs) {
    CU(cudaGraphLaunch(ctx->exec, us), "cudaGraphLaunch");
    g_launches += ctx->nodes;
    return FST_OK;
  }
  if (!ctx) {
    if (g_ragged.size() >= 4) {
      free_ctx(g_ragged.front());
      g_ragged.erase(g_ragged.begin());
    }
    ctx = new RaggedCtx();
    ctx->sig = sig;
    ctx->plans.assign(plans, plans + count);
    ctx->state.records = ragged_graphs_enabled();
    g_ragged.push_back(ctx);
  }
  for (int64_t i = 0; i < count; ++i) plans[i]->R->set_stream(stream);
  if (ctx->seen == 0 || !graphs) {
    ctx->seen = 1;
    return run_ragged(plans, y, out, count, dtype, ctx->state);
  }
  // second call: record the batch into a graph on a private stream
  if (!g_ragged_cap) CU(cudaStreamCreateWithFlags(&g_ragged_cap, cudaStreamNonBlocking), "stream");
  for (int64_t i = 0; i < count; ++i) plans[i]->R->set_stream((void *)g_ragged_cap);
  const long long l0 = g_launches;
  CU(cudaStreamBeginCapture(g_ragged_cap, cudaStreamCaptureModeThreadLocal), "cudaStreamBeginCapture");
  ctx->state.branches = true;
  fst_status st = run_ragged(plans, y, out, count, dtype, ctx->state);
  ctx->state.branches = false;
  if (st != FST_OK) plans[0]->R->branch_join();   // no branch may be left in the capture
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamEndCapture(g_ragged_cap, &g);
  for (int64_t i = 0; i < count; ++i) plans[i]->R->set_stream(stream);
  ctx->nodes = g_launches - l0;
  g_launches = l0;
  if (st != FST_OK) {
    if (g) cudaGraphDestroy(g);
    return st;
  }
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
  e = cudaGraphInstantiate(&ctx->exec, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
  ctx->gens.resize(count);
  for (int64_t i = 0; i < count; ++i) ctx->gens[i] = plans[i]->ws_gen;
  CU(cudaGraphLaunch(ctx->exec, us), "cudaGraphLaunch");
  g_launches += ctx->nodes;
  return FST_OK;
}

namespace fst {
// A plan about to be destroyed: every recorded ragged batch that uses it points at its
// device data and is dropped (after its launches finish), with its descriptor arrays.
void forget_ragged(fst_plan_t p) {
  std::lock_guard<std::recursive_mutex> lk(g_ragged_mu);
  for (size_t i = 0; i < g_ragged.size();) {
    RaggedCtx *c = g_ragged[i];
    if (std::find(c->plans.begin(), c->plans.end(), p) != c->plans.end()) {
      free_ctx(c);
      g_ragged.erase(g_ragged.begin() + i);
    } else {
      ++i;
    }
  }
}
}  // namespace fst

extern "C" fst_status fst_ragged_tuning(const fst_plan_t *plans, const void *const *y, void *const *out,
                                        int64_t count, int dtype, int64_t *pairs, double *ms) {
  if (count <= 0 || !plans || !y || !out || !pairs) return fail(FST_EINVAL, "bad arguments");
  std::lock_guard<std::recursive_mutex> lk(g_ragged_mu);
  std::vector<const void *> sig;
  sig.reserve(3 * count + 1);
  sig.push_back((const void *)(intptr_t)dtype);
  for (int64_t i = 0; i < count; ++i) {
    sig.push_back(plans[i]);
    sig.push_back(y[i]);
    sig.push_back(out[i]);
  }
  for (RaggedCtx *c : g_ragged)
    if (c->sig == sig) {
      for (int lg = 0; lg < 32; ++lg) {
        pairs[lg] = lg < (int)c->state.chunk.size() ? c->state.chunk[lg] : 0;
        if (ms) ms[lg] = lg < (int)c->state.tune_ms.size() ? c->state.tune_ms[lg] : 0.0;
      }
      return FST_OK;
    }
  return fail(FST_EINVAL, "no ragged call with this signature has run");
}

extern "C" fst_status fst_test_alloc_fail(int after, int allocations) {
  if (after < 0 || allocations < 0) return fail(FST_EINVAL, "bad allocation count");
  fst::g_alloc_after.store(after);
  fst::g_alloc_fail.store(allocations);
  return FST_OK;
}

extern "C" fst_status fst_test_tc_stall(int launches, double limit_s) {
  if (launches < 0 || !(limit_s > 0.0) || limit_s > 2.0) return fail(FST_EINVAL, "bad stall request");
  fst::g_tc_stall_limit_ns = (unsigned long long)(limit_s * 1e9);
  fst::g_tc_stall.store(launches);
  return FST_OK;
}
