// Radial kinetic kernels for any line length N = N1 N2 (N1 even), FP32 and FP64: the DST-II
// kinetic of the sine DVR through a length-N complex FFT carrying two real lines (as in
// mw3_kinetic.cu and mw3_wdft.cuh), in two register levels.
//
// With n = N2 n1 + n2 and k = k1 + N1 k2, on z[n][p] = line 2p + i line 2p+1 (p: the pairs of the
// tile, next to each other in shared memory):
//   A  per (p, n2): N1-point DFT over n1, twiddle w_N^(n2 k1), in place (n1 -> k1);
//   B  per (p, rows k1 and N1 - k1): N2-point DFTs over n2, the spectral scale
//      W_k = sigma_k Z_k + f_k Z_(N-k), whose partner N - k sits in the other row of the same
//      thread (rows 0 and N1/2 pair with themselves and go to one thread), inverse DFTs over k2,
//      conjugate twiddle, in place;
//   C  per (p, n2): inverse N1-point DFT over k1.
// In pass B (and in every pass of the column kernel) a warp's lanes are 32 (long FP64 lines:
// 16) pairs of one or two values of k1: shared accesses are conflict-free, twiddles and scale factors
// warp-wide broadcasts, and all lanes work whatever N1 and N2 are. A tile has 2^lg pairs, fewer
// than the most where the grid would leave SMs idle.
//
// What bounds it: FP32 issue and shared memory. Against the half-warp form (one line pair per 16
// lanes, 128/192/256 only) a value takes three shared-memory round trips instead of four and a
// half, no lane idles where N1 < 16, and the column kernel reads and writes global memory
// straight from passes A and C, without a staged tile. FP64 is bound by the FP64 pipe (2 FMA per
// clock and SM): the two radix levels take about 27 FP64 operations per value against 38 of the
// lane-distributed form.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>

#include "mw3_internal.h"
#include "mw3_wdft.cuh"

namespace mw3 {
namespace {

template <typename T>
struct Vec2;
template <>
struct Vec2<float> {
  using type = float2;
};
template <>
struct Vec2<double> {
  using type = double2;
};

// line pairs per tile: z of 32 pairs of the longest FP64 lines does not fit in shared memory
template <typename T, int N>
constexpr int kPairs = sizeof(T) == 4 || N <= 256 ? 32 : 16;
constexpr int kPThreads = 256;

// Tables in shared memory: w_N^(n2 k1) at [k1][n2], f_k and sigma_k (see wscale in
// mw3_kinetic_w.cu).
template <typename T, int N>
struct PTables {
  cpx<T> tw[N];
  cpx<T> fk[N];
  T sig[N];
};

template <typename T, int N, int N2>
__device__ __forceinline__ void p_load_tables(PTables<T, N>& tb, const cpx<T>* __restrict__ twg,
                                              const cpx<T>* __restrict__ phg, const T* __restrict__ lamg) {
  for (int k = threadIdx.x; k < N; k += kPThreads) {
    const T lr = lamg[N - k], li = lamg[k];
    const cpx<T> e1 = phg[k];
    const cpx<T> e2 = {e1.x * e1.x - e1.y * e1.y, -(T)2 * e1.x * e1.y};
    const T dl = (T)0.5 * (lr - li);
    tb.tw[k] = twg[(k / N2) * (k % N2)];
    tb.sig[k] = (T)0.5 * (lr + li);
    tb.fk[k] = {dl * e2.x, dl * e2.y};
  }
}

template <typename T, int N1, int N2>
__device__ __forceinline__ void fwd_n1(cpx<T>* v, int n2, const cpx<T>* tw) {
  dftR<T, N1>(v, (T)-1);
#pragma unroll
  for (int k1 = 1; k1 < N1; ++k1) v[k1] = cm(v[k1], tw[k1 * N2 + n2]);
}

// a <- sigma_k a + f_k b and b <- sigma_(N-k) b + f_(N-k) a (k != N - k)
template <typename T, int N>
__device__ __forceinline__ void scale2(cpx<T>& a, cpx<T>& b, int k, const PTables<T, N>& tb) {
  const int kp = N - k;
  const cpx<T> fa = cm(tb.fk[k], b), fb = cm(tb.fk[kp], a);
  const T sa = tb.sig[k], sb = tb.sig[kp];
  a = {fma(sa, a.x, fa.x), fma(sa, a.y, fa.y)};
  b = {fma(sb, b.x, fb.x), fma(sb, b.y, fb.y)};
}
template <typename T, int N>
__device__ __forceinline__ void scale1(cpx<T>& a, int k, const PTables<T, N>& tb) {   // k = 0 or N / 2
  const cpx<T> fa = cm(tb.fk[k], a);
  a = {fma(tb.sig[k], a.x, fa.x), fma(tb.sig[k], a.y, fa.y)};
}

// Pass B of every (pair, row pair) item; z[n][p] with row pitch PP.
template <typename T, int N1, int N2, int PP>
__device__ __forceinline__ void pass_b(cpx<T>* z, const PTables<T, N1 * N2>& tb, int lg) {
  constexpr int N = N1 * N2;
#pragma unroll 1
  for (int e = threadIdx.x; e < (N1 / 2) << lg; e += kPThreads) {
    const int p = e & ((1 << lg) - 1), h = e >> lg;
    const int ka = h, kb = h ? N1 - h : N1 / 2;
    cpx<T>* za = z + (long)(N2 * ka) * PP + p;
    cpx<T>* zb = z + (long)(N2 * kb) * PP + p;
    cpx<T> u[N2], w[N2];
#pragma unroll
    for (int i = 0; i < N2; ++i) {
      u[i] = za[i * PP];
      w[i] = zb[i * PP];
    }
    dftR<T, N2>(u, (T)-1);
    dftR<T, N2>(w, (T)-1);
    if (h) {
#pragma unroll
      for (int i = 0; i < N2; ++i) scale2<T, N>(u[i], w[N2 - 1 - i], ka + N1 * i, tb);
    } else {
      scale1<T, N>(u[0], 0, tb);
#pragma unroll
      for (int i = 1; i < (N2 + 1) / 2; ++i) scale2<T, N>(u[i], u[N2 - i], N1 * i, tb);
      if (N2 % 2 == 0) scale1<T, N>(u[N2 / 2], N / 2, tb);
#pragma unroll
      for (int i = 0; i < N2 / 2; ++i) scale2<T, N>(w[i], w[N2 - 1 - i], N1 / 2 + N1 * i, tb);
      if (N2 % 2) scale1<T, N>(w[N2 / 2], N / 2, tb);
    }
    dftR<T, N2>(u, (T)1);
    dftR<T, N2>(w, (T)1);
#pragma unroll
    for (int i = 1; i < N2; ++i) {
      u[i] = cmc(u[i], tb.tw[ka * N2 + i]);
      w[i] = cmc(w[i], tb.tw[kb * N2 + i]);
    }
#pragma unroll
    for (int i = 0; i < N2; ++i) {
      za[i * PP] = u[i];
      zb[i * PP] = w[i];
    }
  }
}

// The row kernel takes both residues per thread where 2 N1 complex values fit in registers.
template <typename T, int N1>
constexpr bool kBoth = sizeof(T) == 4 && N1 <= 18;
// complex values held by a thread
template <typename T, int N1, int N2>
constexpr int kRegs = std::max(2 * N2, kBoth<T, N1> ? 2 * N1 : N1 + 6);
template <typename T, int N1, int N2>
constexpr int kMinCtas = sizeof(T) == 4 ? (kRegs<T, N1, N2> <= 20 ? 3 : (kRegs<T, N1, N2> <= 36 ? 2 : 1))
                                        : (kRegs<T, N1, N2> <= 20 ? 2 : 1);

// Row pitch of z in the row kernel, where pass A and C lanes run over n2: neighbouring n2 are four
// banks apart.
template <typename T, int N>
constexpr int kRowPitch = kPairs<T, N> + 2;

template <typename T, int N1, int N2>
constexpr size_t rows_smem() {
  return sizeof(PTables<T, N1 * N2>) + sizeof(cpx<T>) * (size_t)(N1 * N2) * kRowPitch<T, N1 * N2> + 64 * 4;
}

// R direction: tiles of 2^lg line pairs (2^(lg + 1) consecutive rows), persistent over the tiles.
// Neighbouring elements (2n, 2n + 1) of a row are the values n and N - 1 - n (with a minus sign)
// of the packed sequence, i.e. residues n2 and N2 - 1 - n2: a thread takes both residues, so that
// every access is a pair of elements and a warp's lanes (n2, then p) cover whole sectors. For
// long N1 the two residues would not fit in registers: one each, element by element.
template <typename T, int N1, int N2>
__global__ void __launch_bounds__(kPThreads, (kMinCtas<T, N1, N2>)) k_rows_p(
    const T* __restrict__ q, T* __restrict__ t, long nrows, const cpx<T>* __restrict__ twg,
    const cpx<T>* __restrict__ phg, const T* __restrict__ lamg, const DevBlock* __restrict__ blocks,
    int ng, int nr, int lg) {
  constexpr int N = N1 * N2, PP = kRowPitch<T, N1 * N2>, H1 = N1 / 2;
  constexpr bool BOTH = kBoth<T, N1>;
  constexpr int NI = BOTH ? (N2 + 1) / 2 : N2;     // items per pair
  using V = typename Vec2<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PTables<T, N>& tb = *reinterpret_cast<PTables<T, N>*>(smem_raw);
  cpx<T>* z = reinterpret_cast<cpx<T>*>(smem_raw + sizeof(PTables<T, N>));
  int* live = reinterpret_cast<int*>(z + N * PP);
  p_load_tables<T, N, N2>(tb, twg, phg, lamg);
  const int P = 1 << lg;
  const long ntile = (nrows + 2 * P - 1) / (2 * P);
  for (long tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    const long row0 = tile * 2 * P;
    if (threadIdx.x < P) {   // nr is even: a pair never straddles planes
      const long row = row0 + 2 * threadIdx.x;
      const long plane = row / nr;
      live[threadIdx.x] = row < nrows && (int)(plane % ng) < blocks[plane / ng].nrow;
    }
    __syncthreads();         // also: the previous tile's readers of z are done
#pragma unroll 1
    for (int e = threadIdx.x; e < NI << lg; e += kPThreads) {
      const int p = e / NI, n2 = e - p * NI;
      const T* qa = q + (row0 + 2 * p) * N;
      const T* qb = qa + N;
      const bool on = live[p];
      cpx<T>* s = z + n2 * PP + p;
      if constexpr (BOTH) {
        const int m2 = N2 - 1 - n2;
        cpx<T> u[N1], w[N1];
#pragma unroll
        for (int i = 0; i < H1; ++i) {
          V a{}, b{}, c{}, d{};
          if (on) {
            a = *reinterpret_cast<const V*>(qa + 2 * (N2 * i + n2));
            b = *reinterpret_cast<const V*>(qb + 2 * (N2 * i + n2));
            c = *reinterpret_cast<const V*>(qa + 2 * (N2 * i + m2));
            d = *reinterpret_cast<const V*>(qb + 2 * (N2 * i + m2));
          }
          u[i] = {a.x, b.x};
          w[N1 - 1 - i] = {-a.y, -b.y};
          w[i] = {c.x, d.x};
          u[N1 - 1 - i] = {-c.y, -d.y};
        }
        fwd_n1<T, N1, N2>(u, n2, tb.tw);
#pragma unroll
        for (int i = 0; i < N1; ++i) s[i * N2 * PP] = u[i];
        if (N2 % 2 == 0 || m2 != n2) {
          fwd_n1<T, N1, N2>(w, m2, tb.tw);
          cpx<T>* s2 = z + m2 * PP + p;
#pragma unroll
          for (int i = 0; i < N1; ++i) s2[i * N2 * PP] = w[i];
        }
      } else {
        cpx<T> v[N1];
#pragma unroll
        for (int i = 0; i < N1; ++i) {
          const int m = i < H1 ? 2 * (N2 * i + n2) : 2 * (N - 1 - N2 * i - n2) + 1;
          T a = 0, b = 0;
          if (on) {
            a = __ldg(qa + m);
            b = __ldg(qb + m);
          }
          v[i] = i < H1 ? cpx<T>{a, b} : cpx<T>{-a, -b};
        }
        fwd_n1<T, N1, N2>(v, n2, tb.tw);
#pragma unroll
        for (int i = 0; i < N1; ++i) s[i * N2 * PP] = v[i];
      }
    }
    __syncthreads();
    pass_b<T, N1, N2, PP>(z, tb, lg);
    __syncthreads();
#pragma unroll 1
    for (int e = threadIdx.x; e < NI << lg; e += kPThreads) {
      const int p = e / NI, n2 = e - p * NI;
      if (!live[p]) continue;
      T* ta = t + (row0 + 2 * p) * N;
      T* tc = ta + N;
      const cpx<T>* s = z + n2 * PP + p;
      if constexpr (BOTH) {
        const int m2 = N2 - 1 - n2;
        const cpx<T>* s2 = z + m2 * PP + p;
        cpx<T> u[N1], w[N1];
#pragma unroll
        for (int i = 0; i < N1; ++i) {
          u[i] = s[i * N2 * PP];
          w[i] = s2[i * N2 * PP];
        }
        dftR<T, N1>(u, (T)1);
        dftR<T, N1>(w, (T)1);
#pragma unroll
        for (int i = 0; i < H1; ++i) {
          V o;
          o.x = u[i].x;
          o.y = -w[N1 - 1 - i].x;
          *reinterpret_cast<V*>(ta + 2 * (N2 * i + n2)) = o;
          o.x = u[i].y;
          o.y = -w[N1 - 1 - i].y;
          *reinterpret_cast<V*>(tc + 2 * (N2 * i + n2)) = o;
          if (N2 % 2 == 0 || m2 != n2) {
            o.x = w[i].x;
            o.y = -u[N1 - 1 - i].x;
            *reinterpret_cast<V*>(ta + 2 * (N2 * i + m2)) = o;
            o.x = w[i].y;
            o.y = -u[N1 - 1 - i].y;
            *reinterpret_cast<V*>(tc + 2 * (N2 * i + m2)) = o;
          }
        }
      } else {
        cpx<T> v[N1];
#pragma unroll
        for (int i = 0; i < N1; ++i) v[i] = s[i * N2 * PP];
        dftR<T, N1>(v, (T)1);
#pragma unroll
        for (int i = 0; i < N1; ++i) {
          const int m = i < H1 ? 2 * (N2 * i + n2) : 2 * (N - 1 - N2 * i - n2) + 1;
          ta[m] = i < H1 ? v[i].x : -v[i].x;
          tc[m] = i < H1 ? v[i].y : -v[i].y;
        }
      }
    }
    __syncthreads();         // live and z are rewritten by the next tile
  }
}

template <typename T, int N1, int N2>
constexpr size_t cols_smem() {
  return sizeof(PTables<T, N1 * N2>) + sizeof(cpx<T>) * (size_t)(N1 * N2) * kPairs<T, N1 * N2> +
         sizeof(T) * (size_t)N2 * kPairs<T, N1 * N2> * 4;
}

// r direction: one CTA = one (block, i) plane and the column pairs [c0, c0 + 2 P). Passes A and C
// read and update global memory directly (a warp's lanes are neighbouring pairs); the flux cut
// sums each thread's N1 rows in order, then the N2 partial sums in order.
template <typename T, int N1, int N2>
__global__ void __launch_bounds__(kPThreads, (kMinCtas<T, N1, N2>)) k_cols_p(
    const T* __restrict__ q, T* __restrict__ t, int NR, const cpx<T>* __restrict__ twg,
    const cpx<T>* __restrict__ phg, const T* __restrict__ lamg, int ng,
    const T* __restrict__ wpsi, const T* __restrict__ wdpsi, T* __restrict__ cut,
    const DevBlock* __restrict__ blocks, const int* __restrict__ ncut_J, int m_inf,
    T* __restrict__ qcol, int lg) {
  constexpr int N = N1 * N2, P = kPairs<T, N>;
  using V = typename Vec2<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PTables<T, N>& tb = *reinterpret_cast<PTables<T, N>*>(smem_raw);
  cpx<T>* z = reinterpret_cast<cpx<T>*>(smem_raw + sizeof(PTables<T, N>));
  T* part = reinterpret_cast<T*>(z + N * P);   // [N2][P][4]: psi and dpsi of both columns
  const long plane = blockIdx.y;
  const int b = (int)(plane / ng);
  const int n = (int)(plane - (long)b * ng);
  const DevBlock B = blocks[b];
  if (n >= B.nrow) return;
  p_load_tables<T, N, N2>(tb, twg, phg, lamg);
  const int c0 = blockIdx.x << (lg + 1), pmask = (1 << lg) - 1;
  const T* qp = q + plane * (long)N * NR + c0;
  T* tp = t + plane * (long)N * NR + c0;
  __syncthreads();
#pragma unroll 1
  for (int e = threadIdx.x; e < N2 << lg; e += kPThreads) {
    const int p = e & pmask, n2 = e >> lg;
    const bool in = c0 + 2 * p < NR;   // NR is even
    cpx<T> v[N1];
    // element n = N2 i + n2 is row 2 n (i < N1 / 2) or, with a minus sign, 2 (N - 1 - n) + 1
#pragma unroll
    for (int i = 0; i < N1; ++i) {
      const int kr = i < N1 / 2 ? 2 * (N2 * i + n2) : 2 * (N - 1 - N2 * i - n2) + 1;
      V x{};
      if (in) x = *reinterpret_cast<const V*>(qp + (long)kr * NR + 2 * p);
      v[i] = {x.x, x.y};
    }
    if (cut != nullptr) {
      T s0 = 0, s1 = 0, d0 = 0, d1 = 0;
#pragma unroll
      for (int i = 0; i < N1; ++i) {
        const int kr = i < N1 / 2 ? 2 * (N2 * i + n2) : 2 * (N - 1 - N2 * i - n2) + 1;
        const T wp = __ldg(wpsi + kr), wd = __ldg(wdpsi + kr);
        s0 = fma(wp, v[i].x, s0);
        s1 = fma(wp, v[i].y, s1);
        d0 = fma(wd, v[i].x, d0);
        d1 = fma(wd, v[i].y, d1);
      }
      T* o = part + (n2 * P + p) * 4;
      o[0] = s0;
      o[1] = d0;
      o[2] = s1;
      o[3] = d1;
    }
    if (qcol != nullptr && m_inf >= c0 && (m_inf - c0) >> 1 == p) {
#pragma unroll
      for (int i = 0; i < N1; ++i) {
        const int kr = i < N1 / 2 ? 2 * (N2 * i + n2) : 2 * (N - 1 - N2 * i - n2) + 1;
        qcol[plane * N + kr] = (m_inf & 1) ? v[i].y : v[i].x;
      }
    }
#pragma unroll
    for (int i = N1 / 2; i < N1; ++i) v[i] = {-v[i].x, -v[i].y};
    fwd_n1<T, N1, N2>(v, n2, tb.tw);
    cpx<T>* s = z + n2 * P + p;
#pragma unroll
    for (int i = 0; i < N1; ++i) s[i * N2 * P] = v[i];
  }
  __syncthreads();
  if (cut != nullptr) {
    const long ncut = ncut_J[B.iJ];
    for (int o = threadIdx.x; o < 4 << lg; o += kPThreads) {
      const int p = o >> 2, m = c0 + 2 * p + ((o >> 1) & 1);
      if (m >= NR) continue;
      T s = 0;
#pragma unroll
      for (int n2 = 0; n2 < N2; ++n2) s += part[(n2 * P + p) * 4 + (o & 3)];
      cut[B.cutcol + (long)(o & 1) * ncut + (long)n * NR + m] = s;
    }
  }
  pass_b<T, N1, N2, P>(z, tb, lg);
  __syncthreads();
#pragma unroll 1
  for (int e = threadIdx.x; e < N2 << lg; e += kPThreads) {
    const int p = e & pmask, n2 = e >> lg;
    const bool in = c0 + 2 * p < NR;
    cpx<T>* s = z + n2 * P + p;
    cpx<T> v[N1];
#pragma unroll
    for (int i = 0; i < N1; ++i) v[i] = s[i * N2 * P];
    dftR<T, N1>(v, (T)1);
    if (!in) continue;
    constexpr int G = N1 <= 10 ? N1 : (N1 % 8 == 0 ? 8 : (N1 % 10 == 0 ? 10 : (N1 % 6 == 0 ? 6 : N1)));
#pragma unroll
    for (int g = 0; g < N1; g += G) {   // G updates in flight
      V o[G];
#pragma unroll
      for (int i = g; i < g + G; ++i) {
        const int kr = i < N1 / 2 ? 2 * (N2 * i + n2) : 2 * (N - 1 - N2 * i - n2) + 1;
        o[i - g] = *reinterpret_cast<const V*>(tp + (long)kr * NR + 2 * p);
      }
#pragma unroll
      for (int i = g; i < g + G; ++i) {
        const int kr = i < N1 / 2 ? 2 * (N2 * i + n2) : 2 * (N - 1 - N2 * i - n2) + 1;
        o[i - g].x += i < N1 / 2 ? v[i].x : -v[i].x;
        o[i - g].y += i < N1 / 2 ? v[i].y : -v[i].y;
        *reinterpret_cast<V*>(tp + (long)kr * NR + 2 * p) = o[i - g];
      }
    }
  }
}

// log2 of the pairs per tile: the most, halved (down to 4) while fewer tiles than SMs result.
inline int tile_lg(int most, long pairs_per_line, long lines) {
  const int nsm = sm_count();
  int lg = most == 32 ? 5 : 4;
  while (lg > 2 && ((pairs_per_line + (1 << lg) - 1) >> lg) * lines < nsm) --lg;
  return lg;
}

template <typename T, int N1, int N2>
cudaError_t rows_p(const T* q, T* t, long nrows, const void* tw, const void* ph, const T* lam,
                   const DevBlock* blocks, int ng, int nr, cudaStream_t st) {
  constexpr size_t sm = rows_smem<T, N1, N2>();
  static_assert(sm <= 227 * 1024, "shared memory of the row kernel");
  static OncePerDevice attr;
  static IntPerDevice per;
  const cudaError_t e = allow_smem(attr, k_rows_p<T, N1, N2>, sm);
  if (e != cudaSuccess) return e;
  const int grid_max = sm_count() * per.get(current_device(), [&] {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_rows_p<T, N1, N2>, kPThreads, sm);
    return std::max(n, 1);
  });
  const int lg = tile_lg(kPairs<T, N1 * N2>, nrows / 2, 1);
  const long ntile = ((nrows + 1) / 2 + (1 << lg) - 1) >> lg;
  k_rows_p<T, N1, N2><<<(unsigned)std::min<long>(ntile, grid_max), kPThreads, sm, st>>>(
      q, t, nrows, static_cast<const cpx<T>*>(tw), static_cast<const cpx<T>*>(ph), lam, blocks, ng, nr, lg);
  return cudaGetLastError();
}

template <typename T, int N1, int N2>
cudaError_t cols_p(const T* q, T* t, long nplanes, int NR, const void* tw, const void* ph,
                   const T* lam, int ng, const T* wpsi, const T* wdpsi, T* cut,
                   const DevBlock* blocks, const int* ncut_J, int m_inf, T* qcol, cudaStream_t st) {
  constexpr size_t sm = cols_smem<T, N1, N2>();
  static_assert(sm <= 227 * 1024, "shared memory of the column kernel");
  static OncePerDevice attr;
  const cudaError_t e = allow_smem(attr, k_cols_p<T, N1, N2>, sm);
  if (e != cudaSuccess) return e;
  const int lg = tile_lg(kPairs<T, N1 * N2>, NR / 2, nplanes);
  dim3 grid((unsigned)((NR / 2 + (1 << lg) - 1) >> lg), (unsigned)nplanes);
  k_cols_p<T, N1, N2><<<grid, kPThreads, sm, st>>>(q, t, NR, static_cast<const cpx<T>*>(tw),
                                                   static_cast<const cpx<T>*>(ph), lam, ng, wpsi,
                                                   wdpsi, cut, blocks, ncut_J, m_inf, qcol, lg);
  return cudaGetLastError();
}

}  // namespace

// Line lengths with a two-level form and their factors (N1, N2): every even 2^a 3^b 5^c from 24 to
// 512. N2 = 16 for 128, 192 and 256, where the fused radial kernel (mw3_radial.cu) runs the same
// transform on half-warps, bit for bit; elsewhere the two levels are about even and no thread
// holds more than 27 pairs. Three parts, one per translation unit (compile time).
#define MW3_PSIZES_A(X) \
  X(6, 4) X(6, 5) X(8, 4) X(6, 6) X(8, 5) X(8, 6) X(10, 5) X(6, 9) X(10, 6) X(8, 8) X(12, 6) X(10, 8) \
  X(10, 9) X(12, 8) X(10, 10) X(12, 9) X(12, 10) X(8, 16)
#define MW3_PSIZES_B(X) \
  X(16, 9) X(10, 15) X(16, 10) X(18, 9) X(18, 10) X(12, 16) X(20, 10) X(24, 9) X(16, 15) X(10, 25) \
  X(16, 16) X(18, 15) X(18, 16)
#define MW3_PSIZES_C(X) \
  X(20, 15) X(20, 16) X(18, 18) X(24, 15) X(24, 16) X(20, 20) X(24, 18) X(30, 15) X(32, 15) X(18, 27) \
  X(20, 25) X(32, 16)

// The dispatch of one part and one precision; false where the length is not in the part.
#define MW3_PDEFINE(NAME, T, SIZES)                                                                   \
  bool NAME##_rows(int N, const T* q, T* t, long nrows, const void* tw, const void* ph, const T* lam, \
                   const DevBlock* blocks, int ng, int nr, cudaStream_t st, cudaError_t* err) {       \
    switch (N) { SIZES(MW3_PROW) default: return false; }                                             \
  }                                                                                                   \
  bool NAME##_cols(int N, const T* q, T* t, long nplanes, int NR, const void* tw, const void* ph,     \
                   const T* lam, int ng, const T* wpsi, const T* wdpsi, T* cut,                       \
                   const DevBlock* blocks, const int* ncut_J, int m_inf, T* qcol, cudaStream_t st,    \
                   cudaError_t* err) {                                                                \
    switch (N) { SIZES(MW3_PCOL) default: return false; }                                             \
  }
#define MW3_PROW(n1, n2)                                                                          \
  case n1 * n2:                                                                                   \
    *err = rows_p<MW3_PT, n1, n2>(q, t, nrows, tw, ph, lam, blocks, ng, nr, st);                  \
    return true;
#define MW3_PCOL(n1, n2)                                                                          \
  case n1 * n2:                                                                                   \
    *err = cols_p<MW3_PT, n1, n2>(q, t, nplanes, NR, tw, ph, lam, ng, wpsi, wdpsi, cut, blocks,   \
                                  ncut_J, m_inf, qcol, st);                                       \
    return true;

}  // namespace mw3
