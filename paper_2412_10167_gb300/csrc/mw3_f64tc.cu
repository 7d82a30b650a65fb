// FP64 angular step on the tensor cores: the gamma transforms, the potential, the FBR and
// Coriolis terms, the damped Chebyshev recursion and the norm partials of the FP64 form
// (Section 2.1 items 3-5, Section 2.2, Eq. wvp-k) in one launch.
//
// What bounds it. FP64 arithmetic runs at 1/64 of FP32 on this part (2 FMA per clock and SM),
// so the two n_gamma x n_gamma products of a step cost 2 n_gamma FP64 FMAs per grid value on
// the CUDA cores. Here they are exact integer products on tcgen05 instead (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication", 2012):
//   * a column of the operand becomes fixed point relative to its largest element,
//     X = round(|x| 2^(54 - e)), |x| < 2^e, and X seven balanced base-256 digits
//     d_s in [-128, 127] (54 bits: an element of the column's own binade is exact), each held
//     as FP16 in tensor memory; the matrix rows likewise, once, at set-up;
//   * level l collects the digit products with i + j = l, l = 0..7. Every partial sum is an
//     integer below 7 K 2^14 < 2^23.5 for K <= 96, so the FP32 accumulator holds it exactly. The
//     levels left out are below 2^-59 of (column maximum) x (row maximum) per term: at most 2^-53
//     for K = 96 terms, about 2^-59 for digits of either sign. (Without level 7 the
//     products left out add up to several 2^-53, ten times the error of an FP64 sum.)
//   * the eight level sums are combined in 64-bit integers and rounded to FP64 once.
// The error is that of the 54-bit operands: 2^-54 of the column's (row's) largest element, so that an
// element 2^-k of it keeps 54 - k bits. An FP64 sum over the column has the same bound, its rounding
// errors being those of the largest terms, and the measured errors agree; a column is scaled by
// itself, so that nothing is lost between columns or blocks. FP64 units do 2 operations per
// output instead of n_gamma / 2 (after the parity split) or n_gamma.
//
// Parity split of the Gauss-Legendre rule as in the mixed form: T^Omega[i][n'] =
// (-1)^i T^Omega[i][n] for mirrored nodes n, n', so each transform is an even and an odd half
// of K = ceil(n_gamma / 2). For odd n_gamma the middle node is its own mirror image: it enters
// the even sum once and the odd functions vanish there.
//
// One CTA works on one tile of 128 tensor-memory lanes: 128 (r, R) columns of one state, or 64
// columns of both diabatic states (lanes 0-63 and 64-127), through four products in turn:
//   0: E = even coefficients -> nodes,  1: O = odd coefficients -> nodes, u = E +- O,
//   2: w_even from y(n) + y(n'),        3: w_odd from y(n) - y(n'),  y = V u,
// and the epilogue of 2 and 3 finishes the coefficient rows. Digit matrices stream through two
// shared-memory buffers (they are read from L2 once per tile). Accumulators take 8 NC
// tensor-memory columns beside the 7 K / 2 of the operand digits, which sets the output chunk
// NC for each K (the last chunk of K = 48 is narrower).
//
// Measured (GB300, ms per step): 256 x 192 x 96, J = 10 (11 blocks): 23.1 for the two FP64 GEMMs
// and 0.16 for the norms -> 2.78; 64 x 48 x 24, J = 0: 0.116 -> 0.038. Relative error of 256
// iterations against FP64 matrix products: 4.0e-13 for both forms.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "mw3_internal.h"
#include "mw3_tcgen.cuh"

namespace mw3 {
namespace {

constexpr int kThreads = 512;
constexpr int kSlices = kF64Slices;
constexpr int kLevels = kSlices + 1;

template <int KH>
constexpr bool kNodesInSmem = KH <= 80;

template <int KH>
constexpr size_t bbuf_bytes() {
  return (size_t)kSlices * f64tc_chunk(KH) * KH * 2;
}
template <int KH>
constexpr size_t f64tc_smem() {
  return 2 * bbuf_bytes<KH>() + (kNodesInSmem<KH> ? 2 * (size_t)KH * TC_M * 8 : 0) + 4 * TC_M * 4 +
         16 * sizeof(double) + 32;
}

// D (+)= A B, FP16 operands, FP32 accumulators; A (M x K) in tensor memory, two FP16 per column
__device__ __forceinline__ void mma_f16_ta(uint32_t dtmem, uint32_t atmem, uint64_t bd,
                                           uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(dtmem),
      "r"(atmem), "l"(bd), "r"(idesc), "r"(accum));
}

__device__ __forceinline__ void tmem_st2(uint32_t taddr, uint32_t v0, uint32_t v1) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(taddr), "r"(v0),
               "r"(v1)
               : "memory");
}

// Fixed-point digits of x (ex: biased exponent of the column's largest element, >= x's own):
// the seven low bytes of the result hold digit + 128, byte 6 the leading one.
__device__ __forceinline__ uint64_t digits_of(double x, int ex) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int xi = (int)((hi >> 20) & 0x7ffu);
  const uint64_t m = xi ? (((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << 2 : 0ull;
  const int d = min(ex - xi, 63);
  const long long X = (long long)(((m >> d) + 1) >> 1);
  return (uint64_t)(((int)hi < 0 ? -X : X) + 0x0080808080808080ll);
}

// FP16 pair (digit of a, digit of b) from byte `sel` of their low or high words: the byte under
// the bits of 1024 reads as 1024 + byte, minus 1152.
__device__ __forceinline__ uint32_t digit_pair(uint32_t a, uint32_t b, int byte) {
  const uint32_t w = __byte_perm(a, b, (uint32_t)(byte | ((4 + byte) << 8)));
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"((w & 0x00ff00ffu) | 0x64006400u), "r"(0x64806480u));
  return r;
}

// Integer value of a level sum: |acc| < 2^22 through the FP32 rounding constant, larger ones
// by conversion.
template <bool SMALL>
__device__ __forceinline__ int level_int(uint32_t bits) {
  if constexpr (SMALL) {
    return __float_as_int(__uint_as_float(bits) + 12582912.0f) - 0x4B400000;
  } else {
    return __float2int_rn(__uint_as_float(bits));
  }
}

// sum_l acc_l 2^(-8 l) scaled by 2^(sc + 44), rounded once. |sum| < 2^18.7.
template <int KH>
__device__ __forceinline__ double combine(const uint32_t* l, int stride, int sc) {
  auto lv = [&](auto tag) {
    constexpr int i = decltype(tag)::value;
    constexpr long pairs = i < kSlices ? i + 1 : 2 * kSlices - 1 - i;
    return level_int<(pairs * KH * 16384 < (1L << 22))>(l[i * stride]);
  };
  const int a0 = lv(std::integral_constant<int, 0>{}), a1 = lv(std::integral_constant<int, 1>{}),
            a2 = lv(std::integral_constant<int, 2>{}), a3 = lv(std::integral_constant<int, 3>{}),
            a4 = lv(std::integral_constant<int, 4>{}), a5 = lv(std::integral_constant<int, 5>{}),
            a6 = lv(std::integral_constant<int, 6>{}), a7 = lv(std::integral_constant<int, 7>{});
  long long V = (long long)a2 * (1 << 28) + (long long)a3 * (1 << 20) + (long long)a4 * (1 << 12) +
                (long long)a5 * 16 + ((a6 + (a7 >> 8) + 8) >> 4);
  V += (long long)((uint64_t)(uint32_t)((a0 << 12) + (a1 << 4)) << 32);
  // 64-bit integer to FP64: the high word at 2^32, offset by 2^84 + 2^63, then the low word
  const double hi = __hiloint2double(0x45300000, (int)((uint32_t)((uint64_t)V >> 32) ^ 0x80000000u)) -
                    (0x1p84 + 0x1p63 + 0x1p52);
  const double v = hi + __hiloint2double(0x43300000, (int)(uint32_t)(uint64_t)V);
  const int e = ((__double2hiint(v) >> 20) & 0x7ff) + sc;
  return (V == 0 || e <= 0) ? 0.0 : __hiloint2double(__double2hiint(v) + (sc << 20), __double2loint(v));
}

template <int KH, int NE>
__global__ void __launch_bounds__(kThreads, 1) k_angular_f64(const __grid_constant__ F64Args a) {
  extern __shared__ __align__(1024) unsigned char sm[];
  constexpr int S = kSlices;
  constexpr int NC = f64tc_chunk(KH), NCH = (KH + NC - 1) / NC;
  constexpr int kq = KH / 4;                 // operand elements per thread
  constexpr bool SMEM = kNodesInSmem<KH>;
  constexpr int CT = TC_M / NE;
  unsigned char* bbuf = sm;
  double* U1 = reinterpret_cast<double*>(sm + 2 * bbuf_bytes<KH>());
  double* U2 = U1 + (SMEM ? KH * TC_M : 0);
  uint32_t* mx = reinterpret_cast<uint32_t*>(U2 + (SMEM ? KH * TC_M : 0));
  double* red = reinterpret_cast<double*>(mx + 4 * TC_M);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(red + 16);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q = warp & 3, part = warp >> 2;
  const int m = q * 32 + lane;
  const int L = NE == 2 ? m >> 6 : 0, cl = NE == 2 ? (m & 63) : m;
  const uint32_t mb = smem_u32(mbar);
  const uint32_t lane_base = (uint32_t)(q * 32) << 16;
  const int ng = a.ng, hh = (ng + 1) / 2;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
        smem_u32(tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mb), "r"(kLevels));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;
  const uint32_t tA = tmem, tD = tmem + S * (KH / 2);

  const long total = (long)a.ngroups * a.ntiles;
  const long f0 = (long)blockIdx.x * total / gridDim.x;
  const long f1 = (long)(blockIdx.x + 1) * total / gridDim.x;
  const long nb = (f1 - f0) * 4 * NCH;         // digit-matrix chunks this CTA consumes
  auto issue_b = [&](long k) {                 // chunk k of the CTA's sequence -> buffer k & 1
    if (k < nb) {
      const long f = f0 + k / (4 * NCH);
      const int r = (int)(k % (4 * NCH));
      const int om = a.blocks[(f / a.ntiles) * NE].omega;
      const int ch = r % NCH;
      const int bytes = S * min(NC, KH - ch * NC) * KH * 2;
      const unsigned char* src = a.Td + ((long)om * 4 + r / NCH) * (S * KH * KH * 2) +
                                 (long)ch * bbuf_bytes<KH>();
      unsigned char* dst = bbuf + (k & 1) * bbuf_bytes<KH>();
      for (int e = tid; e < bytes / 16; e += kThreads)
        cp_async16(dst + 16 * e, src + 16 * e);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  uint32_t phase = 0;
  bool ok = true;
  long kb = 0;
  issue_b(0);
  issue_b(1);

  for (long f = f0; f < f1 && ok; ++f) {
    const int g = (int)(f / a.ntiles);
    const int tile = (int)(f - (long)g * a.ntiles);
    const int b = g * NE + L;
    const DevBlock B = a.blocks[b];
    const int nrow = B.nrow;
    const long col = (long)tile * CT + cl;
    const bool live = col < a.ncol;
    const int kr = live ? (int)(col / a.NR) : 0;
    const int mR = live ? (int)(col - (long)kr * a.NR) : 0;
    const double* c = a.ck + (long)b * a.npts + col;
    const double invdE = a.dj[B.iJ].invdE;
    const double D = live ? a.DR[mR] * a.Dr[kr] : 0.0;
    const double s1 = a.mode == 1 ? invdE : D * a.alpha * invdE, s3 = a.beta * D * D;
    double ss = 0.0;
    // node values: u(n) and u(n') of (lane, n < hh)
    auto u1 = [&](int n, int l) -> double* {
      if constexpr (SMEM) return U1 + n * TC_M + l;
      else return a.u + (long)(g * NE + (NE == 2 ? l >> 6 : 0)) * a.npts + (long)n * a.ncol + col;
    };
    auto u2 = [&](int n, int l) -> double* {
      if constexpr (SMEM) return U2 + n * TC_M + l;
      else return a.u + (long)(g * NE + (NE == 2 ? l >> 6 : 0)) * a.npts + (long)(ng - 1 - n) * a.ncol + col;
    };

#pragma unroll 1
    for (int sg = 0; sg < 4 && ok; ++sg) {
      // ---- operand column: coefficients of one parity, or y(n) +- y(n')
      double x[kq];
      if (sg < 2) {
#pragma unroll
        for (int s = 0; s < kq; ++s) {
          const int i = 2 * (part * kq + s) + sg;
          x[s] = (live && i < nrow) ? __ldg(c + (long)i * a.ncol) : 0.0;
        }
      } else {
        const double* Vl = a.V + (long)(L * NE) * a.npts + col;
#pragma unroll
        for (int s = 0; s < kq; ++s) {
          const int n = part * kq + s;
          x[s] = 0.0;
          if (live && n < hh) {
            const int n2 = ng - 1 - n;
            double ya, yb;
            if constexpr (NE == 1) {
              ya = __ldg(Vl + (long)n * a.ncol) * *u1(n, m);
              yb = 0.0;
              if (n2 != n) {
                const double w = __ldg(Vl + (long)n2 * a.ncol) * *u2(n, m);
                yb = w;
              }
            } else {
              const double* V2 = Vl + a.npts;
              ya = __ldg(Vl + (long)n * a.ncol) * *u1(n, cl) + __ldg(V2 + (long)n * a.ncol) * *u1(n, 64 + cl);
              yb = 0.0;
              if (n2 != n)
                yb = __ldg(Vl + (long)n2 * a.ncol) * *u2(n, cl) + __ldg(V2 + (long)n2 * a.ncol) * *u2(n, 64 + cl);
            }
            x[s] = sg == 2 ? ya + yb : (n2 != n ? ya - yb : 0.0);
          }
        }
      }
      uint32_t top = 0;
#pragma unroll
      for (int s = 0; s < kq; ++s) top = max(top, (uint32_t)__double2hiint(x[s]) & 0x7fffffffu);
      mx[part * TC_M + m] = top;
      __syncthreads();
      top = max(max(mx[m], mx[TC_M + m]), max(mx[2 * TC_M + m], mx[3 * TC_M + m]));
      const int ex = (int)(top >> 20);
      const bool bad = ex == 0x7ff;            // NaN or infinity in the column
#pragma unroll
      for (int s = 0; s < kq; s += 4) {
        uint32_t lo[4], hi[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint64_t y = digits_of(x[s + j], ex);
          lo[j] = (uint32_t)y;
          hi[j] = (uint32_t)(y >> 32);
        }
        const uint32_t cc = tA + lane_base + (uint32_t)((part * kq + s) / 2);
#pragma unroll
        for (int i = 0; i < S; ++i) {          // slice i: byte 6 - i
          const uint32_t p0 = i < 3 ? digit_pair(hi[0], hi[1], 2 - i) : digit_pair(lo[0], lo[1], 6 - i);
          const uint32_t p1 = i < 3 ? digit_pair(hi[2], hi[3], 2 - i) : digit_pair(lo[2], lo[3], 6 - i);
          tmem_st2(cc + (uint32_t)(i * (KH / 2)), p0, p1);
        }
      }
      tmem_st_wait();
      const int sc0 = ex - 1022 - 56;
      const int* eT = a.eT + ((long)B.omega * 4 + sg) * KH;

#pragma unroll 1
      for (int ch = 0; ch < NCH && ok; ++ch) {
        const int nc = min(NC, KH - ch * NC);                  // 16 or 32 output rows
        asm volatile("cp.async.wait_group 1;" ::: "memory");   // this chunk's digits
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        // one issuing thread per level (they write different accumulators): a single thread
        // needs about 130 cycles per product, 13,000 for the 102 of K = 48
        if (warp < kLevels && elect_one()) {
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint64_t bd = smem_desc(smem_u32(bbuf + (kb & 1) * bbuf_bytes<KH>()), 128, KH * 16);
          const uint32_t idesc = (1u << 4) | ((uint32_t)(nc >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
          const uint32_t bslice = (uint32_t)(nc * KH * 2) >> 4;
          const int l = warp, i0 = max(0, l - S + 1), i1 = min(l, S - 1);
          const uint32_t d = tD + (uint32_t)(l * NC);
          uint32_t ta = tA + (uint32_t)(i0 * (KH / 2));
          uint64_t db = bd + (uint64_t)((l - i0) * bslice);
#pragma unroll 1
          for (int i = i0; i <= i1; ++i, ta += KH / 2, db -= bslice) {
#pragma unroll
            for (int ks = 0; ks < KH / 16; ++ks)
              mma_f16_ta(d, ta + (uint32_t)(ks * 8), db + (uint64_t)(ks * 16), idesc, i != i0 || ks != 0);
          }
          mma_commit(mb);
        }
        ok = __syncthreads_and(mbar_wait(mb, phase, a.wait_limit) ? 1 : 0) != 0;
        phase ^= 1;
        asm volatile("tcgen05.fence::after_thread_sync;");
        issue_b(kb + 2);
        ++kb;
        if (!ok) break;
#pragma unroll 1
        for (int s0 = 0; s0 < nc / 4; s0 += 4) {
          const int nloc = part * (nc / 4) + s0;
          const int n0 = ch * NC + nloc;
          uint32_t r[kLevels * 4];
#pragma unroll
          for (int l = 0; l < kLevels; ++l)
            tmem_ld4_issue(tD + lane_base + (uint32_t)(l * NC + nloc), r + 4 * l);
          // the epilogue's rows are read while the levels arrive
          double cv[4], h0[4], pv[4];
          if (sg >= 2) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int i = 2 * (n0 + j) + sg - 2;
              const bool in = live && i < nrow;
              const long off = (long)i * a.ncol;
              cv[j] = in ? __ldg(c + off) : 0.0;
              h0[j] = in ? __ldg(a.t + (long)b * a.npts + col + off) : 0.0;
              pv[j] = (in && a.mode == 0) ? a.ckm1[(long)b * a.npts + col + off] : 0.0;
            }
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;"
                       : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                         "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                         "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]),
                         "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                         "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                         "+r"(r[30]), "+r"(r[31])
                       :
                       : "memory");
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int n = n0 + j;
            double w = combine<KH>(r + j, 4, sc0 + __ldg(eT + n));
            if (bad) w = __hiloint2double(0x7ff80000, 0);
            if (sg < 2) {
              if (live && n < hh) {
                if (sg == 0) {
                  *u1(n, m) = w;                 // E
                } else {
                  const double E = *u1(n, m);
                  *u1(n, m) = E + w;
                  if (2 * n != ng - 1) *u2(n, m) = E - w;
                }
              }
            } else {
              const int i = 2 * n + sg - 2;
              if (!live || i >= ng) continue;
              const long idx = (long)b * a.npts + col + (long)i * a.ncol;
              if (i >= nrow) {                   // beyond the block's angular functions
                if (a.mode == 1) a.out[idx] = 0.0; else a.ckm1[idx] = 0.0;
                continue;
              }
              const double* G = a.gtab + ((long)B.coef * 3 * ng + i) * a.NR + mR;
              const double aa = __ldg(a.rot + ((long)B.coef * ng + i) * a.nr + kr) + __ldg(G);
              double h = fma(aa, cv[j], h0[j] + w);
              if (B.up >= 0 && i >= 1)
                h = fma(__ldg(G + (long)ng * a.NR),
                        __ldg(a.ck + (long)B.up * a.npts + col + (long)(i - 1) * a.ncol), h);
              if (B.dn >= 0)
                h = fma(__ldg(G + 2L * ng * a.NR),
                        __ldg(a.ck + (long)B.dn * a.npts + col + (long)(i + 1) * a.ncol), h);
              if (a.mode == 1) {
                a.out[idx] = s1 * h;
              } else {
                const double nv = fma(s1, h, -s3 * pv[j]);
                a.ckm1[idx] = nv;
                ss = fma(nv, nv, ss);
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
      }
      __syncthreads();                          // node values written; accumulators read
      asm volatile("tcgen05.fence::after_thread_sync;");
    }
    if (a.mode == 0) {
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_down_sync(0xffffffffu, ss, o);
      if (lane == 0) red[warp] = ss;
      __syncthreads();
      if (tid == 0 && a.npart) {
        double s2 = 0;
        for (int w2 = 0; w2 < kThreads / 32; ++w2) s2 += red[w2];
        a.npart[(long)g * a.ntiles + tile] = s2;
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (!ok && tid == 0) atomicExch(a.err, 1);
  drain_expired(ok, mb, phase ^ 1u);   // ok is CTA-uniform; the failed wait toggled phase
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

template <int KH, int NE>
cudaError_t launch_inst(const F64Args& a, cudaStream_t st) {
  constexpr size_t sm = f64tc_smem<KH>();
  static_assert(sm <= 227 * 1024, "shared memory of the FP64 angular step");
  static_assert(kSlices * (KH / 2) + kLevels * f64tc_chunk(KH) <= 512, "tensor memory of the FP64 angular step");
  static_assert((long)kSlices * KH * 16384 < (1L << 24), "level sums exact in FP32");
  static OncePerDevice attr;
  const cudaError_t e = allow_smem(attr, k_angular_f64<KH, NE>, sm);
  if (e != cudaSuccess) return e;
  const long total = (long)a.ngroups * a.ntiles;
  const unsigned grid = (unsigned)std::min<long>(a.nsm, total);
  k_angular_f64<KH, NE><<<grid, kThreads, sm, st>>>(a);
  return cudaGetLastError();
}

template <int NE>
cudaError_t launch_ne(const F64Args& a, cudaStream_t st) {
  switch (a.kh) {
#define CASE(k) case k: return launch_inst<k, NE>(a, st);
    CASE(16) CASE(32) CASE(48) CASE(64) CASE(80) CASE(96)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

int angular_f64_kh(int ng) {
  const int kh = (((ng + 1) / 2 + 15) / 16) * 16;
  return kh <= 96 ? kh : 0;
}

// The form applies to n_gamma <= 192 (K = 96: beyond it the operand digits and eight accumulators
// of 16 columns do not fit in tensor memory); larger ones keep the GEMMs of mw3_gamma.cu. It is
// taken at every smaller size: at n_gamma = 24 and one block, where a launch is 24 tiles on 152
// SMs, it is already 2.6 times faster than the GEMM pair, which pads to 64 x 64 tiles.
cudaError_t launch_angular_f64(const F64Args& a, const int* g_begin, int nJ, double* norm_out,
                               cudaStream_t st) {
  const cudaError_t e = a.nelec == 1 ? launch_ne<1>(a, st) : launch_ne<2>(a, st);
  if (e != cudaSuccess || !norm_out || !a.npart) return e;
  return launch_tc_norm_final(a.npart, g_begin, nJ, a.ntiles, norm_out, st);
}

}  // namespace mw3
