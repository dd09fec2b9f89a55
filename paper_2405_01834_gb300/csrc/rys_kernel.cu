// Rys-quadrature kernel: shellsets of one primitive quartet, one block per shell quartet.
//
// The Coulomb integral over a primitive quartet is an integral over t in [0, 1] of exp(-T t^2) times a polynomial
// of degree L in t^2 that factorises by axis, so n = L/2 + 1 quadrature nodes give it exactly:
//   [ab|cd] = sum_r w_r Ix[ax bx; cx dx]_r Iy[ay by; cy dy]_r Iz[az bz; cz dz]_r .
// The axis tables are the Hermite transforms of this engine with R replaced by a product of one-dimensional
// Hermite functions of node r, h_{m+1} = s (X h_m + m h_{m-1}), s = -2 rho t_r^2 (Eq. r one axis at a time):
//   I[a b; c d]_r = sum_t E^{ab}_t sum_tau (-1)^tau E^{cd}_tau h_{t+tau, r},
// so nothing cancels that does not cancel in the McMurchie-Davidson form (no transfer relation a -> b).
//
// What it costs: 2 n FP64 instructions per integral plus the tables, against the bra and ket steps of the
// axis-factored transforms: [ii|ii] 17.0 M against 28.1 M per shellset, [ff|ff] 0.18 M against 0.24 M. The
// kernel is bound by the FP64 pipe (an SM starts a warp's FP64 instruction every 19 clocks), which leaves three
// shared-memory loads per pair of them free; lanes run over the ket components, so that stores are whole
// lines and a row of a table is read without bank conflicts. The tables of one quartet stay in shared memory up to
// [gg|gg] (135 KB); larger classes keep them in a global area per resident block (749 KB at [ii|ii], L2) and copy the rows
// of one bra component a at a time (107 KB of the block's 163 KB at [ii|ii]: one block of 16 warps per SM, FP64 pipe 85 %
// busy).
// Contracted quartets keep the step programs, which fold the ket primitives before the bra steps.
#include <algorithm>
#include <utility>

#include "kernels.cuh"

namespace mdx {
namespace {

__device__ __forceinline__ int eoff(int lb, int a, int b) {   // etab_off in closed form
  return (lb + 1) * (a * (a + 1) / 2) + a * (lb * (lb + 1) / 2) + b * (a + 1) + b * (b - 1) / 2;
}
// Cartesian component k of shell l (library order): (x, y), z = l - x - y
__device__ __forceinline__ int2 component(int l, int k) {
  int i = 0;
  while (k > i) k -= ++i;   // x = l - i, and y runs from i down
  return make_int2(l - i, i - k);
}

// A free area of the axis tables for this block. Launches that share the areas may overlap on the GPU (runs of a
// batch on several streams, other batches, replayed graphs): there are as many areas as blocks that can be
// resident together, so one is always free, and the search starts at the block's own (the first try succeeds unless
// launches overlap). -1 after a bounded search.
__device__ int take_area(int32_t* used, int n, int first) {
  for (int round = 0; round < 4096; ++round)
    for (int i = 0; i < n; ++i) {
      const int k = first + i < n ? first + i : first + i - n;
      if (atomicCAS(used + k, 0, 1) == 0) {
        __threadfence();   // the last holder's accesses come before this block's
        return k;
      }
    }
  return -1;
}

template <int NR>
struct Rule {
  static constexpr int64_t first = rys_offset(NR);
};

// AREAS: the tables live in global memory, in a free one of a.rys_areas areas. An instance of its own: one that also serves
// the classes with tables in shared memory (and the one-shot calls, whose block b uses area b) costs the smallest of those
// up to 1 %, and dropping the global tables from theirs up to 5 % ([6|10] 374 -> 392 us), by the compiler's
// choice of registers alone.
template <int NR, bool AREAS>
__global__ void __launch_bounds__(512) k_rys(const QuartetLaunch a) {
  extern __shared__ __align__(16) double sm[];
  const PlanDev& P = a.plan;
  const int tid = threadIdx.x, T = blockDim.x;
  const int la = P.la, lb = P.lb, lc = P.lc, ld = P.ld, L = P.L, Lb = P.Lb;
  const int na = (la + 1) * (la + 2) / 2, nb = (lb + 1) * (lb + 2) / 2, nd = (ld + 1) * (ld + 2) / 2;
  const int nab1 = (la + 1) * (lb + 1), ncd1 = (lc + 1) * (ld + 1);   // one-axis index pairs
  const int RS = NR * ncd1;                                           // doubles of a table row (one axis, one ab)
  const int Nb = P.Nb, Nk = P.Nk;
  double* recb = sm;
  double* reck = sm + P.recb;
  double* sr = sm + P.ry_h;                   // -2 rho t_r^2, then pref w_r
  double* h = sr + 2 * NR;                    // [axis][m][r]
  double* Nt = sm + P.ry_N;                   // [axis][t][r][cd of the chunk]
  double* tab = sm + P.ry_T;                  // [axis][ab][r][cd], or the rows of one a
  uint32_t* abt = reinterpret_cast<uint32_t*>(sm + P.ry_idx);   // table rows (x, y, z) of ab
  uint32_t* cdt = abt + Nb;                                     // columns of cd
  uint32_t* rowE = cdt + Nk;                                    // per one-axis ab: E block start, length
  uint32_t* colE = rowE + nab1;                                 // per one-axis cd
  int* area = reinterpret_cast<int*>(colE + ncd1);              // of the tables in global memory
  const bool stash = AREAS || P.ry_stash != 0;
  double* gtab = stash ? a.rys_tab + (int64_t)blockIdx.x * a.rys_stride : tab;
  if constexpr (AREAS) {
    if (tid == 0) {
      *area = take_area(a.rys_used, a.rys_areas, (int)(blockIdx.x % (unsigned)a.rys_areas));
      if (*area < 0) atomicExch(a.err, kDevTimeout);
    }
  }

  for (int e = tid; e < Nb; e += T) {
    const int ia = e / nb, ib = e - ia * nb;
    const int2 A = component(la, ia), B = component(lb, ib);
    const int az = la - A.x - A.y, bz = lb - B.x - B.y, w = lb + 1;
    abt[e] = stash ? (uint32_t)B.x | (uint32_t)(w + B.y) << 8 | (uint32_t)(2 * w + bz) << 16
                   : (uint32_t)(A.x * w + B.x) | (uint32_t)(nab1 + A.y * w + B.y) << 8 |
                         (uint32_t)(2 * nab1 + az * w + bz) << 16;
  }
  for (int e = tid; e < Nk; e += T) {
    const int ic = e / nd, id = e - ic * nd;
    const int2 C = component(lc, ic), D = component(ld, id);
    const int cz = lc - C.x - C.y, dz = ld - D.x - D.y, w = ld + 1;
    cdt[e] = (uint32_t)(C.x * w + D.x) | (uint32_t)(C.y * w + D.y) << 8 | (uint32_t)(cz * w + dz) << 16;
  }
  for (int e = tid; e < nab1; e += T) {
    const int x = e / (lb + 1), y = e - x * (lb + 1);
    rowE[e] = (uint32_t)eoff(lb, x, y) | (uint32_t)(x + y + 1) << 16;
  }
  for (int e = tid; e < ncd1; e += T) {
    const int x = e / (ld + 1), y = e - x * (ld + 1);
    colE[e] = (uint32_t)eoff(ld, x, y) | (uint32_t)(x + y + 1) << 16;
  }
  if constexpr (AREAS) {
    __syncthreads();
    if (*area < 0) return;
    gtab = a.rys_tab + *area * a.rys_stride;
  }
  const int EB = (P.recb - kRecHeader) / 3, EK = (P.reck - kRecHeader) / 3;   // one axis of a record's tables
  // (the record is padded to an even length: the table length is the integer part)

  for (int64_t q = blockIdx.x; q < a.nq; q += gridDim.x) {
    const int2 qp = a.qpairs[q];
    const double* gb = a.recs + a.pair_rec[qp.x + a.bra_var_off];
    const double* gk = a.recs_signed + a.pair_rec[qp.y + a.ket_var_off];
    __syncthreads();   // the previous quartet's readers are done
    for (int i = tid; i < P.recb; i += T) recb[i] = __ldg(gb + i);
    for (int i = tid; i < P.reck; i += T) reck[i] = __ldg(gk + i);
    if (tid < 32) {
      // nodes and weights: lane r < n the node r, lane n + r its weight
      const double zp = __ldg(gb), zq = __ldg(gk);
      const double X = __ldg(gb + 2) - __ldg(gk + 2), Y = __ldg(gb + 3) - __ldg(gk + 3),
                   Z = __ldg(gb + 4) - __ldg(gk + 4);
      const double rs = rsqrt(zp + zq);
      const double rho = zp * zq * rs * rs;
      const double Tb = rho * (X * X + Y * Y + Z * Z);
      const double* t = a.rys + Rule<NR>::first;
      if (tid < 2 * NR) {
        double f;
        if (Tb < (double)kRysIntervals) {
          const int i = min((int)Tb, kRysIntervals - 1);
          const double u = Tb - ((double)i + 0.5);
          const double* c = t + (int64_t)i * (kRysTerms * 2 * NR) + tid;
          f = __ldg(c + (kRysTerms - 1) * 2 * NR);
#pragma unroll
          for (int k = kRysTerms - 2; k >= 0; --k) f = fma(f, u, __ldg(c + k * 2 * NR));
        } else {
          const double y = rsqrt(Tb);
          f = __ldg(t + (int64_t)kRysIntervals * (kRysTerms * 2 * NR) + tid) * (tid < NR ? y * y : y);
        }
        // 2 pi^(5/2) / (zp zq sqrt(zp+zq)) * c_a c_b K_ab * c_c c_d K_cd goes with the weights
        sr[tid] = tid < NR ? -2.0 * rho * f
                           : 34.986836655249725693 * __ldg(gb + 6) * __ldg(gk + 6) * rs * f;
      }
    }
    __syncthreads();
    for (int e = tid; e < 3 * NR; e += T) {
      const int ax = e / NR, r = e - ax * NR;
      const double X = recb[2 + ax] - reck[2 + ax], s = sr[r];
      double* hr = h + ax * (L + 1) * NR + r;
      double h0 = ax == 2 ? sr[NR + r] : 1.0, hm = 0.0;   // the weight goes with z
      hr[0] = h0;
      for (int m = 0; m < L; ++m) {
        const double h1 = s * fma(X, h0, (double)m * hm);
        hr[(m + 1) * NR] = h1;
        hm = h0;
        h0 = h1;
      }
    }
    // axis tables, `ry_cw` of the ket indices c at a time
    for (int c0 = 0; c0 <= lc; c0 += P.ry_cw) {
      const int cw = min(P.ry_cw, lc + 1 - c0) * (ld + 1), cb = c0 * (ld + 1);
      const int RC = NR * cw;
      __syncthreads();
      for (int e = tid; e < 3 * (Lb + 1) * RC; e += T) {
        const int j = e / cw, cd = e - j * cw;
        const int at = j / NR, r = j - at * NR;
        const int ax = at / (Lb + 1), t = at - ax * (Lb + 1);
        const uint32_t w = colE[cb + cd];
        const double* E = reck + kRecHeader + ax * EK + (w & 0xffff);
        const double* hh = h + (ax * (L + 1) + t) * NR + r;
        double v = 0.0;
        for (int k = 0; k < (int)(w >> 16); ++k) v = fma(E[k], hh[k * NR], v);
        Nt[e] = v;
      }
      __syncthreads();
      for (int e = tid; e < 3 * nab1 * RC; e += T) {
        const int row = e / RC, j = e - row * RC;
        const int ax = row / nab1;
        const uint32_t w = rowE[row - ax * nab1];
        const double* E = recb + kRecHeader + ax * EB + (w & 0xffff);
        const double* x = Nt + ax * (Lb + 1) * RC + j;
        double v = 0.0;
        for (int k = 0; k < (int)(w >> 16); ++k) v = fma(E[k], x[k * RC], v);
        if (cw == ncd1) {
          gtab[e] = v;
        } else {
          const int r = j / cw;
          gtab[row * RS + r * ncd1 + cb + (j - r * cw)] = v;
        }
      }
    }
    __syncthreads();
    double* outq = a.out + (a.qout ? a.qout[q] : q * (int64_t)Nb * Nk);
    const int slabs = stash ? na : 1, count = stash ? nb * Nk : Nb * Nk;
    const int de = T / Nk, dc = T - de * Nk;
    int lastx = -1;
    for (int s = 0; s < slabs; ++s) {
      if (stash) {
        const int2 A = component(la, s);
        const int len = (lb + 1) * RS, o[3] = {A.x, A.y, la - A.x - A.y};
        if (s > 0) __syncthreads();
        for (int ax = A.x == lastx ? 1 : 0; ax < 3; ++ax) {
          const double* src = gtab + (int64_t)(ax * nab1 + o[ax] * (lb + 1)) * RS;
          for (int i = tid; i < len; i += T) tab[ax * len + i] = src[i];
        }
        lastx = A.x;
        __syncthreads();
      }
      int ab = tid / Nk, cd = tid - ab * Nk;
      const uint32_t* rows = abt + (stash ? s * nb : 0);
      double* o = outq + (int64_t)s * count;
      for (int e = tid; e < count; e += T) {
        const uint32_t w = rows[ab], c = cdt[cd];
        const double* px = tab + (int)(w & 0xff) * RS + (c & 0xff);
        const double* py = tab + (int)((w >> 8) & 0xff) * RS + ((c >> 8) & 0xff);
        const double* pz = tab + (int)(w >> 16) * RS + (c >> 16);
        double v = 0.0;
#pragma unroll
        for (int r = 0; r < NR; ++r) v = fma(px[r * ncd1] * py[r * ncd1], pz[r * ncd1], v);
        o[e] = v;
        ab += de;
        cd += dc;
        if (cd >= Nk) { cd -= Nk; ++ab; }
      }
    }
  }
  if constexpr (AREAS) {
    __syncthreads();   // every thread has read its tables
    if (tid == 0) {
      __threadfence();
      atomicExch(a.rys_used + *area, 0);
    }
  }
}

using RysKernel = void (*)(const QuartetLaunch);
template <int... I>
RysKernel rys_kernel(int n, bool areas, std::integer_sequence<int, I...>) {
  static const RysKernel table[2][kRysMax] = {{k_rys<I + 1, false>...}, {k_rys<I + 1, true>...}};
  return table[areas][n - 1];
}
RysKernel rys_kernel(int n, bool areas) {
  return n >= 1 && n <= kRysMax ? rys_kernel(n, areas, std::make_integer_sequence<int, kRysMax>{}) : nullptr;
}

}  // namespace

cudaError_t rys_attributes_init() {
  for (int n = 1; n <= kRysMax; ++n)
    for (const bool areas : {false, true}) {
      const cudaError_t e =
          cudaFuncSetAttribute(rys_kernel(n, areas), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

cudaError_t rys_grid(const PlanDev& P, int64_t nq, int* grid, int* resident) {
  *resident = 0;
  if (!P.ry_stash) {
    *grid = (int)std::min<int64_t>(nq, 0x7fffffff);
    return cudaSuccess;
  }
  int bps = 1, dev = 0, sms = 0;   // blocks per SM: the larger number of the two instances
  cudaError_t e = cudaSuccess;
  for (const bool areas : {false, true}) {
    int n = 0;
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, rys_kernel(P.rys, areas), P.ry_threads,
                                                        (size_t)P.ry_doubles * sizeof(double));
    bps = std::max(bps, n);
  }
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  *resident = bps * sms;
  *grid = (int)std::max<int64_t>(1, std::min<int64_t>(nq, *resident));
  return cudaSuccess;
}

cudaError_t launch_rys(const QuartetLaunch& a, int grid, cudaStream_t s) {
  if (a.nq <= 0) return cudaSuccess;
  const PlanDev& P = a.plan;
  const RysKernel k = rys_kernel(P.rys, P.ry_stash && a.rys_used);
  if (!k || !a.rys || a.D || a.grad || grid < 1) return cudaErrorInvalidValue;
  if (P.ry_stash && (!a.rys_tab || a.rys_stride < P.ry_table || a.rys_areas < (a.rys_used ? 1 : grid)))
    return cudaErrorInvalidValue;
  k<<<grid, P.ry_threads, (size_t)P.ry_doubles * sizeof(double), s>>>(a);
  return cudaGetLastError();
}

}  // namespace mdx
