// FP64 CUDA kernels of the HFX force/stress hot path (sm_103a).
//
// Stages of one evaluation (paper Sec. 2 and 3; the factorisation is the
// distributive law applied to Eq. exx_expand):
//   K1  block generation   C, grad C (C pairs); norms of V, grad V (V pairs);
//                          V, grad V blocks for the V pairs the items need
//   K2  screening           step 1 per-tensor norms, step 2 Cauchy-Schwarz
//                          bounds per item (Sec. 3.2, Algorithm 1)
//   K3  Y^{XZ} = sum_W C_XW D_WZ for every key an item needs
//   K4  first exchange product, per (A,B) pair over its kept F:
//          U = D_AB . Y^{BF};  R_AB += <C_AF, U>;  g^C_AF += -2 <grad C_AF, V_AB . U>
//   K5  second exchange product, per (A,B) pair:
//          R2_AB = <Y^{AB}, Y^{BA}>;  Z = V_AB . Y^{BA};  g^C_AF += -2 <grad C_AF, Z . D_FB^T>
//   K7  E = -sum <V, R>, g^V = -<grad V, R>, forces F_I += g, F_J -= g and the
//       virial sum g (x) d that gives sigma = -(1/Omega) sum g (x) d (Eq. stress)
//
// All arithmetic is FP64.  Per-pair gradient contributions from different
// CTAs meet in FP64 atomics (order-dependent only at the last bits).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>

#include "hfx_accum.cuh"
#include "hfx_internal.h"
#include "hfx_model.cuh"

namespace hfx {
namespace {

using namespace model;

constexpr int kThreads = 256;
std::atomic<long long> g_launches{0};   // host-side count of kernel launches (all threads)

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of v over the block; every thread gets the result.  `red` needs
// kThreads/32 doubles of shared memory and is reused across calls.
__device__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  const int nw = (blockDim.x + 31) >> 5;
  for (int i = 0; i < nw; ++i) t += red[i];
  return t;
}

__device__ __forceinline__ int dlut_get(const DevPlan& P, int i, int j, int r0, int r1, int r2) {
  if (r0 < -P.HD0 || r0 > P.HD0 || r1 < -P.HD1 || r1 > P.HD1 || r2 < -P.HD2 || r2 > P.HD2) return -1;
  const long long n0 = 2 * P.HD0 + 1, n1 = 2 * P.HD1 + 1, n2 = 2 * P.HD2 + 1;
  const long long idx = (((((long long)i * P.N + j) * n0 + (r0 + P.HD0)) * n1 + (r1 + P.HD1)) * n2) + (r2 + P.HD2);
  return P.dlut[idx];
}

__device__ __forceinline__ int ylut_get(const DevPlan& P, int i, int j, int r0, int r1, int r2) {
  if (r0 < -P.HY0 || r0 > P.HY0 || r1 < -P.HY1 || r1 > P.HY1 || r2 < -P.HY2 || r2 > P.HY2) return -1;
  const long long n0 = 2 * P.HY0 + 1, n1 = 2 * P.HY1 + 1, n2 = 2 * P.HY2 + 1;
  const long long idx = (((((long long)i * P.N + j) * n0 + (r0 + P.HY0)) * n1 + (r1 + P.HY1)) * n2) + (r2 + P.HY2);
  return P.ylut[idx];
}

// ---------------------------------------------------------------- K2: D norms
__global__ void k_dnorm(DevPlan P) {
  __shared__ double red[kThreads / 32];
  unsigned long long kept = 0;
  for (long long k = blockIdx.x; k < P.n_d; k += gridDim.x) {
    const long long b = P.Doff[k], e = P.Doff[k + 1];
    double s = 0.0;
    for (long long t = b + threadIdx.x; t < e; t += blockDim.x) s += P.Dval[t] * P.Dval[t];
    s = block_sum(s, red);
    if (threadIdx.x == 0) {
      const double n = sqrt(s);
      const bool keep = n > P.thD;
      P.Dkept[k] = keep ? n : 0.0;
      kept += keep;
    }
  }
  if (threadIdx.x == 0 && kept) atomicAdd(&P.cnt[CNT_D], kept);
}

// ---------------------------------------------------------------- K1: C blocks
// One CTA per C pair: C = G f(r) [+ G' f(r) (d.e)/R_C], grad_d C, and the
// step-1 decision ||C|| > theta_C or ||grad C|| > theta_dC.
__global__ void k_cblocks(DevPlan P, int frozen) {
  __shared__ double red[kThreads / 32];
  for (int p = blockIdx.x; p < P.nC; p += gridDim.x) {
    const int A = P.c_home[p], j = P.c_j[p];
    const int* R = P.c_R + 3 * p;
    double d[3];
    pair_vector(P, A, j, R, d);
    const bool onsite = (A == j) && R[0] == 0 && R[1] == 0 && R[2] == 0;
    const double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    double f = 1.0, fp = 0.0;
    if (!onsite) radial_f(r, P.RC, f, fp);
    double g[3] = {0.0, 0.0, 0.0};
    double ga[3] = {0.0, 0.0, 0.0};
    double fa = 0.0;
    if (!onsite) {
#pragma unroll
      for (int c = 0; c < 3; ++c) g[c] = fp * d[c] / r;
      if (P.Gp) {
        const double de = d[0] * P.e[0] + d[1] * P.e[1] + d[2] * P.e[2];
        fa = f * de / P.RC;
#pragma unroll
        for (int c = 0; c < 3; ++c) ga[c] = (fp * (d[c] / r) * de + f * P.e[c]) / P.RC;
      }
    }
    const int sA = P.species[A], sj = P.species[j];
    const long long go = P.G_off[sA * P.S + sj];
    const int n = P.n_abf[sA] * P.n_ao[sA] * P.n_ao[sj];
    if (threadIdx.x < 8) {   // the pair's scalars (c_pair_eval), for the split stores of wide plans
      const double v[8] = {f, fa, g[0], g[1], g[2], ga[0], ga[1], ga[2]};
      P.c_sc[8 * (long long)p + threadIdx.x] = v[threadIdx.x];
    }
    double* C = P.Cst + P.c_off[p];
    double* dC = P.dCst + 3 * P.c_off[p];
    double sc = 0.0, sg = 0.0;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      const double Gv = P.G[go + t];
      double c = Gv * f;
      double g0 = Gv * g[0], g1 = Gv * g[1], g2 = Gv * g[2];
      if (P.Gp && !onsite) {
        const double Gq = P.Gp[go + t];
        c = c + Gq * fa;
        g0 = g0 + Gq * ga[0];
        g1 = g1 + Gq * ga[1];
        g2 = g2 + Gq * ga[2];
      }
      C[t] = c;
      dC[t] = g0;
      dC[n + t] = g1;
      dC[2 * n + t] = g2;
      sc += c * c;
      sg += g0 * g0 + g1 * g1 + g2 * g2;
    }
    sc = block_sum(sc, red);
    sg = block_sum(sg, red);
    if (threadIdx.x == 0) {
      const double nc = sqrt(sc), ng = sqrt(sg);
      bool keep;
      if (frozen) {
        keep = P.c_keep[p] != 0;
      } else {
        keep = (nc > P.thC) || (ng > P.thdC);
        P.c_keep[p] = keep;
      }
      P.c_norm[p] = keep ? fmax(nc, ng) : 0.0;
      if (keep) atomicAdd(&P.cnt[CNT_C], 1ull);
    }
  }
}

// Split path: one thread per C pair.  The scalars of C = G f + G' fa and
// grad_c C = G g_c + G' ga_c are stored for the kernels that write the
// operand stores, and the norms come from the template moments:
// ||C||^2 = f^2 S_GG + 2 f fa S_GG' + fa^2 S_G'G', and the same with
// (g_c, ga_c) summed over c for ||grad C||^2.
__global__ void k_cnorm(DevPlan P, int frozen) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P.nC; p += gridDim.x * blockDim.x) {
    double sc[8];
    c_pair_eval(P, p, sc);
    double* o = P.c_sc + 8 * (long long)p;
#pragma unroll
    for (int k = 0; k < 8; ++k) o[k] = sc[k];
    const double* mo = P.Gmom + 3 * (P.species[P.c_home[p]] * P.S + P.species[P.c_j[p]]);
    const double nc2 = sc[0] * sc[0] * mo[0] + 2.0 * sc[0] * sc[1] * mo[1] + sc[1] * sc[1] * mo[2];
    double ng2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c)
      ng2 += sc[2 + c] * sc[2 + c] * mo[0] + 2.0 * sc[2 + c] * sc[5 + c] * mo[1] + sc[5 + c] * sc[5 + c] * mo[2];
    const double nc = sqrt(fmax(nc2, 0.0)), ng = sqrt(fmax(ng2, 0.0));
    bool keep;
    if (frozen) {
      keep = P.c_keep[p] != 0;
    } else {
      keep = (nc > P.thC) || (ng > P.thdC);
      P.c_keep[p] = keep;
    }
    P.c_norm[p] = keep ? fmax(nc, ng) : 0.0;
    if (keep) atomicAdd(&P.cnt[CNT_C], 1ull);
  }
}

// ---------------------------------------------------------------- K1: V norms
// One thread per V pair.  V = M h(r) and grad_d V = M h'(r) d/r (on-site:
// V = M, grad V = 0), so ||V|| = |h| ||M|| and ||grad V|| = |h'| ||M|| (the
// three components of d/r have unit length): the template norm ||M_st||_F is
// taken once per species pair when the plan is made.
__global__ void k_vnorm(DevPlan P, int frozen) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P.nV; p += gridDim.x * blockDim.x) {
    const int A = P.v_home[p], j = P.v_j[p];
    const int* R = P.v_R + 3 * p;
    const bool onsite = (A == j) && R[0] == 0 && R[1] == 0 && R[2] == 0;
    double h = 1.0, hp = 0.0, g[3] = {0.0, 0.0, 0.0};
    if (!onsite) {
      double d[3];
      pair_vector(P, A, j, R, d);
      const double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
      radial_h(r, P.omega, h, hp);
#pragma unroll
      for (int c = 0; c < 3; ++c) g[c] = hp * d[c] / r;
    }
    double* hg = P.v_hg + 4 * (long long)p;   // for the kernels that evaluate V = M h, grad V = M g
    hg[0] = h;
    hg[1] = g[0];
    hg[2] = g[1];
    hg[3] = g[2];
    const double mn = P.Mnorm[P.species[A] * P.S + P.species[j]];
    const double nv = fabs(h) * mn, ng = fabs(hp) * mn;
    bool keep;
    if (frozen) {
      keep = P.v_keep[p] != 0;
    } else {
      keep = (nv > P.thV) || (ng > P.thdV);
      P.v_keep[p] = keep;
    }
    P.v_norm[p] = keep ? fmax(nv, ng) : 0.0;
    if (keep) atomicAdd(&P.cnt[CNT_V], 1ull);
  }
}

// ---------------------------------------------------------------- K2: yhat
// yhat_{XZ} = sum_{W in C(X), kept} c_XW d_WZ: the factor of the
// Cauchy-Schwarz bounds that sums over the inner atom (Sec. 3.2).
__global__ void k_yhat(DevPlan P) {
  for (int y = blockIdx.x * blockDim.x + threadIdx.x; y < P.nY; y += gridDim.x * blockDim.x) {
    const int X = P.y_home[y], z = P.y_j[y];
    const int* Rz = P.y_R + 3 * y;
    double acc = 0.0;
    for (int q = P.c_ptr[X]; q < P.c_ptr[X + 1]; ++q) {
      const double c = P.c_norm[q];
      if (c == 0.0) continue;
      const int* Rw = P.c_R + 3 * q;
      const int di = dlut_get(P, P.c_j[q], z, Rz[0] - Rw[0], Rz[1] - Rw[1], Rz[2] - Rw[2]);
      if (di < 0) continue;
      acc += c * P.Dkept[di];
    }
    P.yhat[y] = acc;
  }
}

// ---------------------------------------------------------------- K2: items
// One thread per V pair (A,B).  First product: F in C(A) is kept iff
// c_AF v_AB d_AB yhat_BF > theta_CS.  Second product: (A,B) is kept iff
// v_AB yhat_AB yhat_BA > theta_CS.  Marks the Y keys the kept items read.
// Only home atoms A in [h0, h1) have items (the plan's share of the sum over
// A of Eq. exx_expand).
__global__ void k_screen(DevPlan P) {
  unsigned long long trip = 0;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P.nV; p += gridDim.x * blockDim.x) {
    unsigned int mask[kMaskWords];
#pragma unroll
    for (int w = 0; w < kMaskWords; ++w) mask[w] = 0u;
    int t2 = 0;
    const int A = P.v_home[p];
    const double v = (A >= P.h0 && A < P.h1) ? P.v_norm[p] : 0.0;
    if (v > 0.0) {
      const int b = P.v_j[p];
      const int* Rb = P.v_R + 3 * p;
      if (P.terms & 1) {
        const int di = P.v_didx[p];
        const double dab = di >= 0 ? P.Dkept[di] : 0.0;
        if (dab > 0.0) {
          const int q0 = P.c_ptr[A], q1 = P.c_ptr[A + 1];
          for (int q = q0; q < q1; ++q) {
            const double c = P.c_norm[q];
            if (c == 0.0) continue;
            const int* Rf = P.c_R + 3 * q;
            const int yc = ylut_get(P, b, P.c_j[q], Rf[0] - Rb[0], Rf[1] - Rb[1], Rf[2] - Rb[2]);
            if (yc < 0) continue;
            if (c * v * dab * P.yhat[yc] > P.thCS) {
              const int s = q - q0;
              mask[s >> 5] |= 1u << (s & 31);
              P.y_flag[yc] = 1;
              ++trip;
            }
          }
        }
      }
      if (P.terms & 2) {
        const int y1 = ylut_get(P, A, b, Rb[0], Rb[1], Rb[2]);
        const int y2 = ylut_get(P, b, A, -Rb[0], -Rb[1], -Rb[2]);
        if (y1 >= 0 && y2 >= 0 && v * P.yhat[y1] * P.yhat[y2] > P.thCS) {
          t2 = 1;
          P.y_flag[y1] = 1;
          P.y_flag[y2] = 1;
        }
      }
    }
    bool any = t2 != 0;
#pragma unroll
    for (int w = 0; w < kMaskWords; ++w) {
      P.v_mask[(size_t)p * kMaskWords + w] = mask[w];
      any = any || mask[w] != 0u;
    }
    P.v_t2[p] = (unsigned char)t2;
    P.v_flag[p] = any ? 1 : 0;
  }
  if (trip) atomicAdd(&P.cnt[CNT_TRIP], trip);
}

// ---------------------------------------------------------------- K1: V blocks
__global__ void k_vblocks(DevPlan P, const int* list, int n_list) {
  for (int k = blockIdx.x; k < n_list; k += gridDim.x) {
    const int p = list[k];
    const int A = P.v_home[p], j = P.v_j[p];
    double h, g[3];
    v_pair(P, p, h, g);
    const int sA = P.species[A], sj = P.species[j];
    const double* M = P.M + P.M_off[sA * P.S + sj];
    const int n = P.n_abf[sA] * P.n_abf[sj];
    double* V = P.Vst + P.v_off[p];
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      const double m = M[t];
      V[t] = m * h;
      V[n + t] = m * g[0];
      V[2 * n + t] = m * g[1];
      V[3 * n + t] = m * g[2];
    }
  }
}

// ---------------------------------------------------------------- K3: Y
// One CTA per needed key (X; Z): Y[alpha,x,z] = sum_{W kept} sum_w
// C_XW[alpha,x,w] D_WZ[w,z], D_WZ = D(w, z, R_Z - R_W) when kept.
// A CTA takes one of P.parts ranges of the key's elements: with whole keys the
// last wave of a small cell left most SMs idle (5-atom perovskite 17.1 ms, 13.8 now: 1.0 TFLOP/s).
__global__ void k_ybuild(DevPlan P, const int* list, int n_list) {
  __shared__ int dsel[kMaxCPerAtom];
  for (int u = blockIdx.x; u < n_list * P.parts; u += gridDim.x) {
    const int k = u / P.parts, part = u - k * P.parts;
    const int y = list[k];
    const int X = P.y_home[y], z = P.y_j[y];
    const int* Rz = P.y_R + 3 * y;
    const int q0 = P.c_ptr[X], nq = P.c_ptr[X + 1] - q0;
    __syncthreads();
    for (int t = threadIdx.x; t < nq; t += blockDim.x) {
      const int q = q0 + t;
      int di = -1;
      if (P.c_keep[q]) {
        const int* Rw = P.c_R + 3 * q;
        di = dlut_get(P, P.c_j[q], z, Rz[0] - Rw[0], Rz[1] - Rw[1], Rz[2] - Rw[2]);
        if (di >= 0 && P.Dkept[di] == 0.0) di = -1;
      }
      dsel[t] = di;
    }
    __syncthreads();
    const int sX = P.species[X];
    const int mX = P.n_abf[sX], nX = P.n_ao[sX], nZ = P.n_ao[P.species[z]];
    const int rows = mX * nX;
    const int n = rows * nZ;
    double* Y = P.Yst + P.y_off[y];
    double fl = 0.0;
    const int e1 = (int)((long long)n * (part + 1) / P.parts);
    for (int e = (int)((long long)n * part / P.parts) + threadIdx.x; e < e1; e += blockDim.x) {
      const int row = e / nZ, col = e - row * nZ;
      double acc = 0.0;
      for (int t = 0; t < nq; ++t) {
        const int di = dsel[t];
        if (di < 0) continue;
        const int q = q0 + t;
        const int nW = P.n_ao[P.species[P.c_j[q]]];
        const double* Cq = P.Cst + P.c_off[q] + (long long)row * nW;
        const double* Dq = P.Dval + P.Doff[di] + col;
        for (int w = 0; w < nW; ++w) acc += Cq[w] * Dq[w * nZ];
        if (e == 0) fl += 2.0 * (double)n * nW;
      }
      Y[e] = acc;
    }
    if (threadIdx.x == 0 && fl != 0.0) atomicAdd(&P.acc[ACC_FY], fl);
  }
}

// The warps' parts of <V_AB, R> and <grad V_AB, R>, added up by four threads
// into E and g^V of pair p (behind a barrier).
__device__ __forceinline__ void add_pair(const DevPlan& P, int p, const double (*ew)[4], int nwarp) {
  if (threadIdx.x >= 4) return;
  double s = 0.0;
  for (int k = 0; k < nwarp; ++k) s += ew[k][threadIdx.x];
  if (s == 0.0) return;
  if (threadIdx.x == 0) dev::add_E(P, -s, blockIdx.x & (kESlots - 1));
  else dev::add_gV(P, 3 * p + (int)threadIdx.x - 1, -s);
}

// ---------------------------------------------------------------- K4: term 1
// One CTA per (A,B) pair with kept F.  Shared memory: D_AB, R_AB, and a
// beta-chunk of U (bc x n_ao(A) x n_ao(F)).
//
// The FP64 pipe bounds it (1.1 TFLOP/s on the whole chip).  The warps leave
// their parts of a gradient in shared memory, where three threads add them up
// behind the next F's barrier, so the only block barriers are the two around a
// chunk of U.  (Eight atomic additions, one per warp, cost the same time and
// left E and F 2 to 5 times further off.)  A chunk is all of U where that leaves room for
// two or three CTAs per SM (they fill each other's barriers), else as much as
// fits: every chunk repeats the three products with grad C.  Small blocks take
// 64 threads per CTA, and small cells divide a pair's F over P.parts CTAs, so
// that the last wave is short.  With block sums per F, 256 threads and whole
// pairs: 1.31 ms on the 8-atom minimal cell (0.58 now) and 47.1 ms on the
// 5-atom perovskite (45.6 now, 0.91 TFLOP/s).
__global__ void k_term1(DevPlan P, const int* list, int n_list, int BC) {
  extern __shared__ double sm[];
  __shared__ double gw[2][kThreads / 32][3], ew[kThreads / 32][4];   // the warps' parts, of this and the last F
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int u = blockIdx.x; u < n_list * P.parts; u += gridDim.x) {
    const int part = u % P.parts, p = list[u / P.parts];
    const int A = P.v_home[p], b = P.v_j[p];
    const int* Rb = P.v_R + 3 * p;
    const int sA = P.species[A], sB = P.species[b];
    const int nA = P.n_ao[sA], nB = P.n_ao[sB], mA = P.n_abf[sA], mB = P.n_abf[sB];
    double* Dab = sm;                      // nA*nB
    double* Rs = Dab + nA * nB;            // mA*mB
    double* Uc = Rs + mA * mB;             // BC*nA*nF
    const double* Dg = P.Dval + P.Doff[P.v_didx[p]];
    const double* V = P.Vst + P.v_off[p];  // [alpha][beta]
    __syncthreads();
    for (int t = threadIdx.x; t < nA * nB; t += blockDim.x) Dab[t] = Dg[t];
    for (int t = threadIdx.x; t < mA * mB; t += blockDim.x) Rs[t] = 0.0;
    __syncthreads();
    const int q0 = P.c_ptr[A];
    double fl = 0.0;
    int turn = 0;   // this part's F: every P.parts-th kept one
    int last = -1, buf = 0;   // C pair whose parts are in gw[buf ^ 1]
    auto add_last = [&]() {   // (behind a barrier)
      if (last < 0 || threadIdx.x >= 3) return;
      double g = 0.0;
      for (int k = 0; k < nwarp; ++k) g += gw[buf ^ 1][k][threadIdx.x];
      if (g != 0.0) dev::add_gC(P, 3 * last + threadIdx.x, -2.0 * g);
    };
    for (int w = 0; w < kMaskWords; ++w) {
      unsigned bits = P.v_mask[(size_t)p * kMaskWords + w];
      while (bits) {
        const int s = __ffs(bits) - 1;
        bits &= bits - 1u;
        const bool mine = turn == part;
        if (++turn == P.parts) turn = 0;
        if (!mine) continue;
        const int q = q0 + w * 32 + s;
        const int f = P.c_j[q];
        const int* Rf = P.c_R + 3 * q;
        const int nF = P.n_ao[P.species[f]];
        const int yc = ylut_get(P, b, f, Rf[0] - Rb[0], Rf[1] - Rb[1], Rf[2] - Rb[2]);
        const double* Y = P.Yst + P.y_off[yc];          // [beta][b][f]
        const double* C = P.Cst + P.c_off[q];           // [alpha][a][f]
        const double* dC = P.dCst + 3 * P.c_off[q];
        const int naf = nA * nF;
        const int nc = mA * naf;
        double g0 = 0.0, g1 = 0.0, g2 = 0.0;
        for (int b0 = 0; b0 < mB; b0 += BC) {
          const int bc = min(BC, mB - b0);
          // U_c[bl][a][f] = sum_b D_AB[a][b] Y[b0+bl][b][f]
          for (int e = threadIdx.x; e < bc * naf; e += blockDim.x) {
            const int bl = e / naf, af = e - bl * naf;
            const int a = af / nF, ff = af - a * nF;
            const double* Yr = Y + ((long long)(b0 + bl) * nB) * nF + ff;
            const double* Dr = Dab + a * nB;
            double s2 = 0.0;
            for (int bb = 0; bb < nB; ++bb) s2 += Dr[bb] * Yr[bb * nF];
            Uc[e] = s2;
          }
          __syncthreads();
          if (b0 == 0) add_last();
          // R[alpha][b0+bl] += sum_{a,f} C[alpha][a][f] U_c[bl][a][f]
          for (int e = threadIdx.x; e < mA * bc; e += blockDim.x) {
            const int al = e / bc, bl = e - al * bc;
            const double* Cr = C + (long long)al * naf;
            const double* Ur = Uc + bl * naf;
            double s2 = 0.0;
            for (int t = 0; t < naf; ++t) s2 += Cr[t] * Ur[t];
            Rs[al * mB + b0 + bl] += s2;
          }
          // (V_AB . U)[alpha][a][f] over this chunk, dotted with grad C_AF
          for (int e = threadIdx.x; e < nc; e += blockDim.x) {
            const int al = e / naf, af = e - al * naf;
            const double* Vr = V + (long long)al * mB + b0;
            double s2 = 0.0;
            for (int bl = 0; bl < bc; ++bl) s2 += Vr[bl] * Uc[bl * naf + af];
            g0 += dC[e] * s2;
            g1 += dC[nc + e] * s2;
            g2 += dC[2 * nc + e] * s2;
          }
          __syncthreads();
        }
        g0 = warp_sum(g0);
        g1 = warp_sum(g1);
        g2 = warp_sum(g2);
        if (lane < 3) gw[buf][warp][lane] = lane == 0 ? g0 : lane == 1 ? g1 : g2;
        last = q;
        buf ^= 1;
        if (threadIdx.x == 0) fl += 2.0 * mB * nA * nB * nF + 4.0 * mA * mB * nA * nF;
      }
    }
    // E += -<V_AB, R>,  g^V += -<grad V_AB, R> (the last chunk's barrier orders R)
    const int n = mA * mB;
    double e0 = 0.0, h0 = 0.0, h1 = 0.0, h2 = 0.0;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      const double r = Rs[t];
      e0 += V[t] * r;
      h0 += V[n + t] * r;
      h1 += V[2 * n + t] * r;
      h2 += V[3 * n + t] * r;
    }
    e0 = warp_sum(e0);
    h0 = warp_sum(h0);
    h1 = warp_sum(h1);
    h2 = warp_sum(h2);
    if (lane < 4) ew[warp][lane] = lane == 0 ? e0 : lane == 1 ? h0 : lane == 2 ? h1 : h2;
    __syncthreads();
    add_last();
    add_pair(P, p, ew, nwarp);
    if (threadIdx.x == 0) atomicAdd(&P.acc[ACC_F1], fl);
  }
}

// ---------------------------------------------------------------- K5: term 2
// One CTA per (A,B) pair of the second exchange product and one of P.parts2
// ranges of alpha.  Shared memory: per-F gradient partials and an alpha-chunk
// of Z (ac x n_ao(A) x n_ao(B)).  Q2 takes one F per warp at a time (D_FB
// straight from L1: a few KB), with no block barrier but the two around a
// chunk of Z.  With one F per block, block sums and whole pairs: 1.99 ms on
// the 8-atom minimal cell (0.35 now), 24.9 ms on the 5-atom perovskite (22.2
// now).
__global__ void k_term2(DevPlan P, const int* list, int n_list, int AC) {
  extern __shared__ double sm[];
  __shared__ double ew[kThreads / 32][4];   // the warps' parts of E and g^V
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int u = blockIdx.x; u < n_list * P.parts2; u += gridDim.x) {
    const int part = u % P.parts2, p = list[u / P.parts2];
    const int A = P.v_home[p], b = P.v_j[p];
    const int* Rb = P.v_R + 3 * p;
    const int sA = P.species[A], sB = P.species[b];
    const int nA = P.n_ao[sA], nB = P.n_ao[sB], mA = P.n_abf[sA], mB = P.n_abf[sB];
    const int m0 = mA * part / P.parts2, m1 = mA * (part + 1) / P.parts2;   // this CTA's rows alpha
    const int y1 = ylut_get(P, A, b, Rb[0], Rb[1], Rb[2]);
    const int y2 = ylut_get(P, b, A, -Rb[0], -Rb[1], -Rb[2]);
    const double* Yab = P.Yst + P.y_off[y1];   // [alpha][a][b]
    const double* Yba = P.Yst + P.y_off[y2];   // [beta][b][a]
    const double* V = P.Vst + P.v_off[p];
    const int nvb = mA * mB;
    const int nab = nA * nB;
    // R2[alpha][beta] = sum_{a,b} Yab[alpha][a][b] Yba[beta][b][a], dotted at once
    double e0 = 0.0, h0 = 0.0, h1 = 0.0, h2 = 0.0;
    for (int t = m0 * mB + threadIdx.x; t < m1 * mB; t += blockDim.x) {
      const int al = t / mB, be = t - al * mB;
      const double* Ya = Yab + (long long)al * nab;
      const double* Yb = Yba + (long long)be * nab;
      double s2 = 0.0;
      for (int a = 0; a < nA; ++a)
        for (int bb = 0; bb < nB; ++bb) s2 += Ya[a * nB + bb] * Yb[bb * nA + a];
      e0 += V[t] * s2;
      h0 += V[nvb + t] * s2;
      h1 += V[2 * nvb + t] * s2;
      h2 += V[3 * nvb + t] * s2;
    }
    e0 = warp_sum(e0);
    h0 = warp_sum(h0);
    h1 = warp_sum(h1);
    h2 = warp_sum(h2);
    if (lane < 4) ew[warp][lane] = lane == 0 ? e0 : lane == 1 ? h0 : lane == 2 ? h1 : h2;
    const int q0 = P.c_ptr[A], nq = P.c_ptr[A + 1] - q0;
    double* gF = sm;                        // nq*3: component c of an F by lane c of the warp that takes it, and no other
    double* Zc = gF + 3 * kMaxCPerAtom;     // AC*nA*nB
    for (int t = warp; t < nq; t += nwarp)
      if (lane < 3) gF[3 * t + lane] = 0.0;
    double fl = threadIdx.x == 0 ? 4.0 * (m1 - m0) * mB * nA * nB : 0.0;
    for (int a0 = m0; a0 < m1; a0 += AC) {
      const int ac = min(AC, m1 - a0);
      __syncthreads();
      if (a0 == m0) add_pair(P, p, ew, nwarp);
      // Z[al][a][b] = sum_beta V[a0+al][beta] Yba[beta][b][a]
      for (int e = threadIdx.x; e < ac * nab; e += blockDim.x) {
        const int al = e / nab, ab = e - al * nab;
        const int a = ab / nB, bb = ab - a * nB;
        const double* Vr = V + (long long)(a0 + al) * mB;
        double s2 = 0.0;
        for (int be = 0; be < mB; ++be) s2 += Vr[be] * Yba[(long long)be * nab + bb * nA + a];
        Zc[e] = s2;
      }
      __syncthreads();
      for (int t = warp; t < nq; t += nwarp) {
        const int q = q0 + t;
        if (!P.c_keep[q]) continue;
        const int f = P.c_j[q];
        const int* Rf = P.c_R + 3 * q;
        const int di = dlut_get(P, f, b, Rb[0] - Rf[0], Rb[1] - Rf[1], Rb[2] - Rf[2]);
        if (di < 0 || P.Dkept[di] == 0.0) continue;
        const int nF = P.n_ao[P.species[f]];
        const double* Dfb = P.Dval + P.Doff[di];   // [f][b]
        const double* dC = P.dCst + 3 * P.c_off[q];
        const int naf = nA * nF;
        const int nc = mA * naf;
        double g0 = 0.0, g1 = 0.0, g2 = 0.0;
        // Q2[a0+al][a][f] = sum_b Z[al][a][b] D_FB[f][b]
        for (int e = lane; e < ac * naf; e += 32) {
          const int al = e / naf, af = e - al * naf;
          const int a = af / nF, ff = af - a * nF;
          const double* Zr = Zc + (long long)al * nab + a * nB;
          const double* Dr = Dfb + ff * nB;
          double s2 = 0.0;
          for (int bb = 0; bb < nB; ++bb) s2 += Zr[bb] * Dr[bb];
          const long long ci = (long long)(a0 + al) * naf + af;
          g0 += dC[ci] * s2;
          g1 += dC[nc + ci] * s2;
          g2 += dC[2 * nc + ci] * s2;
        }
        g0 = warp_sum(g0);
        g1 = warp_sum(g1);
        g2 = warp_sum(g2);
        if (lane < 3) gF[3 * t + lane] += lane == 0 ? g0 : lane == 1 ? g1 : g2;
        if (lane == 0) fl += 2.0 * ac * nA * nB * nF;
      }
    }
    for (int t = warp; t < nq; t += nwarp)
      if (lane < 3 && gF[3 * t + lane] != 0.0) dev::add_gC(P, 3 * (q0 + t) + lane, -2.0 * gF[3 * t + lane]);
    if (lane == 0) atomicAdd(&P.acc[ACC_F2], fl);
    __syncthreads();   // gF and Zc are free for the next pair
  }
}

// ---------------------------------------------------------------- K7: reduce
// Forces F_I += g, F_J -= g for every pair p = (I -> J, R) and the virial
// sum g (x) d.  out = [E, F (n*3), sigma (9)]; E and the virial come from acc.
__global__ void k_reduce_pairs(DevPlan P, double* F) {
  __shared__ double red[kThreads / 32];
  double w[9];
#pragma unroll
  for (int c = 0; c < 9; ++c) w[c] = 0.0;
  const int total = P.nC + P.nV;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    int A, j;
    const int* R;
    double g[3];
    if (t < P.nC) {
      A = P.c_home[t];
      j = P.c_j[t];
      R = P.c_R + 3 * t;
      g[0] = dev::get_gC(P, 3LL * t);
      g[1] = dev::get_gC(P, 3LL * t + 1);
      g[2] = dev::get_gC(P, 3LL * t + 2);
    } else {
      const int p = t - P.nC;
      A = P.v_home[p];
      j = P.v_j[p];
      R = P.v_R + 3 * p;
      g[0] = dev::get_gV(P, 3LL * p);
      g[1] = dev::get_gV(P, 3LL * p + 1);
      g[2] = dev::get_gV(P, 3LL * p + 2);
    }
    if (g[0] == 0.0 && g[1] == 0.0 && g[2] == 0.0) continue;
    double d[3];
    pair_vector(P, A, j, R, d);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (P.fxF) {   // deterministic plan: exact cells, written to F by k_finish
        dev::fx_add(P.fxF + 2 * (3 * A + c), g[c]);
        dev::fx_add(P.fxF + 2 * (3 * j + c), -g[c]);
      } else {
        atomicAdd(&F[3 * A + c], g[c]);
        atomicAdd(&F[3 * j + c], -g[c]);
      }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int c = 0; c < 3; ++c) w[3 * a + c] += g[a] * d[c];
  }
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    const double s = block_sum(w[c], red);
    if (threadIdx.x == 0 && s != 0.0) dev::add_W(P, c, s);
  }
}

__global__ void k_finish(DevPlan P, double* out) {
  if (P.fxF)
    for (int i = threadIdx.x; i < 3 * P.N; i += blockDim.x) out[1 + i] = dev::fx_get(P.fxF + 2 * i);
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double L[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) L[k] = P.L[k];
  const double det = L[0] * (L[4] * L[8] - L[5] * L[7]) - L[1] * (L[3] * L[8] - L[5] * L[6]) +
                     L[2] * (L[3] * L[7] - L[4] * L[6]);
  const double vol = fabs(det);
  out[0] = dev::get_E(P);
  double* sig = out + 1 + 3 * P.N;
  for (int c = 0; c < 9; ++c) sig[c] = -dev::get_W(P, c) / vol;
}

// ---------------------------------------------------------------- scans
__device__ __forceinline__ long long scan_value(const int* flag, const long long* size, const unsigned* mask,
                                                const unsigned char* bytes, int mode, int i) {
  switch (mode) {
    case 0: return flag[i] != 0 ? 1 : 0;
    case 1: return flag[i] != 0 ? size[i] : 0;
    case 2: {
      unsigned any = 0u;
      for (int w = 0; w < kMaskWords; ++w) any |= mask[(size_t)i * kMaskWords + w];
      return any ? 1 : 0;
    }
    case 3: return bytes[i] != 0 ? 1 : 0;
    default: return flag[i];
  }
}

constexpr int kScanItems = 4;
constexpr int kScanTile = kThreads * kScanItems;

// Block-local exclusive scan of a tile; writes block totals.
template <bool kFromValues>
__global__ void k_scan_tile(const int* flag, const long long* size, const unsigned* mask,
                            const unsigned char* bytes, int mode, const long long* vin, int n, long long* out,
                            long long* block_tot) {
  __shared__ long long wsum[kThreads / 32];
  const int base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  long long v[kScanItems];
  long long s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const int i = base + k;
    long long x = 0;
    if (i < n) x = kFromValues ? vin[i] : scan_value(flag, size, mask, bytes, mode, i);
    v[k] = s;
    s += x;
  }
  // inclusive warp scan of per-thread sums
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  long long incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) wsum[wid] = incl;
  __syncthreads();
  long long wpre = 0;
  for (int w = 0; w < wid; ++w) wpre += wsum[w];
  const long long excl = wpre + incl - s;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const int i = base + k;
    if (i < n) out[i] = excl + v[k];
  }
  if (threadIdx.x == blockDim.x - 1) block_tot[blockIdx.x] = excl + s;
}

__global__ void k_scan_add(long long* out, int n, const long long* block_pre) {
  const int i = blockIdx.x * kScanTile + threadIdx.x;
  const long long a = block_pre[blockIdx.x];
  for (int k = 0; k < kScanItems; ++k) {
    const int j = i + k * kThreads;
    if (j < n && j < (blockIdx.x + 1) * kScanTile) out[j] += a;
  }
}

__global__ void k_scan_total(const long long* out, const int* flag, const long long* size, const unsigned* mask,
                             const unsigned char* bytes, int mode, int n, long long* total) {
  if (threadIdx.x == 0 && blockIdx.x == 0)
    *total = n > 0 ? out[n - 1] + scan_value(flag, size, mask, bytes, mode, n - 1) : 0;
}

__global__ void k_scatter(const int* flag, const unsigned* mask, const unsigned char* bytes, int mode, int n,
                          const long long* off, int* list, int base) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    if (scan_value(flag, nullptr, mask, bytes, mode == 1 ? 0 : mode, i)) list[off[i]] = base + i;
}

int grid_for(long long n, int per_block, int cap = 152 * 32) {
  long long g = (n + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

// Recursive exclusive scan of values (block totals) in place into out.
cudaError_t scan_values(long long* vals, int n, long long* out, long long* tmp, size_t tmp_cap, cudaStream_t s) {
  const int nb = (n + kScanTile - 1) / kScanTile;
  if ((size_t)nb > tmp_cap) return cudaErrorInvalidValue;
  ++g_launches;
  k_scan_tile<true><<<nb, kThreads, 0, s>>>(nullptr, nullptr, nullptr, nullptr, 0, vals, n, out, tmp);
  if (nb > 1) {
    cudaError_t e = scan_values(tmp, nb, tmp, tmp + nb, tmp_cap - nb, s);
    if (e != cudaSuccess) return e;
    ++g_launches;
    k_scan_add<<<nb, kThreads, 0, s>>>(out, n, tmp);
  }
  return cudaGetLastError();
}

}  // namespace

long long launch_count() { return g_launches; }

// Block totals plus the levels of the recursive scan fit in 2*nb + 64.
size_t scan_tmp_need(int n) {
  const size_t nb = n > 0 ? ((size_t)n + kScanTile - 1) / kScanTile : 0;
  return 2 * nb + 64;
}

cudaError_t scan_flags(const int* flag, const long long* size, const unsigned* mask, const unsigned char* bytes,
                       int mode, int n, long long* out, long long* total, ScanTmp& tmp, cudaStream_t s) {
  if (n <= 0) {
    cudaError_t e = cudaMemsetAsync(total, 0, sizeof(long long), s);
    return e;
  }
  const int nb = (n + kScanTile - 1) / kScanTile;
  const size_t need = scan_tmp_need(n);
  if (tmp.cap < need) {
    if (tmp.fixed) return cudaErrorMemoryAllocation;
    tmp.mem.put(tmp.buf, tmp.cap * sizeof(long long));
    tmp.buf = nullptr;
    tmp.cap = 0;
    void* p = nullptr;
    cudaError_t e = tmp.mem.get(&p, need * sizeof(long long));
    if (e != cudaSuccess) return e;
    tmp.buf = static_cast<long long*>(p);
    tmp.cap = need;
  }
  ++g_launches;
  k_scan_tile<false><<<nb, kThreads, 0, s>>>(flag, size, mask, bytes, mode, nullptr, n, out, tmp.buf);
  if (nb > 1) {
    cudaError_t e = scan_values(tmp.buf, nb, tmp.buf, tmp.buf + nb, tmp.cap - nb, s);
    if (e != cudaSuccess) return e;
    ++g_launches;
    k_scan_add<<<nb, kThreads, 0, s>>>(out, n, tmp.buf);
  }
  ++g_launches;
  k_scan_total<<<1, 32, 0, s>>>(out, flag, size, mask, bytes, mode, n, total);
  return cudaGetLastError();
}

cudaError_t scatter_list(const int* flag, const unsigned* mask, const unsigned char* bytes, int mode, int n,
                         const long long* off, int* list, int base, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  ++g_launches;
  k_scatter<<<grid_for(n, kThreads), kThreads, 0, s>>>(flag, mask, bytes, mode, n, off, list, base);
  return cudaGetLastError();
}

cudaError_t launch_dnorm(const DevPlan& P, cudaStream_t s) {
  if (P.n_d == 0) return cudaSuccess;
  ++g_launches;
  k_dnorm<<<grid_for(P.n_d, 1, 152 * 64), kThreads, 0, s>>>(P);
  return cudaGetLastError();
}

cudaError_t launch_cblocks(const DevPlan& P, int frozen, cudaStream_t s) {
  if (P.nC == 0) return cudaSuccess;
  ++g_launches;
  k_cblocks<<<grid_for(P.nC, 1, 152 * 64), kThreads, 0, s>>>(P, frozen);
  return cudaGetLastError();
}

cudaError_t launch_cnorm(const DevPlan& P, int frozen, cudaStream_t s) {
  if (P.nC == 0) return cudaSuccess;
  ++g_launches;
  k_cnorm<<<grid_for(P.nC, kThreads), kThreads, 0, s>>>(P, frozen);
  return cudaGetLastError();
}

cudaError_t launch_vnorm(const DevPlan& P, int frozen, cudaStream_t s) {
  if (P.nV == 0) return cudaSuccess;
  ++g_launches;
  k_vnorm<<<grid_for(P.nV, kThreads), kThreads, 0, s>>>(P, frozen);
  return cudaGetLastError();
}

cudaError_t launch_yhat(const DevPlan& P, cudaStream_t s) {
  if (P.nY == 0) return cudaSuccess;
  ++g_launches;
  k_yhat<<<grid_for(P.nY, kThreads), kThreads, 0, s>>>(P);
  return cudaGetLastError();
}

cudaError_t launch_screen(const DevPlan& P, cudaStream_t s) {
  if (P.nV == 0) return cudaSuccess;
  ++g_launches;
  k_screen<<<grid_for(P.nV, kThreads), kThreads, 0, s>>>(P);
  return cudaGetLastError();
}

cudaError_t launch_vblocks(const DevPlan& P, const int* list, int n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  ++g_launches;
  k_vblocks<<<grid_for(n, 1, 152 * 64), kThreads, 0, s>>>(P, list, n);
  return cudaGetLastError();
}

cudaError_t launch_ybuild(const DevPlan& P, const int* list, int n, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  ++g_launches;
  k_ybuild<<<grid_for((long long)n * P.parts, 1, 152 * 64), P.small ? 64 : kThreads, 0, s>>>(P, list, n);
  return cudaGetLastError();
}

cudaError_t allow_max_dynamic_smem(const void* f) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes a{};
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, f);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)a.sharedSizeBytes);
}

cudaError_t set_kernel_smem_limits() {
  cudaError_t e = allow_max_dynamic_smem((const void*)k_term1);
  if (e != cudaSuccess) return e;
  return allow_max_dynamic_smem((const void*)k_term2);
}

cudaError_t launch_term1(const DevPlan& P, const int* list, int n, int beta_chunk, size_t smem, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  ++g_launches;
  k_term1<<<grid_for((long long)n * P.parts, 1, 152 * 64), P.small ? 64 : kThreads, smem, s>>>(P, list, n, beta_chunk);
  return cudaGetLastError();
}

cudaError_t launch_term2(const DevPlan& P, const int* list, int n, int alpha_chunk, size_t smem, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  ++g_launches;
  k_term2<<<grid_for((long long)n * P.parts2, 1, 152 * 64), P.small ? 64 : kThreads, smem, s>>>(P, list, n, alpha_chunk);
  return cudaGetLastError();
}

// ------------------------------------------------------------ LRI fit
// Eq. C_VA and the gradient equation after Eq. V_inverse, per atom pair p of
// a batch:
//   A X = B                       X = the C^I rows, then the C^K rows
//   A dX[c] = dB[c] - dA[c] X     c = x, y, z (gradient in K's position)
// A (n x n, SPD) is factored as L L^T (right-looking Cholesky, L in shared
// memory as the packed lower triangle, column after column).  A CTA then
// solves 32 RHS columns of a pair, one per lane: X in one warp, then the
// three components of dX in three.  A lane runs the product dA[c] X and
// both substitutions in blocks of eight rows held in registers: eight
// independent chains, one load of the column per eight multiply-adds, and no
// division (reciprocals of the diagonal with one correction).  Several CTAs
// share an SM, so that one's loads and barriers hide behind another's FP64
// work, which bounds it (n = 100, w = 169 with gradients: 512 pairs 13.9 ms =
// 0.89 TFLOP/s; 128 pairs, 5 CTAs per SM, 4.7 + 0.2 ms.  One CTA per pair, a row
// at a time with its column in global memory: 0.72 TFLOP/s).  A pivot <= 0 (A
// not positive definite) sets *err and is replaced by 1 so that the CTA finishes.
namespace {

constexpr int kLriCols = 32;   // columns per CTA
constexpr int kLB = 8;   // rows per block

// L(i, k), i >= k, of the packed triangle
__device__ __forceinline__ int lri_at(int i, int k, int n) { return k * n - k * (k + 1) / 2 + i; }

// L and the reciprocals of its diagonal (inv).  A pivot is A's element less the
// sum of its row's squares, which inv holds until then: with each square
// subtracted from the element in turn, X and dX were 1.25 times further off
// (n 55 and 100).  After each column the rest of
// the triangle is updated by all warps, a column each at a time: the work
// spreads over the SM's four FP64 pipes.
__device__ void lri_cholesky(double* L, double* inv, const double* A, int n, int* err) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = (blockDim.x + 31) >> 5;
  for (int e = tid; e < n * n; e += blockDim.x) {
    const int i = e / n, k = e - i * n;
    if (k <= i) L[lri_at(i, k, n)] = A[e];
  }
  for (int i = tid; i < n; i += blockDim.x) inv[i] = 0.0;
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    double* Lj = L + lri_at(0, j, n);   // column j, by row
    if (tid == 0) {
      double d = Lj[j] - inv[j];
      if (!(d > 0.0)) {
        atomicExch(err, 1);
        d = 1.0;
      }
      const double r = rsqrt(d);
      Lj[j] = d * r;
      inv[j] = r;
    }
    __syncthreads();
    const double ljj = Lj[j], rj = inv[j];
    for (int i = j + 1 + tid; i < n; i += blockDim.x) {
      const double t = Lj[i], y = t * rj, l = y + rj * (t - ljj * y);
      Lj[i] = l;
      inv[i] += l * l;
    }
    __syncthreads();
    for (int k = j + 1 + warp; k < n; k += nwarp) {
      double* Lk = L + lri_at(0, k, n);
      const double ljk = Lj[k];
      for (int i = k + 1 + lane; i < n; i += 32) Lk[i] -= Lj[i] * ljk;
    }
    __syncthreads();
  }
}

// One RHS column: out = L^-T L^-1 (rhs - M x), M (n x n, row-major) and x (its
// column, stride w) optional; rhs and out have stride w (out is written in the
// forward pass and read back by the same thread).
__device__ void lri_column(const double* L, const double* inv, int n, int w, const double* rhs, const double* M,
                           const double* x, double* out) {
  for (int i0 = 0; i0 < n; i0 += kLB) {   // L y = rhs - M x
    const int nb = min(kLB, n - i0);
    double a[kLB];
#pragma unroll
    for (int r = 0; r < kLB; ++r) a[r] = r < nb ? rhs[(size_t)(i0 + r) * w] : 0.0;
    if (M)
#pragma unroll 4
      for (int j = 0; j < n; ++j) {
        const double xj = x[(size_t)j * w];
#pragma unroll
        for (int r = 0; r < kLB; ++r)
          if (r < nb) a[r] -= M[(size_t)(i0 + r) * n + j] * xj;
      }
#pragma unroll 4
    for (int k = 0; k < i0; ++k) {
      const double yk = out[(size_t)k * w];
      const double* Lk = L + lri_at(i0, k, n);
#pragma unroll
      for (int r = 0; r < kLB; ++r)
        if (r < nb) a[r] -= Lk[r] * yk;
    }
#pragma unroll
    for (int r = 0; r < kLB; ++r)
      if (r < nb) {
        const double* Lr = L + lri_at(i0 + r, i0 + r, n);   // column i0 + r from the diagonal down
        const double ri = inv[i0 + r], y0 = a[r] * ri, y = y0 + ri * (a[r] - Lr[0] * y0);
        out[(size_t)(i0 + r) * w] = y;
#pragma unroll
        for (int t = r + 1; t < kLB; ++t)
          if (t < nb) a[t] -= Lr[t - r] * y;
      }
  }
  for (int i0 = (n - 1) / kLB * kLB; i0 >= 0; i0 -= kLB) {   // L^T x = y
    const int nb = min(kLB, n - i0);
    double a[kLB];
#pragma unroll
    for (int r = 0; r < kLB; ++r) a[r] = r < nb ? out[(size_t)(i0 + r) * w] : 0.0;
#pragma unroll 4
    for (int k = i0 + nb; k < n; ++k) {
      const double xk = out[(size_t)k * w];
#pragma unroll
      for (int r = 0; r < kLB; ++r)
        if (r < nb) a[r] -= L[lri_at(k, i0 + r, n)] * xk;
    }
#pragma unroll
    for (int r = kLB - 1; r >= 0; --r)
      if (r < nb) {
        const double ri = inv[i0 + r], y0 = a[r] * ri;
        const double y = y0 + ri * (a[r] - L[lri_at(i0 + r, i0 + r, n)] * y0);
        out[(size_t)(i0 + r) * w] = y;
#pragma unroll
        for (int t = 0; t < r; ++t) a[t] -= L[lri_at(i0 + r, i0 + t, n)] * y;
      }
  }
}

// The factor of every pair: packed triangle and reciprocals at Lw.
__global__ void __launch_bounds__(256) k_lri_chol(int batch, int n, const double* A, double* Lw, int* err) {
  extern __shared__ double L[];
  const int nl = n * (n + 1) / 2;
  for (int p = blockIdx.x; p < batch; p += gridDim.x) {
    __syncthreads();
    lri_cholesky(L, L + nl, A + (size_t)p * n * n, n, err);
    for (int e = threadIdx.x; e < nl + n; e += blockDim.x) Lw[(size_t)p * (nl + n) + e] = L[e];
  }
}

// Columns [32 part, ..) of X and dX (null: X alone) of every pair; the factor from Lw, or (Lw null) made here.
// With gradients a CTA has four warps: one makes X, the others a component of
// dX each; which is which turns with the unit, since a warp stays on one of the
// SM's four FP64 pipes.
__global__ void __launch_bounds__(4 * kLriCols) k_lri_solve(int batch, int parts, int n, int w, const double* A,
                                                            const double* Lw, const double* B, const double* dA,
                                                            const double* dB, double* X, double* dX, int* err) {
  extern __shared__ double L[];   // packed triangle, then the reciprocals of the diagonal
  const int nl = n * (n + 1) / 2, lane = threadIdx.x & 31;
  double* inv = L + nl;
  const size_t nn = (size_t)n * n, nw = (size_t)n * w;
  for (long long u = blockIdx.x; u < (long long)batch * parts; u += gridDim.x) {
    const int p = (int)(u / parts), col = kLriCols * (int)(u % parts) + lane;
    const int c = dX ? (int)((threadIdx.x >> 5) + u) & 3 : 3;   // component of dX, or 3: X
    __syncthreads();   // the previous unit's L is no longer read
    if (Lw) {
      for (int e = threadIdx.x; e < nl + n; e += blockDim.x) L[e] = Lw[(size_t)p * (nl + n) + e];
      __syncthreads();
    } else {
      lri_cholesky(L, inv, A + p * nn, n, err);
    }
    if (c == 3 && col < w) lri_column(L, inv, n, w, B + p * nw + col, nullptr, nullptr, X + p * nw + col);
    if (dX == nullptr) continue;
    __syncthreads();   // X of these columns complete
    const size_t pc = (size_t)p * 3 + c;
    if (c < 3 && col < w) lri_column(L, inv, n, w, dB + pc * nw + col, dA + pc * nn, X + p * nw + col, dX + pc * nw + col);
  }
}

}  // namespace

// (the accepted n: a full n x n matrix in shared memory)
size_t lri_fit_smem(int n) { return (size_t)n * n * sizeof(double); }

size_t lri_factor_size(int n, int w) { return w <= kLriCols ? 0 : (size_t)(n * (n + 1) / 2 + n); }

cudaError_t launch_lri_chol(int batch, int n, const double* A, double* Lw, int* err, cudaStream_t s) {
  if (batch <= 0) return cudaSuccess;
  const size_t smem = (size_t)(n * (n + 1) / 2 + n) * sizeof(double);
  cudaError_t e = allow_max_dynamic_smem((const void*)k_lri_chol);
  if (e != cudaSuccess) return e;
  ++g_launches;
  k_lri_chol<<<grid_for(batch, 1, 152 * 8), n <= 32 ? 64 : 256, smem, s>>>(batch, n, A, Lw, err);
  return cudaGetLastError();
}

cudaError_t launch_lri_solve(int batch, int n, int w, const double* A, const double* Lw, const double* B,
                             const double* dA, const double* dB, double* X, double* dX, int* err, cudaStream_t s) {
  if (batch <= 0) return cudaSuccess;
  const size_t smem = (size_t)(n * (n + 1) / 2 + n) * sizeof(double);
  cudaError_t e = allow_max_dynamic_smem((const void*)k_lri_solve);
  if (e != cudaSuccess) return e;
  const int parts = (w + kLriCols - 1) / kLriCols;
  ++g_launches;
  k_lri_solve<<<grid_for((long long)batch * parts, 1, 152 * 64), dX ? 4 * kLriCols : kLriCols, smem, s>>>(
      batch, parts, n, w, A, Lw, B, dA, dB, X, dX, err);
  return cudaGetLastError();
}

cudaError_t launch_reduce(const DevPlan& P, double* out, cudaStream_t s) {
  double* F = out + 1;
  const int total = P.nC + P.nV;
  ++g_launches;
  k_reduce_pairs<<<grid_for(total, kThreads, 152 * 4), kThreads, 0, s>>>(P, F);
  ++g_launches;
  k_finish<<<1, 32, 0, s>>>(P, out);
  return cudaGetLastError();
}

}  // namespace hfx
