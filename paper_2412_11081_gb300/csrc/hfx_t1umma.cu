// First exchange product of the HFX force/stress on the 5th-generation tensor
// cores (tcgen05 MMAs with accumulators in tensor memory), operands in two 16-bit pieces.
//
// For a kept C pair (A,F) (an "item") and its kept V pairs (A,B), the first
// product of Eq. exx_expand, factorised through Y^{BF} = sum_W C_BW D_WF:
//   U_B[beta][(f,a)] = sum_b Y^{BF}[f][beta][b] D_AB[a][b]
//   R_B = C_AF . U_B^T        (M = alpha, N = beta, K = (f,a))  -> g^V_AB = -<grad V_AB, R_B>
//   Q  += V_AB . U_B          (M = alpha, N = (f,a), K = beta)  -> E = -<C_AF, Q>, g^C_AF = -2 <grad C_AF, Q>
// (E through Q: <V_AB, C U^T> = <C, V_AB U>, so the per-B epilogue carries
// only the three gradient planes of V.)
//
// All three products run on the tensor cores.  U is made in tensor memory
// from the fp16 pieces of Y (the Y build's own store, copied as it lies) and
// D (three piece products, 22 bits), read back, split into two pieces and
// stored to shared memory as the operand of R and Q.  Both pieces of C (and
// of V) lie as alternating 8-row groups of one M = 128 operand and both
// pieces of U side by side in N, so R takes one instruction per k step for
// all four piece products and Q two; M = 64 instructions take as long as
// M = 128 ones.
//
// What bounds it: per kept triplet (n_ao 13, n_abf 50) about 2,500 cycles of
// tensor-core work (18 U, 13 R, 8 Q instructions) and as much shared-memory
// traffic, 105 KB of L2 reads.  The kernel before built U in FP32 on the CUDA
// cores, two warps per scheduler with 64 registers of D each: 12,900 cycles
// per triplet, most of them the latency of its shared-memory loads and FMA
// chains; this one takes 5,200 (64-atom Si cell 36.7 -> 13.7 ms, 8 atoms 7.0 ->
// 1.7 ms; tensor pipe active 34 %), the hand-offs between its roles being what
// is left.  (Y and V fetched into L2 some B ahead: 14.7-20 ms.)
//
// Column order (f,a) = 16 f + a with a padded to 16.  All matrices sit in
// shared memory in the no-swizzle core-matrix order (8 rows x 16 bytes); U
// serves R as a K-major B operand and Q as an MN-major one.
//
// Warp roles (16 warps of 128 registers, one CTA per SM, persistent over units; a unit is an
// item or, on small cells, a part of its B):
//   warp 0       Y producer: 128-row tiles of Y^{BF} into a ring of NS slots
//   warp 1       scheduler and producer: takes units from a global counter
//                (dynamic load balance), hands them to the other roles through
//                a ring two units ahead, and copies C (per unit), D_AB and
//                V_AB pieces (per B)
//   warp 2       tensor-memory owner; lane 0 issues the U products
//   warp 3       lane 0 issues the Q and R products
//   warps 4-11   epilogue: R -> g^V per B; Q -> E, g^C per run of B
//   warps 12-15  U tiles from tensor memory to the pieces in shared memory
// All hand-offs are mbarriers (bounded waits; a timeout sets the error flag
// and every role stops), no block barrier inside the pipeline.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "hfx_accum.cuh"
#include "hfx_device.cuh"
#include "hfx_model.cuh"

namespace hfx {
namespace {

using namespace dev;

std::atomic<long long> g_t1u_launches{0};

constexpr int kWarpY = 0, kWarpV = 1, kWarpU = 2, kWarpR = 3, kWarpE = 4, kNE = 8, kWarpS = 12, kNU = 4;
constexpr int kThreads = 32 * (kWarpS + kNU);
constexpr int kItemRing = 4;
constexpr int kItemReaders = 3 + kNE + kNU;   // Y, U and R / Q issuers, epilogue warps, U splitters
constexpr int kMaxNS = 12;                    // Y ring slots
constexpr int kYG = 32;                        // 8-row groups per Y slot: two 128-row tiles
constexpr uint32_t kYPiece = kYG * 256;        // bytes of one piece of a slot
constexpr uint32_t kYSlot = 2 * kYPiece;
constexpr int kND = 4;                        // D ring slots
constexpr int kMaxUT = 6;                     // pairs of U tiles in tensor memory

__device__ __forceinline__ bool aborted(const volatile int* f) { return *f != 0; }

// Every lane waits (bounded); the result is the same on all lanes.
__device__ __forceinline__ bool wait_all(uint32_t mbar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(mbar, parity)) != 0;
}

// Position in a ring of barriers: slot and phase.  A filled slot is waited for
// with parity ph, a free one with ph ^ 1 (true at once on the first round).
// (Counters divided by the ring's run-time size cost the single issuing
// threads more than the MMAs they issue.)
struct Ring {
  int s = 0;
  uint32_t ph = 0, n = 0;   // n: slots passed in all
  __device__ __forceinline__ void next(int size) {
    ++n;
    if (++s == size) {
      s = 0;
      ph ^= 1;
    }
  }
};

// Lets every copy issued into a ring (in order, `size` slots) land.
__device__ __forceinline__ void drain(uint32_t full, Ring r, int size) {
  for (uint32_t k = r.n < (uint32_t)size ? 0u : r.n - (uint32_t)size; k < r.n; ++k)
    mbar_wait(full + 8 * (k % size), (k / size) & 1);
}

// ------------------------------------------------------------ operand stores
// Order in which the epilogue warps load a 64-row FP32 plane (C, grad C,
// grad V): epilogue warp qd = alpha >> 4 holds row alpha in lane
// (alpha & 15) + 16 h and reads columns 32 j + 16 h + 4 t .. + 3 as one
// float4, so that for each (j, t) a warp's 32 loads are 512 consecutive
// bytes; element (alpha, col) sits at float
// ((((j * 4 + t) * 4 + qd) * 32 + lane) << 2) + (col & 3).  ep_at gives the
// (alpha, col) stored at float w (the stores are written in storage order).
__device__ __forceinline__ void ep_at(int w, int& alpha, int& col) {
  const int k = w & 3, l = (w >> 2) & 31, qd = (w >> 7) & 3, t = (w >> 9) & 3, j = w >> 11;
  alpha = qd * 16 + (l & 15);
  col = 32 * j + 16 * (l >> 4) + 4 * t + k;
}

// The same for the first product, whose accumulators hold the two pieces of
// row alpha in lanes l and l ^ 8 of quarter qd: lane l holds row
// alpha = 16 qd + 8 (l >> 4) + (l & 7) and reads columns 32 j + 16 ((l >> 3) & 1) + 4 t .. + 3.
__device__ __forceinline__ void ep_at1(int w, int& alpha, int& col) {
  const int k = w & 3, l = (w >> 2) & 31, qd = (w >> 7) & 3, t = (w >> 9) & 3, j = w >> 11;
  alpha = qd * 16 + 8 * (l >> 4) + (l & 7);
  col = 32 * j + 16 * ((l >> 3) & 1) + 4 * t + k;
}

// An item's sub-blocks: alpha al0 .. + mA, a a0 .. + nA, f f0 .. + nF of its C pair.
struct Sub {
  int al0, mA, a0, nA, f0, nF, as, fs, als;
};
template <bool SUB = true>   // SUB = false: every block is one sub-block
__device__ __forceinline__ Sub item_sub(int sub, int mA, int nA, int nF) {
  if (!SUB) return Sub{0, mA, 0, nA, 0, nF, 0, 0, 0};
  const int sf = ao_subs(nF), sa = ao_subs(nA), hf = ao_sub(nF), ha = ao_sub(nA), hm = abf_sub(mA);
  Sub r;
  r.fs = sub % sf;
  r.as = (sub / sf) % sa;
  r.als = sub / sf / sa;
  r.al0 = r.als * hm;
  r.a0 = r.as * ha;
  r.f0 = r.fs * hf;
  r.mA = min(hm, mA - r.al0);
  r.nA = min(ha, nA - r.a0);
  r.nF = min(hf, nF - r.f0);
  return r;
}

// Item kk: the pieces of its part of C_AF, per 8 rows alpha first piece 0 and
// then piece 1, (f,a) (KP) columns in core-matrix order, then C and grad C in
// FP32 as four planes of 64 x KP32 (KP rounded up to 32) in epilogue load
// order (ep_at1).  Zero padded.  Each plane ([(alpha,a)][f]) is evaluated from
// the block model into shared memory as FP32; the outputs are written in
// storage order, four elements per thread.
constexpr int kCStoreSmem = 64 * 16 * 16 * 4;   // one plane of 64 alpha, 16 a, 16 f

template <int SP>
__global__ void k_t1u_cstore(DevPlan P, T1UPlan U, const int* list, int n) {
  extern __shared__ float cs[];
  const int KP = U.KP, KP32 = t1u_kp32(KP), PL = 64 * KP32;
  for (int kk = blockIdx.x; kk < n; kk += gridDim.x) {
    const int q = list[kk] & ((1 << kItemShift) - 1);
    const int A = P.c_home[q], F = P.c_j[q];
    const int sA = P.species[A];
    const int nAt = P.n_ao[sA], nFt = P.n_ao[P.species[F]];
    const Sub sb = item_sub(list[kk] >> kItemShift, P.n_abf[sA], nAt, nFt);
    const int mA = sb.mA, nA = sb.nA, nF = sb.nF;
    const int ncq = mA * nA * nF, g8 = (mA + 7) >> 3;
    uint16_t* out = U.Cu + (long long)kk * U.cu_blk;
    float* pl = reinterpret_cast<float*>(out + (long long)NP * U.GA * 8 * KP);
    float scf[8];   // C = G f + G' fa, grad C = G g + G' ga (block model, FP32 as k_cpieces)
#pragma unroll
    for (int k = 0; k < 8; ++k) scf[k] = (float)P.c_sc[8 * (long long)q + k];
    const long long go = P.G_off[sA * P.S + P.species[F]];
    const float sc = pscale<SP>(P.sc.c[A] - P.sc.d[F]);
    for (int c = 0; c < 4; ++c) {
      __syncthreads();
      for (int e = threadIdx.x; e < ncq; e += blockDim.x) {
        const int r = e / nF, f = e - r * nF, al = r / nA, a = r - al * nA;
        cs[e] = model::c_value_f(P, scf, go, ((sb.al0 + al) * nAt + sb.a0 + a) * nFt + sb.f0 + f, c);
      }
      __syncthreads();
      auto val = [&](int al, int col) -> float {
        const int f = col >> 4, a = col & 15;
        return (al < mA && col < KP && f < nF && a < nA) ? cs[(al * nA + a) * nF + f] : 0.f;
      };
      if (c == 0) {
        // pieces: element t of an 8-row group -> (alpha, col), four consecutive columns per thread
        for (int t4 = threadIdx.x; t4 < g8 * 2 * KP; t4 += blockDim.x) {
          const int g = t4 / (2 * KP), t = 4 * (t4 - g * 2 * KP);
          const int al = g * 8 + ((t >> 3) & 7), col = (t >> 6) * 8 + (t & 7);
          const float x[4] = {val(al, col) * sc, val(al, col + 1) * sc,
                              val(al, col + 2) * sc, val(al, col + 3) * sc};
          uint2 pc[NP];
          split4<SP>(x, pc);
#pragma unroll
          for (int pp = 0; pp < NP; ++pp) *reinterpret_cast<uint2*>(out + (long long)(g * NP + pp) * 8 * KP + t) = pc[pp];
        }
      }
      for (int w4 = threadIdx.x; w4 < PL / 4; w4 += blockDim.x) {   // FP32 plane c, storage order
        int al, col;
        ep_at1(4 * w4, al, col);
        *reinterpret_cast<float4*>(pl + (long long)c * PL + 4 * w4) =
            make_float4(val(al, col), val(al, col + 1), val(al, col + 2), val(al, col + 3));
      }
    }
  }
}

// Every needed V pair p = list[k], in one pass: V and grad V evaluated once
// from the block model into shared memory (FP32), then
//   the warp-level second product's store X.Vm at vm_off[p] (unless X.Vz is
//   set): NP planes [alpha][rup16(n_abf(B))] and V, grad V in FP32
//   [4][n_abf(A) n_abf(B)];
//   for the pairs of the first product (any bit of v_mask), the tcgen05
//   store U.Vu at t1_idx[p]: the pieces of V, per 8 rows alpha piece 0 then
//   piece 1, beta 64 in core-matrix order, and grad V in three planes in
//   epilogue load order (ep_at1);
//   for the pairs of the second product (v_t2), with X.Vz set, the store of
//   k_t2_umma at t2_slot[p]: the pieces as [piece][alpha 64][beta 64] and V,
//   grad V in four planes (ep_at).
// Outputs are written in storage order, four elements per thread.
// Rows alpha are taken 64 (abf_sub) at a time; the second product's stores
// have no more than that.
size_t vstore_smem(int max_abf) { return (size_t)4 * 64 * max_abf * sizeof(float); }

template <int SP>
__global__ void k_vstores(DevPlan P, MixPlan X, T1UPlan U, const int* list, int n) {
  extern __shared__ float vsm[];   // [4][mA * mB]: V, grad V of the rows in hand
  for (int k = blockIdx.x; k < n; k += gridDim.x) {
    const int p = list[k];
    const int sA = P.species[P.v_home[p]], sB = P.species[P.v_j[p]];
    const int mAt = P.n_abf[sA], mB = P.n_abf[sB], MB = rup16(mB), hm = abf_sub(mAt);
    double h, g[3];
    model::v_pair(P, p, h, g);   // V = M h, grad V = M g (block model), in FP32
    const float hf = (float)h, g0 = (float)g[0], g1 = (float)g[1], g2 = (float)g[2];
    const float sv = pscale<SP>(v_exp(P, P.v_home[p], P.v_j[p]));
    bool t1 = false;
#pragma unroll
    for (int w = 0; w < kMaskWords; ++w) t1 = t1 || P.v_mask[(long long)p * kMaskWords + w] != 0u;
    for (int als = 0, al0 = 0; al0 < mAt; ++als, al0 += hm) {
    const int mA = min(hm, mAt - al0), nv = mA * mB;
    const float* M = P.Mf + P.M_off[sA * P.S + sB] + al0 * mB;
    __syncthreads();
    for (int e = threadIdx.x; e < nv; e += blockDim.x) {
      const float m = M[e];
      vsm[e] = m * hf;
      vsm[nv + e] = m * g0;
      vsm[2 * nv + e] = m * g1;
      vsm[3 * nv + e] = m * g2;
    }
    __syncthreads();
    // second-product store of the warp-level R2 / Z kernel, where that runs
    if (X.Vm) {
      uint16_t* out = X.Vm + X.vm_off[p];
      for (int e4 = threadIdx.x; e4 < mA * MB / 4; e4 += blockDim.x) {
        const int e = 4 * e4, al = e / MB, be = e - al * MB;
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = be + j < mB ? vsm[al * mB + be + j] * sv : 0.f;
        uint2 pc[NP];
        split4<SP>(x, pc);
#pragma unroll
        for (int pp = 0; pp < NP; ++pp) *reinterpret_cast<uint2*>(out + (long long)pp * mA * MB + e) = pc[pp];
      }
      float* v32 = reinterpret_cast<float*>(out + (long long)NP * mA * MB);
      for (int e = threadIdx.x; e < 4 * nv; e += blockDim.x) v32[e] = vsm[e];
    }
    // the tcgen05 stores: the first product's (U.Vu, per first-product pair and
    // alpha sub: pieces and the three grad V planes) and the second product's
    // (X.Vz, per second-product pair: pieces and the four planes V, grad V)
    for (int st = 0; st < 2; ++st) {
      uint16_t* vu = nullptr;
      if (st == 0 && U.Vu && t1) vu = U.Vu + (U.t1_idx[p] * U.NAL + als) * U.vu_blk;
      if (st == 1 && X.Vz && P.v_t2[p]) vu = X.Vz + X.t2_slot[p] * X.vz_blk;
      if (!vu) continue;
      const int VK = st == 0 ? U.VK : 64, G = st == 0 ? (mA + 7) >> 3 : 8, VC = (VK + 31) & ~31;
      // (the quotients of these small numbers are exact in FP32)
      const float iK = 1.f / (float)(2 * VK), iP = 1.f / (float)(16 * VC);
      for (int t4 = threadIdx.x; t4 < G * 2 * VK; t4 += blockDim.x) {   // core-matrix order, 4 columns per thread
        const int g8 = (int)(((float)t4 + 0.5f) * iK), t = 4 * (t4 - g8 * 2 * VK);
        const int al = g8 * 8 + ((t >> 3) & 7), be = ((t >> 6) << 3) + (t & 7);
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = (al < mA && be + j < mB) ? vsm[al * mB + be + j] * sv : 0.f;
        uint2 pc[NP];
        split4<SP>(x, pc);
#pragma unroll
        for (int pp = 0; pp < NP; ++pp)
          *reinterpret_cast<uint2*>(vu + (st == 0 ? (g8 * NP + pp) * 8 * VK + t : pp * 4096 + g8 * 512 + t)) = pc[pp];
      }
      float* pl = reinterpret_cast<float*>(vu + (st == 0 ? NP * 8 * VK * U.GA : NP * 4096));
      const int c0 = st == 0 ? 1 : 0;   // first plane: grad V (first product) or V (second)
      const int PL4 = 16 * VC;          // float4 per plane
      for (int w4 = threadIdx.x; w4 < (4 - c0) * PL4; w4 += blockDim.x) {   // epilogue load order
        const int pl4 = (int)(((float)w4 + 0.5f) * iP), c = c0 + pl4, w = 4 * (w4 - pl4 * PL4);
        int al, be;
        if (st == 0) ep_at1(w, al, be);
        else ep_at(w, al, be);
        float4 o;
        o.x = (al < mA && be < mB) ? vsm[c * nv + al * mB + be] : 0.f;
        o.y = (al < mA && be + 1 < mB) ? vsm[c * nv + al * mB + be + 1] : 0.f;
        o.z = (al < mA && be + 2 < mB) ? vsm[c * nv + al * mB + be + 2] : 0.f;
        o.w = (al < mA && be + 3 < mB) ? vsm[c * nv + al * mB + be + 3] : 0.f;
        *reinterpret_cast<float4*>(pl + 4 * w4) = o;
      }
    }
    }
  }
}

// ------------------------------------------------- longest-first item order
// Items run on a dynamic queue; handing out the ones with the most kept B
// first keeps the last items short, so the SMs finish together.  Counting
// sort on the bucket (kLptBuckets - 1 - min(qcnt, kLptBuckets - 1)); the
// order of equal keys is not fixed (it does not change any item's result).
// With asc = 1 the same sort orders the items by key[q] ascending (the
// order by F: items of one F, which share many Y^{BF} blocks, run together).
__device__ __forceinline__ int lpt_bucket(const int* key, int q, int asc) {
  const int k = min(key[q & ((1 << kItemShift) - 1)], kLptBuckets - 1);   // (a list entry: C pair and sub)
  return asc ? k : kLptBuckets - 1 - k;
}

__global__ void k_lpt_hist(const int* key, int asc, const int* list, const long long* n_dev, int* hist) {
  const int n = (int)*n_dev;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    atomicAdd(&hist[lpt_bucket(key, list[i], asc)], 1);
}

// Exclusive scan of the histogram, one block of 1024 threads.
__global__ void __launch_bounds__(1024) k_lpt_scan(int* hist) {
  constexpr int kPer = kLptBuckets / 1024;
  __shared__ int part[1024];
  int v[kPer], t = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    v[j] = hist[threadIdx.x * kPer + j];
    t += v[j];
  }
  part[threadIdx.x] = t;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int add = threadIdx.x >= (unsigned)o ? part[threadIdx.x - o] : 0;
    __syncthreads();
    part[threadIdx.x] += add;
    __syncthreads();
  }
  int run = part[threadIdx.x] - t;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    hist[threadIdx.x * kPer + j] = run;
    run += v[j];
  }
}

__global__ void k_lpt_scatter(const int* key, int asc, const int* list, const long long* n_dev, int* hist, int* out) {
  const int n = (int)*n_dev;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int q = list[i];
    out[atomicAdd(&hist[lpt_bucket(key, q, asc)], 1)] = q;
  }
}

// ------------------------------------------------------------------- kernel
// Sizes of one launch, shared by the kernel and the host: KP columns
// (f, a) = 16 f + a, GA and GB row groups of 8 alpha and 8 beta, VK columns
// beta of V, KB sub-blocks of b, UB buffers of U, NS slots of the Y ring.
__host__ __device__ inline uint32_t t1_ubytes(int KP, int G) { return (uint32_t)G * 2u * 16u * KP; }   // C, or one buffer of U
__host__ __device__ inline uint32_t t1_vbytes(int GA, int VK) { return (uint32_t)GA * 2u * 16u * VK; }
__host__ __device__ inline uint32_t t1_base(int KP, int GA, int GB, int KB, int UB) {
  return t1_ubytes(KP, GA) + UB * t1_ubytes(KP, GB) + 2 * t1_vbytes(GA, (8 * GB + 15) & ~15) + kND * KB * 1024u;
}
// Tensor-memory columns: Q at 0, R from the next multiple of 32, then the U tiles in pairs of 32 columns.
__host__ __device__ inline int t1_rcol(int KP) { return (KP + 31) & ~31; }
__host__ __device__ inline int t1_utiles(int KP, int G) {
  const int n = (512 - t1_rcol(KP) - 16 * G) / 32;
  return n < kMaxUT ? n : kMaxUT;
}

// SUB = false: plans with n_ao <= 16 and n_abf <= 64, whose blocks are one
// sub-block each.  With the sub-blocks' index arithmetic and loops in their
// single issuing threads they run at 18.9 instead of 13.7 ms (64-atom Si cell).
template <int SP, bool SUB>
__global__ void __launch_bounds__(kThreads, 1)
    k_t1_umma(DevPlan P, MixPlan X, T1UPlan U, const int* qlist, int n_list, int* work, int* err) {
  const int KP = U.KP, KP32 = t1u_kp32(KP), GB = U.GB, VK = U.VK, NS = U.NS, UB = U.UB, SEG = U.seg, nsplit = U.nsplit;
  const int NT = t1_utiles(KP, GB), n_units = n_list * nsplit;
  const uint32_t rowg = 16u * KP;                    // bytes of one 8-row group of a C or U piece
  const uint32_t vrowg = 16u * VK;                   // and of V
  const uint32_t CB = t1_ubytes(KP, U.GA), UBY = t1_ubytes(KP, GB), VB = t1_vbytes(U.GA, VK), DB = SUB ? X.KB * 1024u : 1024u;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t b_yf[kMaxNS], b_ye[kMaxNS], b_cf, b_ce, b_vf[2], b_ve[2], b_df[kND], b_de[kND],
      b_tf[kMaxUT], b_te[kMaxUT], b_uf[2], b_ue[2], b_rf, b_re, b_qf, b_qe, b_if[kItemRing], b_ie[kItemRing], b_done[2];
  __shared__ int4 s_item[kItemRing];   // a unit: item kk (-1: no more), its list entry, its B [lo, hi) of the list at X.qoff
  __shared__ uint32_t tmem_base;
  __shared__ int s_abort;
  volatile int* abort_flag = &s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto sa = [](const void* p) { return (uint32_t)__cvta_generic_to_shared(p); };
  const uint32_t Cs = sa(smem_raw), Us = Cs + CB, Vs = Us + UB * UBY, Ds = Vs + 2 * VB, Ys = Ds + kND * DB;
  const uint32_t yf = sa(b_yf), ye = sa(b_ye), cf = sa(&b_cf), ce = sa(&b_ce), vf = sa(b_vf), ve = sa(b_ve),
                 df = sa(b_df), de = sa(b_de), tf = sa(b_tf), te = sa(b_te), uf = sa(b_uf), ue = sa(b_ue),
                 rf = sa(&b_rf), re = sa(&b_re), qf = sa(&b_qf), qe = sa(&b_qe), itf = sa(b_if), ite = sa(b_ie),
                 mdone = sa(b_done);
  // Operand rows and columns past a block's own are read (and multiplied by
  // zeros of the other operand, or their results dropped): everything in the
  // buffers has to be finite from the start.
  for (uint32_t o = tid * 16u; o < (Ys - Cs) + (uint32_t)NS * kYSlot; o += kThreads * 16u)
    *reinterpret_cast<uint4*>(smem_raw + o) = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) {
    s_abort = 0;
    for (int s = 0; s < NS; ++s) {
      mbar_init(yf + 8 * s, 1);
      mbar_init(ye + 8 * s, 1);
    }
    for (int s = 0; s < kND; ++s) {
      mbar_init(df + 8 * s, 1);
      mbar_init(de + 8 * s, 1);
    }
    for (int s = 0; s < NT; ++s) {
      mbar_init(tf + 8 * s, 1);
      mbar_init(te + 8 * s, kNU);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(vf + 8 * s, 1);
      mbar_init(ve + 8 * s, 1);
      mbar_init(uf + 8 * s, kNU);
      mbar_init(ue + 8 * s, 1);
    }
    mbar_init(cf, 1);
    mbar_init(ce, 1);
    mbar_init(rf, 1);
    mbar_init(re, kNE);
    mbar_init(qf, 1);
    mbar_init(qe, kNE);
    for (int s = 0; s < kItemRing; ++s) {
      mbar_init(itf + 8 * s, 1);
      mbar_init(ite + 8 * s, kItemReaders);
    }
    for (int s = 0; s < 2; ++s) mbar_init(mdone + 8 * s, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
  }
  if (warp == kWarpU) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(sa(&tmem_base)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t T = tmem_base, TR = T + t1_rcol(KP), TU = TR + 16u * GB;
  // Next unit of the ring for a role (one reader per warp; lane 0 releases
  // the slot); kk < 0 marks the end.  Every lane of the warp calls it.
  struct Unit {
    int kk, code, lo, hi;
    __device__ int q() const { return SUB ? code & ((1 << kItemShift) - 1) : code; }
    __device__ int sub() const { return code >> kItemShift; }
  };
  auto next_unit = [&](Ring& r) -> Unit {
    Unit u{-1, 0, 0, 0};
    if (wait_all(itf + 8 * r.s, r.ph)) {
      const volatile int* v = reinterpret_cast<const volatile int*>(&s_item[r.s]);
      u = Unit{v[0], v[1], v[2], v[3]};
    } else {
      *abort_flag = 1;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(ite + 8 * r.s);
    r.next(kItemRing);
    return u;
  };

  if (warp == kWarpY) {
    // ---------------------------------------------------------- Y producer
    // Y^{BF} as [piece][(g, f)][8 beta x 16 b]: up to 32 row groups (g, f) per
    // slot, the two pieces copied by lanes 0 and 1.
    Ring ik, y;
    for (Unit it = next_unit(ik); it.kk >= 0 && !aborted(abort_flag); it = next_unit(ik)) {
      const int q = it.q(), F = P.c_j[q], sA = P.species[P.c_home[q]];
      const int nFt = P.n_ao[P.species[F]];
      const Sub sb = item_sub<SUB>(it.sub(), P.n_abf[sA], P.n_ao[sA], nFt);
      const int* Rf = P.c_R + 3 * q;
      const long long b0 = X.qoff[q];
      for (int i0 = it.lo; i0 < it.hi && !aborted(abort_flag); i0 += 32) {
        long long yo = 0;
        int g8 = 0, nbs = 0;   // 8-row groups of beta, subs of b
        if (i0 + lane < it.hi) {
          const int p = X.blist[b0 + i0 + lane];
          const int b = P.v_j[p];
          const int* Rb = P.v_R + 3 * p;
          const int yc = ylut_get(P, b, F, Rf[0] - Rb[0], Rf[1] - Rb[1], Rf[2] - Rb[2]);
          yo = yc < 0 ? -1 : P.y_off[yc];
          g8 = (P.n_abf[P.species[b]] + 7) >> 3;
          nbs = SUB ? ao_subs(P.n_ao[P.species[b]]) : 1;
        }
        const int nb = min(32, it.hi - i0);
        for (int j = 0; j < nb; ++j) {
          const long long yoj = __shfl_sync(0xffffffffu, yo, j);
          const int g8j = __shfl_sync(0xffffffffu, g8, j), nbj = SUB ? __shfl_sync(0xffffffffu, nbs, j) : 1;
          const int ngj = g8j * sb.nF;
          const long long xs1 = (long long)g8j * nFt * 128;   // a sub of b; the piece holds nbj of them
          if (yoj < 0) *abort_flag = 1;   // a kept triplet always has its Y block
          for (int r0 = 0; r0 < ngj; r0 += kYG) {
            const uint32_t bytes = 256u * (uint32_t)min(kYG, ngj - r0);
            for (int bs = 0; bs < nbj; ++bs, y.next(NS)) {
              const int s = y.s;
              bool ok = true;
              if (lane == 0) {
                ok = !aborted(abort_flag) && mbar_wait(ye + 8 * s, y.ph ^ 1);
                if (ok) mbar_expect_tx(yf + 8 * s, 2 * bytes);
                else *abort_flag = 1;
              }
              ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
              if (!ok) break;
              if (lane < 2)
                bulk_g2s(Ys + s * kYSlot + lane * kYPiece,
                         U.Yh + yoj + (lane * nbj + bs) * xs1 + (long long)g8j * sb.f0 * 128 + r0 * 128, bytes,
                         yf + 8 * s);
            }
            if (SUB && __shfl_sync(0xffffffffu, (int)aborted(abort_flag), 0)) break;
          }
          if (__shfl_sync(0xffffffffu, (int)aborted(abort_flag), 0)) break;
        }
      }
    }
    __syncwarp();
    if (lane == 0) drain(yf, y, NS);   // copies in flight land before the CTA leaves
  } else if (warp == kWarpV) {
    // -------------------------------------- scheduler, C, D and V producer
    // Lane 0 publishes units two ahead of this warp's own position (a slot
    // is reused once every reader has taken its unit).
    Ring pub;
    bool pub_done = false;
    auto publish = [&]() {
      volatile int* v = reinterpret_cast<volatile int*>(&s_item[pub.s]);
      if (!mbar_wait(ite + 8 * pub.s, pub.ph ^ 1)) {   // every reader has taken the slot's last unit
        *abort_flag = 1;
        pub_done = true;
        return;
      }
      v[0] = -1;
      pub_done = true;
      while (!aborted(abort_flag)) {   // units without a B (fewer B than parts) are passed over
        const int u = atomicAdd(work, 1);
        if (u >= n_units) break;
        const int kk = u / nsplit, part = u - kk * nsplit, code = qlist[kk], n = X.qcnt[code & ((1 << kItemShift) - 1)];
        const int lo = n * part / nsplit, hi = n * (part + 1) / nsplit;
        if (hi <= lo) continue;
        v[1] = code;
        v[2] = lo;
        v[3] = hi;
        v[0] = kk;
        pub_done = false;
        break;
      }
      mbar_arrive(itf + 8 * pub.s);
      pub.next(kItemRing);
    };
    if (lane == 0) {
      publish();
      if (!pub_done) publish();
    }
    __syncwarp();
    uint32_t it_n = 0, ca = 0;
    Ring own, v, d;
    auto own_unit = [&]() -> Unit {
      Unit u{-1, 0, 0, 0};
      if (lane == 0 && own.n < pub.n) {
        const volatile int* w = reinterpret_cast<const volatile int*>(&s_item[own.s]);
        u = Unit{w[0], w[1], w[2], w[3]};
      }
      own.next(kItemRing);
      u.kk = __shfl_sync(0xffffffffu, u.kk, 0);
      u.code = __shfl_sync(0xffffffffu, u.code, 0);
      u.lo = __shfl_sync(0xffffffffu, u.lo, 0);
      u.hi = __shfl_sync(0xffffffffu, u.hi, 0);
      return u;
    };
    for (Unit it = own_unit(); it.kk >= 0 && !aborted(abort_flag); it = own_unit(), ++it_n) {
      const int q = it.q(), sA = P.species[P.c_home[q]];
      const Sub sb = item_sub<SUB>(it.sub(), P.n_abf[sA], P.n_ao[sA], P.n_ao[P.species[P.c_j[q]]]);
      const long long b0 = X.qoff[q];
      const uint32_t gA = (uint32_t)(sb.mA + 7) >> 3;
      if (lane == 0) {
        if (!pub_done) publish();
        if (it_n >= 1 && !mbar_wait(ce, (it_n - 1) & 1)) *abort_flag = 1;
        if (!aborted(abort_flag)) {
          mbar_expect_tx(cf, gA * 2u * rowg);
          bulk_g2s(Cs, U.Cu + (long long)it.kk * U.cu_blk, gA * 2u * rowg, cf);
          ++ca;
        }
      }
      __syncwarp();
      for (int i0 = it.lo; i0 < it.hi && !aborted(abort_flag); i0 += 32) {
        long long vo = 0, dofs = 0;
        int nbs = 0;
        if (i0 + lane < it.hi) {
          const int p = X.blist[b0 + i0 + lane];
          vo = (SUB ? U.t1_idx[p] * U.NAL + sb.als : U.t1_idx[p]) * U.vu_blk;
          const int di = P.v_didx[p];
          nbs = SUB ? ao_subs(P.n_ao[P.species[P.v_j[p]]]) : 1;
          dofs = di >= 0 ? X.dsp_off[di] + sb.as * nbs * 512 : -1;   // a kept triplet always has its D block
        }
        const int nb = min(32, it.hi - i0);
        for (int j = 0; j < nb; ++j) {
          const long long voj = __shfl_sync(0xffffffffu, vo, j);
          const long long doj = __shfl_sync(0xffffffffu, dofs, j);
          const uint32_t dbytes = SUB ? 1024u * (uint32_t)__shfl_sync(0xffffffffu, nbs, j) : 1024u;   // the row a of sub-blocks
          if (lane == 0 && doj < 0) *abort_flag = 1;
          if (lane == 0 && !aborted(abort_flag)) {
            bool ok = mbar_wait(de + 8 * d.s, d.ph ^ 1);
            if (ok) {
              mbar_expect_tx(df + 8 * d.s, dbytes);
              bulk_g2s(Ds + d.s * DB, U.Dh + doj, dbytes, df + 8 * d.s);
              d.next(kND);
            }
            ok = ok && mbar_wait(ve + 8 * v.s, v.ph ^ 1);
            if (ok) {
              mbar_expect_tx(vf + 8 * v.s, gA * 2u * vrowg);
              bulk_g2s(Vs + v.s * VB, U.Vu + voj, gA * 2u * vrowg, vf + 8 * v.s);
              v.next(2);
            } else {
              *abort_flag = 1;
            }
          }
          __syncwarp();
        }
      }
    }
    if (lane == 0) {
      if (ca) mbar_wait(cf, (ca - 1) & 1);
      drain(vf, v, 2);
      drain(df, d, kND);
    }
  } else if (warp == kWarpU) {
    // ------------------------------------------------------------ U issuer
    // Tile of U: 128 rows (g, f, beta of the group) x 16 columns a,
    // U = Y0 D1^T + Y1 D0^T + Y0 D0^T (K = 16 b), always fp16 pieces.  The
    // products of a slot's two tiles alternate: an instruction waits for the
    // one before on the same accumulator (72 cycles each in one chain).
    const uint32_t idU = idesc_split<kSplitHalf>(128, 16, 0);
    Ring ik, y, t, d;
    bool ok = true;
    for (Unit it = next_unit(ik); it.kk >= 0; it = next_unit(ik)) {
      const int q = it.q(), sA = P.species[P.c_home[q]];
      const int nF = item_sub<SUB>(it.sub(), P.n_abf[sA], P.n_ao[sA], P.n_ao[P.species[P.c_j[q]]]).nF;
      const long long b0 = X.qoff[q];
      for (int i0 = it.lo; i0 < it.hi; i0 += 32) {
        int ng = 0, nbs = 0;
        if (i0 + lane < it.hi) {
          const int sB = P.species[P.v_j[X.blist[b0 + i0 + lane]]];
          ng = ((P.n_abf[sB] + 7) >> 3) * nF;
          nbs = SUB ? ao_subs(P.n_ao[sB]) : 1;
        }
        const int nb = min(32, it.hi - i0);
        for (int j = 0; j < nb; ++j) {
          const int ngj = __shfl_sync(0xffffffffu, ng, j), nbj = SUB ? __shfl_sync(0xffffffffu, nbs, j) : 1;
          if (lane == 0 && ok) {
            ok = !aborted(abort_flag) && mbar_wait(df + 8 * d.s, d.ph);
            for (int r0 = 0; r0 < ngj && ok; r0 += kYG) {
              const uint32_t tu = TU + 32u * t.s;
              const bool two = r0 + 16 < ngj;
              ok = mbar_wait(te + 8 * t.s, t.ph ^ 1);
              for (int bs = 0; bs < nbj && ok; ++bs) {
                ok = mbar_wait(yf + 8 * y.s, y.ph);
                if (!ok) break;
                tc_fence_after();
                const uint64_t dD = sdesc2(Ds + d.s * DB + bs * 1024u, 128, 512);   // (pieces alternate by 8 rows)
                const uint64_t dY = sdesc2(Ys + y.s * kYSlot, 128, 256);
                umma_f16(tu, dY, dD + 16, idU, bs > 0);                        // Y0 D1 (the second piece: 256 bytes on)
                if (two) umma_f16(tu + 16, dY + 256, dD + 16, idU, bs > 0);    // (the second tile: 4096 bytes on)
                umma_f16(tu, dY + (kYPiece >> 4), dD, idU, 1u);                // Y1 D0
                if (two) umma_f16(tu + 16, dY + 256 + (kYPiece >> 4), dD, idU, 1u);
                umma_f16(tu, dY, dD, idU, 1u);                                 // Y0 D0
                if (two) umma_f16(tu + 16, dY + 256, dD, idU, 1u);
                if (bs == nbj - 1) umma_commit(tf + 8 * t.s);
                umma_commit(ye + 8 * y.s);
                y.next(NS);
              }
              if (ok) t.next(NT);
            }
            if (ok) umma_commit(de + 8 * d.s);
            else *abort_flag = 1;
            d.next(kND);
          }
          __syncwarp();
        }
      }
    }
    if (lane == 0) {
      umma_commit(mdone);
      mbar_wait(mdone, 0);
    }
  } else if (warp == kWarpR) {
    // ------------------------------------------------------- Q and R issuer
    // Q += V_AB . U_B, K = beta in steps of 16: A = both pieces of V (row
    // groups (g, piece), M = 128), N = 16 n_ao(F) columns (f,a) of one piece
    // of U, read MN-major.
    // R_B = C_AF . U_B^T, K = (f,a), one f per k step: A = both pieces of C
    // (row groups (g, piece), M = 128), B = both pieces of U (N = 16 G), so
    // one instruction per k step makes all four piece products, and R is the
    // sum over the two row groups of an alpha and the two columns of a beta.
    // Q goes first: meanwhile the epilogue empties the accumulator of the R before.
    const uint32_t idR = idesc_split<SP>(128, 16 * GB, 0);
    const uint64_t dC = sdesc2(Cs, 128, rowg);
    const uint64_t kbB = (uint64_t)(2 * rowg) >> 4, pB = (uint64_t)(UBY >> 1) >> 4;
    uint32_t rp = 1, qp = 1, it_n = 0;   // phases of the free accumulators
    Ring ik, ub, v;
    bool ok = true;
    for (Unit it = next_unit(ik); it.kk >= 0; it = next_unit(ik), ++it_n) {
      const int q = it.q(), sA = P.species[P.c_home[q]];
      const int nF = item_sub<SUB>(it.sub(), P.n_abf[sA], P.n_ao[sA], P.n_ao[P.species[P.c_j[q]]]).nF;
      const uint32_t idQ = idesc_split<SP>(128, 16 * nF, 1);
      const long long b0 = X.qoff[q];
      int run = 0;
      for (int i0 = it.lo; i0 < it.hi; i0 += 32) {
        int nk_l = 0;
        if (i0 + lane < it.hi) nk_l = (P.n_abf[P.species[P.v_j[X.blist[b0 + i0 + lane]]]] + 15) >> 4;
        const int nb = min(32, it.hi - i0);
        for (int j = 0; j < nb; ++j) {
          const int nk = __shfl_sync(0xffffffffu, nk_l, j);
          if (lane == 0 && ok) {
            const bool first = run == 0, last = ++run == SEG || i0 + j == it.hi - 1;
            if (last) run = 0;
            ok = !aborted(abort_flag) && mbar_wait(uf + 8 * ub.s, ub.ph) && mbar_wait(vf + 8 * v.s, v.ph) &&
                 (!first || mbar_wait(qe, qp));
            if (ok) {
              tc_fence_after();
              const uint64_t dV = sdesc2(Vs + v.s * VB, 128, vrowg), dU = sdesc2(Us + ub.s * UBY, rowg, 128);
              for (int kb = 0; kb < nk; ++kb) {
                umma_f16(T, dV + 16u * kb, dU + pB + kbB * kb, idQ, (first && kb == 0) ? 0u : 1u);
                umma_f16(T, dV + 16u * kb, dU + kbB * kb, idQ, 1u);
              }
              umma_commit(ve + 8 * v.s);
              v.next(2);
              if (last) {
                umma_commit(qf);
                qp ^= 1;
              }
              ok = (i0 + j > it.lo || mbar_wait(cf, it_n & 1)) && mbar_wait(re, rp);
            }
            if (ok) {
              tc_fence_after();
              const uint64_t dU = sdesc2(Us + ub.s * UBY, 128, rowg);
              for (int f = 0; f < nF; ++f) umma_f16(TR, dC + 16u * f, dU + 16u * f, idR, f > 0 ? 1u : 0u);
              umma_commit(rf);
              umma_commit(ue + 8 * ub.s);
              ub.next(UB);
              rp ^= 1;
              if (i0 + j == it.hi - 1) umma_commit(ce);
            } else {
              *abort_flag = 1;
            }
          }
          __syncwarp();
        }
      }
    }
    if (lane == 0) {
      umma_commit(mdone + 8);
      mbar_wait(mdone + 8, 0);
    }
  } else if (warp >= kWarpE && warp < kWarpE + kNE) {
    // --------------------------------------------------------------- epilogue
    // Eight warps: lane quarter qd (rows alpha 16 qd .. + 15, both pieces) and
    // half h of the columns.  Lane l holds piece (l >> 3) & 1 of row alpha; the
    // lanes l and l ^ 8 add their rows, each keeping 16 of the 32 columns.
    const int qd = warp & 3, h = (warp - kWarpE) >> 2, ew = warp - kWarpE;
    const int alpha = qd * 16 + 8 * (lane >> 4) + (lane & 7), pc = (lane >> 3) & 1;
    const uint32_t tl = (uint32_t)(qd * 32) << 16;
    // x[t] = this lane pair's sum over columns c0 + 16 pc + t (and, with c1, over
    // c1 + 16 pc + t): each lane sends the half that the other keeps
    auto pair_read = [&](uint32_t c0, uint32_t c1, bool two, float (&x)[16]) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t a0[8], a1[8], b0[8], b1[8];
        tmem_ld8(c0 + 8u * q, a0);
        tmem_ld8(c0 + 16u + 8u * q, a1);
        if (two) {
          tmem_ld8(c1 + 8u * q, b0);
          tmem_ld8(c1 + 16u + 8u * q, b1);
        }
        tmem_wait_ld();
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const float lo = two ? __uint_as_float(a0[t]) + __uint_as_float(b0[t]) : __uint_as_float(a0[t]);
          const float hi = two ? __uint_as_float(a1[t]) + __uint_as_float(b1[t]) : __uint_as_float(a1[t]);
          x[8 * q + t] = (pc ? hi : lo) + __shfl_xor_sync(0xffffffffu, pc ? lo : hi, 8);
        }
      }
    };
    const int VP4 = 16 * ((VK + 31) & ~31);   // float4 per plane of grad V
    uint32_t rb = 0, seg = 0;
    Ring ik;
    unsigned long long fl = 0;
    bool ok = true;
    for (Unit it = next_unit(ik); it.kk >= 0 && ok; it = next_unit(ik)) {
      const int q = it.q(), sA = P.species[P.c_home[q]];
      const Sub sb = item_sub<SUB>(it.sub(), P.n_abf[sA], P.n_ao[sA], P.n_ao[P.species[P.c_j[q]]]);
      const int nA = sb.nA, mA = sb.mA, nF = sb.nF;
      const int hA = P.c_home[q], eR = P.sc.c[hA] + kUExp + P.sc.d[hA];   // (R: and d[B] + y[B])
      const long long b0 = X.qoff[q];
      const float* Cf = reinterpret_cast<const float*>(U.Cu + (long long)it.kk * U.cu_blk + (CB >> 1));
      int run = 0;
      for (int i0 = it.lo; i0 < it.hi && ok; i0 += 32) {
        int p_l = 0, mB_l = 0, nB_l = 0, yB_l = 0;
        long long vo_l = 0;
        if (i0 + lane < it.hi) {
          p_l = X.blist[b0 + i0 + lane];
          const int b = P.v_j[p_l], s_b = P.species[b];
          if (SP == kSplitHalf) yB_l = P.sc.d[b] + P.sc.y[b];
          mB_l = P.n_abf[s_b];
          nB_l = P.n_ao[s_b];
          vo_l = (SUB ? U.t1_idx[p_l] * U.NAL + sb.als : U.t1_idx[p_l]) * U.vu_blk;
        }
        const int nb = min(32, it.hi - i0);
        for (int j = 0; j < nb && ok; ++j) {
          ok = __all_sync(0xffffffffu, !aborted(abort_flag)) != 0;
          if (!ok) break;
          const int mB = __shfl_sync(0xffffffffu, mB_l, j);
          const long long vo = __shfl_sync(0xffffffffu, vo_l, j);
          const bool last = ++run == SEG || i0 + j == it.hi - 1;
          // ---- R_B -> g^V_AB, 32 columns beta at a time (two halves of the
          // warps; n_abf <= 64: one turn).  The grad V values of this lane's
          // columns cb .. cb + 15 are fetched before the wait: they do not
          // depend on R, and their latency is the longest of the epilogue.
          const float4* dV4 = reinterpret_cast<const float4*>(U.Vu + vo + (VB >> 1)) + qd * 32 + lane;
          float4 w[3][4];
          float x[16], gv[3] = {0.f, 0.f, 0.f};
          bool act = alpha < mA && 32 * h + 16 * pc < mB;
          if (act) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
              for (int t4 = 0; t4 < 4; ++t4) w[c][t4] = dV4[c * VP4 + h * 512 + t4 * 128];
          }
          ok = wait_all(rf, rb & 1);
          tc_fence_after();
          if (qd * 16 < mA && ok) {
#pragma unroll 1
            for (int jb = h; 32 * jb < mB; jb += 2) {
              const int cb = 32 * jb + 16 * pc;
              if (SUB && jb > h) {
                act = alpha < mA && cb < mB;
                if (act) {
#pragma unroll
                  for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int t4 = 0; t4 < 4; ++t4) w[c][t4] = dV4[c * VP4 + jb * 512 + t4 * 128];
                }
              }
              pair_read(TR + tl + 32u * jb, TR + tl + 8u * GB + 32u * jb, true, x);
              if (!SUB || 32 * (jb + 2) >= mB) {   // the last read of R
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(re);
              }
              if (act) {
#pragma unroll
                for (int t = 0; t < 16; ++t)
                  if (cb + t >= mB) x[t] = 0.f;
#pragma unroll
                for (int t4 = 0; t4 < 4; ++t4)
#pragma unroll
                  for (int c = 0; c < 3; ++c) {
                    gv[c] = fmaf(w[c][t4].x, x[4 * t4], gv[c]);
                    gv[c] = fmaf(w[c][t4].y, x[4 * t4 + 1], gv[c]);
                    gv[c] = fmaf(w[c][t4].z, x[4 * t4 + 2], gv[c]);
                    gv[c] = fmaf(w[c][t4].w, x[4 * t4 + 3], gv[c]);
                  }
              }
              if (!SUB) break;
            }
          }
          if (!(qd * 16 < mA && ok && 32 * h < mB)) {   // nothing to read
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(re);
          } else {
#pragma unroll
            for (int c = 0; c < 3; ++c) gv[c] = warp_sum_f(gv[c]);
            const float g = lane == 0 ? gv[0] : lane == 1 ? gv[1] : gv[2];
            const int p = __shfl_sync(0xffffffffu, p_l, j);
            const int yB = SP == kSplitHalf ? __shfl_sync(0xffffffffu, yB_l, j) : 0;
            if (lane < 3 && g != 0.f) dev::add_gV(P, 3 * p + lane, -(double)g * pscale_d<SP>(-(eR + yB)));
          }
          if (ew == 0)
            fl += (unsigned)(mB * nF * nA) *
                  (unsigned)((sb.als ? 0 : 2 * __shfl_sync(0xffffffffu, nB_l, j)) + 4 * mA);
          ++rb;
          // ---- end of a run: Q -> E, g^C (the two halves take alternate 32-column chunks)
          if (last && ok) {
            run = 0;
            ok = wait_all(qf, seg & 1);
            tc_fence_after();
            if (ok && qd * 16 < mA) {
              double e[4] = {0.0, 0.0, 0.0, 0.0};   // <C, Q>, <grad C, Q> of this warp's part
              for (int jc = h; 32 * jc < 16 * nF; jc += 2) {
                pair_read(T + tl + 32u * jc, 0u, false, x);
                if (alpha < mA && 32 * jc + 16 * pc < 16 * nF) {
                  const float4* src = reinterpret_cast<const float4*>(Cf) + jc * 512 + qd * 32 + lane;
#pragma unroll
                  for (int c = 0; c < 4; ++c) {
                    float s = 0.f;
#pragma unroll
                    for (int t4 = 0; t4 < 4; ++t4) {
                      const float4 y = src[(long long)c * 16 * KP32 + t4 * 128];
                      s = fmaf(y.x, x[4 * t4], s);
                      s = fmaf(y.y, x[4 * t4 + 1], s);
                      s = fmaf(y.z, x[4 * t4 + 2], s);
                      s = fmaf(y.w, x[4 * t4 + 3], s);
                    }
                    e[c] += (double)s;
                  }
                }
              }
#pragma unroll
              for (int c = 0; c < 4; ++c) e[c] = warp_sum_d(e[c]);
              if (lane == 0) {
                const double q1 = pscale_d<SP>(-(P.sc.q[hA] + kUExp + P.sc.d[hA] + P.sc.d[P.c_j[q]]));
                if (e[0] != 0.0) dev::add_E(P, -e[0] * q1);
#pragma unroll
                for (int c = 0; c < 3; ++c)
                  if (e[c + 1] != 0.0) dev::add_gC(P, 3 * q + c, -2.0 * e[c + 1] * q1);
              }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(qe);
            ++seg;
          }
        }
      }
    }
    if (!ok) *abort_flag = 1;
    if (ew == 0 && lane == 0 && fl) atomicAdd(&P.acc[ACC_F1], (double)fl);
  } else if (warp >= kWarpS) {
    // ------------------------------------------------------------ U splitters
    // Lane = row (g, f, beta) of a tile, 16 values over a, split into the two
    // pieces and stored as two core-matrix rows of 16 bytes each; two tiles
    // at a time, so that one's conversions overlap the other's latencies.
    const int qd = warp & 3;
    const uint32_t tl = (uint32_t)(qd * 32) << 16;
    float su = p2f(kUExp - kDExp);   // D.Y -> stored U (bf16 pieces: per B)
    Ring ik, ub, t;
    bool ok = true;
    for (Unit it = next_unit(ik); it.kk >= 0 && ok; it = next_unit(ik)) {
      const int q = it.q(), sA = P.species[P.c_home[q]];
      const int nF = item_sub<SUB>(it.sub(), P.n_abf[sA], P.n_ao[sA], P.n_ao[P.species[P.c_j[q]]]).nF;
      const float inv = 1.0f / (float)nF;
      const long long b0 = X.qoff[q];
      for (int i0 = it.lo; i0 < it.hi && ok; i0 += 32) {
        int ng_l = 0, eU_l = 0;
        if (i0 + lane < it.hi) {
          const int b = P.v_j[X.blist[b0 + i0 + lane]];
          ng_l = ((P.n_abf[P.species[b]] + 7) >> 3) * nF;
          if (SP == kSplitBf16) eU_l = kDExp + P.sc.d[P.c_home[q]] + P.sc.d[b] + y_exp(P, b, P.c_j[q]);
        }
        const int nb = min(32, it.hi - i0);
        for (int j = 0; j < nb && ok; ++j) {
          ok = __all_sync(0xffffffffu, !aborted(abort_flag)) != 0;
          if (!ok) break;
          const int ng = __shfl_sync(0xffffffffu, ng_l, j);
          if (SP == kSplitBf16) su = p2f(-__shfl_sync(0xffffffffu, eU_l, j));
          ok = wait_all(ue + 8 * ub.s, ub.ph ^ 1);
          unsigned char* ubase = smem_raw + CB + ub.s * UBY + (lane & 7) * 16;
          for (int r0 = 0; r0 < ng && ok; r0 += kYG) {
            ok = wait_all(tf + 8 * t.s, t.ph);
            if (!ok) break;
            tc_fence_after();
            uint32_t v[2][16];
            tmem_ld16(TU + tl + 32u * t.s, v[0]);
            tmem_ld16(TU + tl + 32u * t.s + 16u, v[1]);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(te + 8 * t.s);
            t.next(NT);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int r = r0 + 16 * h + qd * 4 + (lane >> 3);
              if (r >= ng) continue;
              int g = (int)((float)r * inv);   // r / nF, exact after the correction
              if (g * nF > r) --g;
              else if ((g + 1) * nF <= r) ++g;
              uint32_t w[8][NP];
#pragma unroll
              for (int k = 0; k < 8; ++k)
                split2<SP>(__uint_as_float(v[h][2 * k]) * su, __uint_as_float(v[h][2 * k + 1]) * su, w[k]);
              unsigned char* d = ubase + g * rowg + (r - g * nF) * 256;
#pragma unroll
              for (int pp = 0; pp < NP; ++pp) {
                *reinterpret_cast<uint4*>(d + pp * (UBY >> 1)) = make_uint4(w[0][pp], w[1][pp], w[2][pp], w[3][pp]);
                *reinterpret_cast<uint4*>(d + pp * (UBY >> 1) + 128) = make_uint4(w[4][pp], w[5][pp], w[6][pp], w[7][pp]);
              }
            }
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(uf + 8 * ub.s);
          ub.next(UB);
        }
      }
    }
    if (!ok) *abort_flag = 1;
  }
  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kWarpU) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(T), "r"(512));
  if (tid == 0 && s_abort) atomicExch(err, 1);
}

// ------------------------------------------------------------------ R2 and Z
// Second exchange product on the tensor cores, per kept pair (A,B) of the
// pass (slot kk of its list), shapes n_abf <= 64, n_ao <= 16:
//   R2 = Y^{AB} . (Y^{BA})^T (M = 64 alpha, N = 64 beta, K = (a, b)) -> E = -<V, R2>, g^V = -<grad V, R2>
//   Z  = V_AB . Y^{BA}       (M = 64 alpha, N = (a, b), K = beta)    -> the Z store read by k_q2_umma
// Both Y operands come whole from the Y build's core-matrix stores (X.ycm):
// Y^{AB} from YspT (rows alpha, K = (a, b)), Y^{BA} from Ysp (rows beta,
// K = (a, b)); Y^{BA} serves R2 as a K-major and Z as an MN-major operand.
// V pieces and FP32 V, grad V from X.Vz.  CTA c takes the pairs c, c + grid,
// ...  Warp 0 lane 0 copies (bulk), warp 1 owns tensor memory and its lane 0
// issues the MMAs, warps 2-5 (one per tensor-memory lane quarter) are the
// epilogue.  R2 is double-buffered in tensor memory, Z single-buffered;
// Y^{AB} is released after R2, Y^{BA} and V after Z, so the next pair's
// Y^{AB} lands while Z runs.  Every wait is bounded (1 s); a timeout sets the
// error flag and every role stops.
constexpr int kT2Threads = 192;
constexpr int kT2RCol = 256;   // tensor-memory column of the first R2 accumulator (Z at column 0)

template <int SP>
__global__ void __launch_bounds__(kT2Threads, 1)
    k_t2_umma(DevPlan P, MixPlan X, const int* list, int n_list, int KKmax, long long zblk, int* err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  uint16_t* Ya = reinterpret_cast<uint16_t*>(smem_raw);   // [NP][rup8(n_abf(A))][KK]
  uint16_t* Yb = Ya + (size_t)NP * 64 * KKmax;            // [NP][rup8(n_abf(B))][KK]
  uint16_t* Vs = Yb + (size_t)NP * 64 * KKmax;            // [NP][64][64]
  __shared__ __align__(8) uint64_t b_af, b_ae, b_bf, b_be, b_rf[2], b_re[2], b_zf, b_ze, b_done;
  __shared__ uint32_t tmem_base;
  __shared__ int s_abort;
  volatile int* abort_flag = &s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto sa = [](const void* p) { return (uint32_t)__cvta_generic_to_shared(p); };
  const uint32_t mAf = sa(&b_af), mAe = sa(&b_ae), mBf = sa(&b_bf), mBe = sa(&b_be), rf = sa(b_rf), re = sa(b_re),
                 zf = sa(&b_zf), ze = sa(&b_ze), mdone = sa(&b_done);
  // rows past n_abf are read as they lie (their results are dropped or meet
  // zero V): the buffers start out finite
  for (int o = tid; o < NP * (2 * 64 * KKmax + 4096) / 8; o += kT2Threads)
    reinterpret_cast<uint4*>(smem_raw)[o] = make_uint4(0u, 0u, 0u, 0u);
  fence_async_smem();
  if (tid == 0) {
    s_abort = 0;
    mbar_init(mAf, 1);
    mbar_init(mAe, 1);
    mbar_init(mBf, 1);
    mbar_init(mBe, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(rf + 8 * s, 1);
      mbar_init(re + 8 * s, 4);
    }
    mbar_init(zf, 1);
    mbar_init(ze, 4);
    mbar_init(mdone, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(sa(&tmem_base)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t T = tmem_base;

  if (warp == 0) {
    // ------------------------------------------------------------- producer
    if (lane == 0) {
      uint32_t na = 0, nb = 0;   // copies issued into Ya and into Yb / V
      for (int kk = blockIdx.x; kk < n_list && !aborted(abort_flag); kk += gridDim.x) {
        const int p = list[kk];
        const int A = P.v_home[p], b = P.v_j[p];
        const int* Rb = P.v_R + 3 * p;
        const int KK = 16 * P.n_ao[P.species[A]];
        const int y1 = ylut_get(P, A, b, Rb[0], Rb[1], Rb[2]);
        const int y2 = ylut_get(P, b, A, -Rb[0], -Rb[1], -Rb[2]);
        if (y1 < 0 || y2 < 0) {   // a kept pair always has both Y blocks
          *abort_flag = 1;
          break;
        }
        // rows alpha (beta) in whole groups of 8
        const uint32_t abytes = (uint32_t)NP * (uint32_t)((P.n_abf[P.species[A]] + 7) & ~7) * (uint32_t)KK * 2u;
        const uint32_t bbytes = (uint32_t)NP * (uint32_t)((P.n_abf[P.species[b]] + 7) & ~7) * (uint32_t)KK * 2u;
        if (na >= 1 && !mbar_wait(mAe, (na - 1) & 1)) {
          *abort_flag = 1;
          break;
        }
        mbar_expect_tx(mAf, abytes);
        bulk_g2s(sa(Ya), X.YspT + X.y_idx[y1] * X.yT_blk, abytes, mAf);
        ++na;
        if (nb >= 1 && !mbar_wait(mBe, (nb - 1) & 1)) {
          *abort_flag = 1;
          break;
        }
        mbar_expect_tx(mBf, bbytes + (uint32_t)NP * 8192u);
        bulk_g2s(sa(Yb), X.Ysp + P.y_off[y2], bbytes, mBf);
        bulk_g2s(sa(Vs), X.Vz + (long long)kk * X.vz_blk, (uint32_t)NP * 8192u, mBf);
        ++nb;
      }
      // copies in flight land before the CTA leaves
      if (na) mbar_wait(mAf, (na - 1) & 1);
      if (nb) mbar_wait(mBf, (nb - 1) & 1);
    }
  } else if (warp == 1) {
    // ----------------------------------------------------------- MMA issuer
    if (lane == 0) {
      const uint32_t idR = idesc_split<SP>(64, 64, 0);
      uint32_t i = 0;
      bool ok = true;
      for (int kk = blockIdx.x; kk < n_list && ok; kk += gridDim.x, ++i) {
        if (aborted(abort_flag)) {
          ok = false;
          break;
        }
        const int pr = list[kk], sA = P.species[P.v_home[pr]], mB = P.n_abf[P.species[P.v_j[pr]]];
        const int nA = P.n_ao[sA];
        const int KK = 16 * nA;
        const uint32_t PA = (uint32_t)((P.n_abf[sA] + 7) & ~7) * (uint32_t)KK * 2u;   // bytes of one piece of Y^{AB}
        const uint32_t PB = (uint32_t)((mB + 7) & ~7) * (uint32_t)KK * 2u;            // and of Y^{BA}
        const uint32_t rowg = 16u * (uint32_t)KK;      // bytes between 8-row groups
        const uint64_t dA = sdesc2(sa(Ya), 128, rowg), dBK = sdesc2(sa(Yb), 128, rowg);
        const uint64_t dV = sdesc2(sa(Vs), 128, 1024), dBM = sdesc2(sa(Yb), rowg, 128);
        const uint32_t idZ = idesc_split<SP>(64, KK, 1);
        const int rbuf = i & 1;
        ok = mbar_wait(mAf, i & 1) && mbar_wait(mBf, i & 1) && (i < 2 || mbar_wait(re + 8 * rbuf, ((i >> 1) - 1) & 1));
        if (!ok) break;
        tc_fence_after();
        // R2: one a (16 columns, 256 bytes) per k step, every piece product
        const uint32_t tR = T + kT2RCol + 64u * rbuf;
        for (int a = 0; a < nA; ++a) {
          const uint64_t o = 16u * (uint32_t)a;
          int k = 0;
#pragma unroll
          for (int sum = NP - 1; sum >= 0; --sum)
#pragma unroll
            for (int ia = 0; ia <= sum; ++ia, ++k)
              umma_f16(tR, dA + ((uint64_t)(ia * PA) >> 4) + o, dBK + ((uint64_t)((sum - ia) * PB) >> 4) + o, idR,
                        (a > 0 || k > 0) ? 1u : 0u);
        }
        umma_commit(mAe);
        umma_commit(rf + 8 * rbuf);
        ok = i < 1 || mbar_wait(ze, (i - 1) & 1);
        if (!ok) break;
        tc_fence_after();
        // Z: K = beta in steps of 16 (V: 256 bytes; Y^{BA} MN-major: two 8-row groups)
        for (int kb = 0; 16 * kb < mB; ++kb) {
          int k = 0;
#pragma unroll
          for (int sum = NP - 1; sum >= 0; --sum)
#pragma unroll
            for (int ia = 0; ia <= sum; ++ia, ++k)
              umma_f16(T, dV + ((uint64_t)(ia * 8192) >> 4) + 16u * kb,
                        dBM + ((uint64_t)((sum - ia) * PB) >> 4) + ((uint64_t)(2 * rowg * kb) >> 4), idZ,
                        (kb > 0 || k > 0) ? 1u : 0u);
        }
        umma_commit(mBe);
        umma_commit(zf);
      }
      if (!ok) *abort_flag = 1;
      // every MMA issued has completed before tensor memory is freed
      umma_commit(mdone);
      mbar_wait(mdone, 0);
    }
  } else {
    // ------------------------------------------------------------- epilogue
    const int qd = warp & 3;                   // tensor-memory lane quarter
    const int alpha = qd * 16 + (lane & 15);   // accumulator row held by this thread
    const int half = lane >> 4;                // columns [0,16) or [16,32) of a 32-column load
    const uint32_t tl = T + ((uint32_t)(qd * 32) << 16);
    uint32_t i = 0;
    bool ok = true;
    double fl = 0.0;
    for (int kk = blockIdx.x; kk < n_list && ok; kk += gridDim.x, ++i) {
      ok = __all_sync(0xffffffffu, !aborted(abort_flag)) != 0;
      if (!ok) break;
      const int p = list[kk];
      const int sA = P.species[P.v_home[p]], sB = P.species[P.v_j[p]];
      const int nA = P.n_ao[sA], nB = P.n_ao[sB], mA = P.n_abf[sA], mB = P.n_abf[sB];
      const int KK = 16 * nA;
      const int rbuf = i & 1;
      const int hA = P.v_home[p], hB = P.v_j[p];
      const float sz = pscale<SP>(P.sc.z[hA] - P.sc.q[hA] - P.sc.d[hA]);   // V.Y -> stored Z
      const double r2 = pscale_d<SP>(-r2_exp(P, hA, hB));
      // ---- R2 -> E, g^V (the V, grad V rows of the first 32 columns are
      // fetched before the wait; they do not depend on R2)
      const float4* V4 = reinterpret_cast<const float4*>(X.Vz + (long long)kk * X.vz_blk + NP * 4096) + qd * 32 + lane;
      float ev[4] = {0.f, 0.f, 0.f, 0.f};
      float4 w[4][4];
      if (alpha < mA && 16 * half < mB)
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int t4 = 0; t4 < 4; ++t4) w[c][t4] = V4[c * 1024 + t4 * 128];
      ok = wait_all(rf + 8 * rbuf, (i >> 1) & 1);
      tc_fence_after();
      if (ok) {
        for (int c0 = 0; c0 < 64; c0 += 32) {
          if (c0 >= mB) break;
          const bool act = alpha < mA && c0 + 16 * half < mB;
          if (c0 > 0 && act)
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
              for (int t4 = 0; t4 < 4; ++t4) w[c][t4] = V4[c * 1024 + 512 + t4 * 128];
          uint32_t v[32];
          tmem_ld32(tl + kT2RCol + 64u * rbuf + c0, v);
          float x[16];
#pragma unroll
          for (int t = 0; t < 16; ++t) {
            const float hi = __shfl_sync(0xffffffffu, __uint_as_float(v[16 + t]), lane & 15);
            x[t] = half ? hi : __uint_as_float(v[t]);
          }
          if (act) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              float s = 0.f;
#pragma unroll
              for (int t4 = 0; t4 < 4; ++t4) {
                s = fmaf(w[c][t4].x, x[4 * t4], s);
                s = fmaf(w[c][t4].y, x[4 * t4 + 1], s);
                s = fmaf(w[c][t4].z, x[4 * t4 + 2], s);
                s = fmaf(w[c][t4].w, x[4 * t4 + 3], s);
              }
              ev[c] += s;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(re + 8 * rbuf);
#pragma unroll
      for (int c = 0; c < 4; ++c) ev[c] = warp_sum_f(ev[c]);
      if (lane == 0 && ok) {
        if (ev[0] != 0.f) dev::add_E(P, -(double)ev[0] * r2);
#pragma unroll
        for (int c = 0; c < 3; ++c)
          if (ev[c + 1] != 0.f) dev::add_gV(P, 3 * p + c, -(double)ev[c + 1] * r2);
      }
      // ---- Z -> the Z store: NP planes of 128-row tiles of rows (alpha, a),
      // 16 columns b each, in the core-matrix order of tix; a thread writes
      // the 16 b of one (alpha, a) as two 16-byte chunks per piece
      ok = ok && wait_all(zf, i & 1);
      tc_fence_after();
      if (ok) {
        uint16_t* Zo = X.Zst + (long long)kk * zblk;
        for (int c0 = 0; c0 < KK; c0 += 32) {
          uint32_t v[32];
          tmem_ld32(tl + c0, v);
          float x[16];
#pragma unroll
          for (int t = 0; t < 16; ++t) {
            const float hi = __shfl_sync(0xffffffffu, __uint_as_float(v[16 + t]), lane & 15);
            x[t] = half ? hi : __uint_as_float(v[t]);
          }
          const int a = (c0 >> 4) + half;
          if (alpha < mA && a < nA) {
            const int r = alpha * nA + a;
            uint16_t* d = Zo + (long long)(r >> 7) * NP * 2048 + (((r & 127) >> 3) << 7) + ((r & 7) << 3);
#pragma unroll
            for (int hb = 0; hb < 2; ++hb) {
              float x0[4], x1[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                x0[k] = x[8 * hb + k] * sz;
                x1[k] = x[8 * hb + 4 + k] * sz;
              }
              uint2 p0[NP], p1[NP];
              split4<SP>(x0, p0);
              split4<SP>(x1, p1);
#pragma unroll
              for (int pp = 0; pp < NP; ++pp)
                *reinterpret_cast<uint4*>(d + pp * 2048 + 64 * hb) = make_uint4(p0[pp].x, p0[pp].y, p1[pp].x, p1[pp].y);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(ze);
      if (warp == 2 && lane == 0) fl += 4.0 * mA * mB * nA * nB;
    }
    if (!ok) *abort_flag = 1;
    if (warp == 2 && lane == 0 && fl != 0.0) atomicAdd(&P.acc[ACC_F2], fl);
  }
  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(T), "r"(512));
  if (tid == 0 && s_abort) atomicExch(err, 1);
}

// The same products for plans with sub-blocks (n_ao beyond 16, n_abf up to
// 128, fp16 pieces): M = 128 rows alpha, and the K = (a, b) and N = (a, b)
// columns in chunks, one sub-block of A's orbitals times one of B's, which
// come from the Y build's sub-block stores (Y^{BA} of a chunk from X.Yh,
// Y^{AB} from X.YspT with a and b exchanged).  R2 runs on over a pair's
// chunks; Z of a chunk goes to the Z store of (slot, sub of b).  Roles and
// buffers as k_t2_umma; V, grad V as four planes [beta / 4][alpha SA][4], so
// that a warp's 32 rows are 512 consecutive bytes.
// What bounds it: the latency of a chunk's copies (one chunk in shared memory,
// 66 KB per operand at n_abf 75 and 13 orbitals) and of the epilogue's reads
// of V, grad V.  The warp-level kernel (k_term2_w, still taken by HFX_BF16X3
// and by shapes beyond shared memory) stages Y element by element and reads
// FP64 V blocks: with the build of those 4.9 ms of a 40-atom perovskite
// evaluation (9,896 pairs), 0.85 ms here with k_t2w_vstore.
__global__ void __launch_bounds__(256) k_t2w_vstore(DevPlan P, MixPlan X, T2WPlan S, const int* list, int n) {
  constexpr int SP = kSplitHalf;
  for (int k = blockIdx.x; k < n; k += gridDim.x) {
    const int p = list[k], sA = P.species[P.v_home[p]], sB = P.species[P.v_j[p]];
    const int mA = P.n_abf[sA], mB = P.n_abf[sB], m8 = (mA + 7) & ~7;
    double h, g[3];
    model::v_pair(P, p, h, g);
    const float f[4] = {(float)h, (float)g[0], (float)g[1], (float)g[2]};
    const float* M = P.Mf + P.M_off[sA * P.S + sB];
    const float sv = pscale<SP>(v_exp(P, P.v_home[p], P.v_j[p]));
    uint16_t* out = X.Vz + (long long)k * X.vz_blk;
    for (int t4 = threadIdx.x; t4 < m8 * S.VK / 4; t4 += blockDim.x) {   // core-matrix order, 4 columns per thread
      const int t = 4 * t4, g8 = t / (8 * S.VK), u = t - g8 * 8 * S.VK;
      const int al = g8 * 8 + ((u >> 3) & 7), be = ((u >> 6) << 3) + (u & 7);
      float x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = (al < mA && be + j < mB) ? M[al * mB + be + j] * f[0] * sv : 0.f;
      uint2 pc[NP];
      split4<SP>(x, pc);
#pragma unroll
      for (int pp = 0; pp < NP; ++pp) *reinterpret_cast<uint2*>(out + pp * m8 * S.VK + t) = pc[pp];
    }
    float4* pl = reinterpret_cast<float4*>(out + NP * S.M8 * S.VK);
    const int nb4 = (mB + 3) >> 2, PL = (S.VK >> 2) * S.SA;
    for (int e = threadIdx.x; e < nb4 * mA; e += blockDim.x) {
      const int b4 = e / mA, al = e - b4 * mA, be = 4 * b4;
      const float* m = M + al * mB + be;
      const float4 v = make_float4(m[0], be + 1 < mB ? m[1] : 0.f, be + 2 < mB ? m[2] : 0.f, be + 3 < mB ? m[3] : 0.f);
#pragma unroll
      for (int c = 0; c < 4; ++c)
        pl[c * PL + b4 * S.SA + al] = make_float4(v.x * f[c], v.y * f[c], v.z * f[c], v.w * f[c]);
    }
  }
}

__global__ void __launch_bounds__(kT2Threads, 1)
    k_t2w_umma(DevPlan P, MixPlan X, T2WPlan S, const int* list, int n_list, long long zblk, int* err) {
  constexpr int SP = kSplitHalf;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t b_af, b_ae, b_bf, b_be, b_vf, b_ve, b_rf[2], b_re[2], b_zf, b_ze, b_done;
  __shared__ uint32_t tmem_base;
  __shared__ int s_abort;
  volatile int* abort_flag = &s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto sa = [](const void* p) { return (uint32_t)__cvta_generic_to_shared(p); };
  const uint32_t Vs = sa(smem_raw), Ya = Vs + S.v_bytes, Yb = Ya + S.y_bytes;
  const uint32_t mAf = sa(&b_af), mAe = sa(&b_ae), mBf = sa(&b_bf), mBe = sa(&b_be), mVf = sa(&b_vf), mVe = sa(&b_ve),
                 rf = sa(b_rf), re = sa(b_re), zf = sa(&b_zf), ze = sa(&b_ze), mdone = sa(&b_done);
  // rows past a block's own are read as they lie (dropped, or against zeros of V): finite from the start
  for (uint32_t o = tid * 16u; o < S.smem; o += kT2Threads * 16u)
    *reinterpret_cast<uint4*>(smem_raw + o) = make_uint4(0u, 0u, 0u, 0u);
  fence_async_smem();
  if (tid == 0) {
    s_abort = 0;
    for (uint32_t m : {mAf, mAe, mBf, mBe, mVf, mVe, rf, rf + 8, zf, mdone}) mbar_init(m, 1);
    for (uint32_t m : {re, re + 8, ze}) mbar_init(m, 4);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(sa(&tmem_base)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t T = tmem_base;
  // A pair's shapes and its chunks (as, bs), bs fastest.
  struct Pair {
    int p, A, B, nA, nB, mA, mB, a8, b8, hA, sA, sB;
    __device__ int n() const { return sA * sB; }
    __device__ int as(int c) const { return c / sB; }
    __device__ int bs(int c) const { return c % sB; }
    __device__ int na(int c) const { return min(hA, nA - as(c) * hA); }   // a of chunk c
  };
  auto pair_of = [&](int kk) {
    Pair q;
    q.p = list[kk];
    q.A = P.v_home[q.p];
    q.B = P.v_j[q.p];
    const int tA = P.species[q.A], tB = P.species[q.B];
    q.nA = P.n_ao[tA];
    q.nB = P.n_ao[tB];
    q.mA = P.n_abf[tA];
    q.mB = P.n_abf[tB];
    q.a8 = (q.mA + 7) & ~7;
    q.b8 = (q.mB + 7) & ~7;
    q.hA = ao_sub(q.nA);
    q.sA = ao_subs(q.nA);
    q.sB = ao_subs(q.nB);
    return q;
  };

  if (warp == 0) {
    // ------------------------------------------------------------- producer
    if (lane == 0) {
      uint32_t na = 0, nb = 0, nv = 0;   // copies issued into Ya, Yb, V
      bool ok = true;
      for (int kk = blockIdx.x; kk < n_list && ok; kk += gridDim.x) {
        const Pair q = pair_of(kk);
        const int* Rb = P.v_R + 3 * q.p;
        const int y1 = ylut_get(P, q.A, q.B, Rb[0], Rb[1], Rb[2]);
        const int y2 = ylut_get(P, q.B, q.A, -Rb[0], -Rb[1], -Rb[2]);
        ok = y1 >= 0 && y2 >= 0;   // a kept pair always has both Y blocks
        for (int c = 0; c < q.n() && ok; ++c) {
          const int n = q.na(c), a0 = q.as(c) * q.hA, bs = q.bs(c);
          const uint32_t ca = 32u * q.a8 * n, cb = 32u * q.b8 * n;   // bytes of one piece of the chunk
          const long long ax = 16ll * q.a8 * q.nA, bx = 16ll * q.b8 * q.nA;   // elements of one sub of b
          const uint16_t* src_a = X.YspT + P.y_off[y1] + bs * ax + 16ll * q.a8 * a0;
          const uint16_t* src_b = X.Yh + P.y_off[y2] + bs * bx + 16ll * q.b8 * a0;
          ok = !aborted(abort_flag) && (na < 1 || mbar_wait(mAe, (na - 1) & 1));
          if (!ok) break;
          mbar_expect_tx(mAf, NP * ca);
          for (int pp = 0; pp < NP; ++pp) bulk_g2s(Ya + pp * ca, src_a + pp * q.sB * ax, ca, mAf);
          ++na;
          if (c == 0) {
            ok = nv < 1 || mbar_wait(mVe, (nv - 1) & 1);
            if (!ok) break;
            const uint32_t vb = (uint32_t)NP * q.a8 * S.VK * 2u;
            mbar_expect_tx(mVf, vb);
            bulk_g2s(Vs, X.Vz + (long long)kk * X.vz_blk, vb, mVf);
            ++nv;
          }
          ok = nb < 1 || mbar_wait(mBe, (nb - 1) & 1);
          if (!ok) break;
          mbar_expect_tx(mBf, NP * cb);
          for (int pp = 0; pp < NP; ++pp) bulk_g2s(Yb + pp * cb, src_b + pp * q.sB * bx, cb, mBf);
          ++nb;
        }
      }
      if (!ok) *abort_flag = 1;
      // copies in flight land before the CTA leaves
      if (na) mbar_wait(mAf, (na - 1) & 1);
      if (nv) mbar_wait(mVf, (nv - 1) & 1);
      if (nb) mbar_wait(mBf, (nb - 1) & 1);
    }
  } else if (warp == 1) {
    // ----------------------------------------------------------- MMA issuer
    if (lane == 0) {
      uint32_t i = 0, t = 0;   // pairs, chunks
      bool ok = true;
      for (int kk = blockIdx.x; kk < n_list && ok; kk += gridDim.x, ++i) {
        const Pair q = pair_of(kk);
        const uint32_t idR = idesc_split<SP>(128, (q.mB + 15) & ~15, 0), tR = T + kT2RCol + 128u * (i & 1);
        const uint64_t vp = (uint64_t)(2u * q.a8 * S.VK) >> 4;   // a piece of V
        const uint64_t dV = sdesc2(Vs, 128, 16u * S.VK);
        ok = i < 2 || mbar_wait(re + 8 * (i & 1), ((i >> 1) - 1) & 1);
        for (int c = 0; c < q.n() && ok; ++c, ++t) {
          const int n = q.na(c), last = c == q.n() - 1;
          const uint32_t rowg = 256u * n;   // bytes between 8-row groups
          const uint64_t pa = (uint64_t)(32u * q.a8 * n) >> 4, pb = (uint64_t)(32u * q.b8 * n) >> 4;
          const uint64_t dA = sdesc2(Ya, 128, rowg), dB = sdesc2(Yb, 128, rowg), dZ = sdesc2(Yb, rowg, 128);
          ok = !aborted(abort_flag) && mbar_wait(mAf, t & 1) && mbar_wait(mBf, t & 1);
          if (!ok) break;
          tc_fence_after();
          for (int a = 0; a < n; ++a) {   // R2: one a (16 columns, 256 bytes) per k step
            const uint64_t o = 16u * (uint32_t)a;
            umma_f16(tR, dA + o, dB + pb + o, idR, (c > 0 || a > 0) ? 1u : 0u);
            umma_f16(tR, dA + pa + o, dB + o, idR, 1u);
            umma_f16(tR, dA + o, dB + o, idR, 1u);
          }
          umma_commit(mAe);
          if (last) umma_commit(rf + 8 * (i & 1));
          ok = (c > 0 || mbar_wait(mVf, i & 1)) && (t < 1 || mbar_wait(ze, (t - 1) & 1));
          if (!ok) break;
          tc_fence_after();
          const uint32_t idZ = idesc_split<SP>(128, 16 * n, 1);
          for (int kb = 0; 16 * kb < q.mB; ++kb) {   // Z: K = beta in steps of 16 (V: 256 bytes; Y^{BA}: two 8-row groups)
            const uint64_t o = 16u * (uint32_t)kb, oz = (uint64_t)(2 * rowg * kb) >> 4;
            umma_f16(T, dV + o, dZ + pb + oz, idZ, kb > 0 ? 1u : 0u);
            umma_f16(T, dV + vp + o, dZ + oz, idZ, 1u);
            umma_f16(T, dV + o, dZ + oz, idZ, 1u);
          }
          umma_commit(mBe);
          if (last) umma_commit(mVe);
          umma_commit(zf);
        }
      }
      if (!ok) *abort_flag = 1;
      // every MMA issued has completed before tensor memory is freed
      umma_commit(mdone);
      mbar_wait(mdone, 0);
    }
  } else {
    // ------------------------------------------------------------- epilogue
    const int qd = warp & 3, alpha = 32 * qd + lane;   // tensor-memory lane quarter, accumulator row
    const uint32_t tl = T + ((uint32_t)(qd * 32) << 16);
    const int PL = (S.VK >> 2) * S.SA;   // float4 per plane
    uint32_t i = 0, t = 0;
    bool ok = true;
    double fl = 0.0;
    for (int kk = blockIdx.x; kk < n_list && ok; kk += gridDim.x, ++i) {
      ok = __all_sync(0xffffffffu, !aborted(abort_flag)) != 0;
      if (!ok) break;
      const Pair q = pair_of(kk);
      const bool rows = 32 * qd < q.mA, act = alpha < q.mA;
      const float sz = pscale<SP>(P.sc.z[q.A] - P.sc.q[q.A] - P.sc.d[q.A]);   // V.Y -> stored Z
      const double r2 = pscale_d<SP>(-r2_exp(P, q.A, q.B));
      const float4* V4 = reinterpret_cast<const float4*>(X.Vz + (long long)kk * X.vz_blk + NP * S.M8 * S.VK) + alpha;
      float4 w[4][4];
      auto fetch = [&](int cb) {   // V, grad V of columns 16 cb .. + 15
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int t4 = 0; t4 < 4; ++t4)
            w[c][t4] = act && 16 * cb + 4 * t4 < q.mB ? V4[c * PL + (4 * cb + t4) * S.SA] : make_float4(0.f, 0.f, 0.f, 0.f);
      };
      for (int c = 0; c < q.n() && ok; ++c, ++t) {
        if (c == q.n() - 1) {   // R2 -> E, g^V
          float ev[4] = {0.f, 0.f, 0.f, 0.f};
          fetch(0);   // (does not depend on R2)
          ok = wait_all(rf + 8 * (i & 1), (i >> 1) & 1);
          tc_fence_after();
          if (ok && rows) {
#pragma unroll 1
            for (int cb = 0; 16 * cb < q.mB; ++cb) {
              if (cb) fetch(cb);
              uint32_t v[16];
              tmem_ld16(tl + kT2RCol + 128u * (i & 1) + 16u * cb, v);
              tmem_wait_ld();
              if (act) {
                float x[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) x[k] = 16 * cb + k < q.mB ? __uint_as_float(v[k]) : 0.f;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  float s = 0.f;
#pragma unroll
                  for (int t4 = 0; t4 < 4; ++t4) {
                    s = fmaf(w[k][t4].x, x[4 * t4], s);
                    s = fmaf(w[k][t4].y, x[4 * t4 + 1], s);
                    s = fmaf(w[k][t4].z, x[4 * t4 + 2], s);
                    s = fmaf(w[k][t4].w, x[4 * t4 + 3], s);
                  }
                  ev[k] += s;
                }
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(re + 8 * (i & 1));
          if (ok && rows) {
#pragma unroll
            for (int k = 0; k < 4; ++k) ev[k] = warp_sum_f(ev[k]);
            if (lane == 0) {
              if (ev[0] != 0.f) dev::add_E(P, -(double)ev[0] * r2);
#pragma unroll
              for (int k = 0; k < 3; ++k)
                if (ev[k + 1] != 0.f) dev::add_gV(P, 3 * q.p + k, -(double)ev[k + 1] * r2);
            }
          }
        }
        // ---- Z of the chunk -> the Z store of (slot, sub of b): 128-row tiles of rows (alpha, a), 16 columns b
        ok = ok && wait_all(zf, t & 1);
        tc_fence_after();
        if (ok && rows) {
          uint16_t* Zo = X.Zst + ((long long)kk * X.KB + q.bs(c)) * zblk;
          const int n = q.na(c), r0 = alpha * q.nA + q.as(c) * q.hA;
#pragma unroll 1
          for (int a = 0; a < n; ++a) {
            uint32_t v[16];
            tmem_ld16(tl + 16u * a, v);
            tmem_wait_ld();
            if (!act) continue;
            const int r = r0 + a;
            uint16_t* d = Zo + (long long)(r >> 7) * NP * 2048 + (((r & 127) >> 3) << 7) + ((r & 7) << 3);
            uint32_t pc[8][NP];
#pragma unroll
            for (int k = 0; k < 8; ++k)
              split2<SP>(__uint_as_float(v[2 * k]) * sz, __uint_as_float(v[2 * k + 1]) * sz, pc[k]);
#pragma unroll
            for (int pp = 0; pp < NP; ++pp) {
              *reinterpret_cast<uint4*>(d + pp * 2048) = make_uint4(pc[0][pp], pc[1][pp], pc[2][pp], pc[3][pp]);
              *reinterpret_cast<uint4*>(d + pp * 2048 + 64) = make_uint4(pc[4][pp], pc[5][pp], pc[6][pp], pc[7][pp]);
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(ze);
      }
      if (warp == 2 && lane == 0) fl += 4.0 * q.mA * q.mB * q.nA * q.nB;
    }
    if (!ok) *abort_flag = 1;
    if (warp == 2 && lane == 0 && fl != 0.0) atomicAdd(&P.acc[ACC_F2], fl);
  }
  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(T), "r"(512));
  if (tid == 0 && s_abort) atomicExch(err, 1);
}

int num_sms() {
  static const int n = [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 152;
  }();
  return n;
}

}  // namespace

long long t1u_launch_count() { return g_t1u_launches; }

size_t t1u_smem(int KP, int GA, int GB, int KB, int UB, int NS) {
  return t1_base(KP, GA, GB, KB, UB) + (size_t)NS * kYSlot;
}

int t1u_utiles(int KP, int GB) { return t1_utiles(KP, GB); }

int t1u_max_slots() { return kMaxNS; }

int sm_count() { return num_sms(); }

namespace {
using T1Kern = void (*)(DevPlan, MixPlan, T1UPlan, const int*, int, int*, int*);
T1Kern t1_kern(int sp, bool sub) {
  if (sp == kSplitBf16) return sub ? k_t1_umma<kSplitBf16, true> : k_t1_umma<kSplitBf16, false>;
  return sub ? k_t1_umma<kSplitHalf, true> : k_t1_umma<kSplitHalf, false>;
}
}  // namespace

cudaError_t t1u_set_smem(int sp, bool sub) { return allow_max_dynamic_smem((const void*)t1_kern(sp, sub)); }

cudaError_t launch_t1u_cstore(const DevPlan& P, const T1UPlan& U, int sp, const int* qlist, int nq, cudaStream_t s) {
  if (nq <= 0) return cudaSuccess;
  ++g_t1u_launches;
  static std::once_flag attr;
  std::call_once(attr, [] {
    cudaFuncSetAttribute(k_t1u_cstore<kSplitBf16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCStoreSmem);
    cudaFuncSetAttribute(k_t1u_cstore<kSplitHalf>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCStoreSmem);
  });
  const int g = nq < 152 * 3 ? nq : 152 * 3;
  if (sp == kSplitBf16) k_t1u_cstore<kSplitBf16><<<g, 256, kCStoreSmem, s>>>(P, U, qlist, nq);
  else k_t1u_cstore<kSplitHalf><<<g, 256, kCStoreSmem, s>>>(P, U, qlist, nq);
  return cudaGetLastError();
}

cudaError_t launch_lpt_order(const int* key, int asc, const int* list, int n_max, const long long* n_dev, int* hist,
                             int* out, cudaStream_t s) {
  if (n_max <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(hist, 0, kLptBuckets * sizeof(int), s);
  if (e != cudaSuccess) return e;
  g_t1u_launches += 3;
  const int g = std::min((n_max + 255) / 256, 152 * 8);
  k_lpt_hist<<<g, 256, 0, s>>>(key, asc, list, n_dev, hist);
  k_lpt_scan<<<1, 1024, 0, s>>>(hist);
  k_lpt_scatter<<<g, 256, 0, s>>>(key, asc, list, n_dev, hist, out);
  return cudaGetLastError();
}

cudaError_t launch_vstores(const DevPlan& P, const MixPlan& X, const T1UPlan& U, int sp, const int* list, int n,
                           cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  ++g_t1u_launches;
  const size_t sm = vstore_smem(U.VK > 64 ? U.VK : 64);
  cudaError_t e = allow_max_dynamic_smem(sp == kSplitBf16 ? (const void*)k_vstores<kSplitBf16>
                                                          : (const void*)k_vstores<kSplitHalf>);
  if (e != cudaSuccess) return e;
  const int g = n < 152 * 3 ? n : 152 * 3;
  if (sp == kSplitBf16) k_vstores<kSplitBf16><<<g, 256, sm, s>>>(P, X, U, list, n);
  else k_vstores<kSplitHalf><<<g, 256, sm, s>>>(P, X, U, list, n);
  return cudaGetLastError();
}

// Entries (C pair, sub) of the kept C pairs q of [q0, q1) from list[idx[q]] on.
__global__ void k_t1_items(DevPlan P, const int* qcnt, const long long* idx, int q0, int q1, int* list) {
  for (int q = q0 + blockIdx.x * blockDim.x + threadIdx.x; q < q1; q += gridDim.x * blockDim.x) {
    if (qcnt[q] == 0) continue;
    const int sA = P.species[P.c_home[q]];
    const int n = abf_subs(P.n_abf[sA]) * ao_subs(P.n_ao[sA]) * ao_subs(P.n_ao[P.species[P.c_j[q]]]);
    for (int k = 0; k < n; ++k) list[idx[q] + k] = q | (k << kItemShift);
  }
}

cudaError_t launch_t1_items(const DevPlan& P, const int* qcnt, const long long* idx, int q0, int q1, int* list,
                            cudaStream_t s) {
  if (q1 <= q0) return cudaSuccess;
  ++g_t1u_launches;
  k_t1_items<<<std::min((q1 - q0 + 255) / 256, 152 * 8), 256, 0, s>>>(P, qcnt, idx, q0, q1, list);
  return cudaGetLastError();
}

size_t t2u_smem(int max_ao) { return (size_t)NP * (2 * 64 * 16 * (size_t)max_ao * 2 + 8192); }

cudaError_t t2u_set_smem(int sp) {
  return allow_max_dynamic_smem(sp == kSplitBf16 ? (const void*)k_t2_umma<kSplitBf16> : (const void*)k_t2_umma<kSplitHalf>);
}

cudaError_t launch_t2_umma(const DevPlan& P, const MixPlan& X, int sp, const int* list, int n, long long zblk,
                           size_t smem, int* err, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  ++g_t1u_launches;
  const int grid = n < num_sms() ? n : num_sms();
  const int KKmax = (int)(smem / NP - 8192) / (2 * 64 * 2);   // 16 x the largest n_ao
  if (sp == kSplitBf16) k_t2_umma<kSplitBf16><<<grid, kT2Threads, smem, s>>>(P, X, list, n, KKmax, zblk, err);
  else k_t2_umma<kSplitHalf><<<grid, kT2Threads, smem, s>>>(P, X, list, n, KKmax, zblk, err);
  return cudaGetLastError();
}

T2WPlan t2w_plan(int max_abf, int max_ao_sub) {
  T2WPlan S;
  S.M8 = (max_abf + 7) & ~7;
  S.VK = (max_abf + 15) & ~15;
  S.SA = (max_abf + 31) & ~31;
  S.v_bytes = (uint32_t)NP * S.M8 * S.VK * 2u;
  const uint32_t col = 32u * max_ao_sub;   // bytes of a row of a chunk
  S.y_bytes = (uint32_t)NP * S.M8 * col;
  // the operands' reads beyond a block's rows: 128 rows of V and of Y^{AB},
  // n_abf(B) rounded up to 16 of Y^{BA}, each from its second piece on
  S.smem = S.v_bytes + 2 * S.y_bytes + 8 * col;
  S.smem = std::max(S.smem, (uint32_t)(S.M8 + 128) * S.VK * 2u);
  S.smem = std::max(S.smem, S.v_bytes + (S.M8 + 128) * col);
  S.smem = (S.smem + 15u) & ~15u;
  return S;
}

cudaError_t t2w_set_smem() { return allow_max_dynamic_smem((const void*)k_t2w_umma); }

cudaError_t launch_t2w(const DevPlan& P, const MixPlan& X, const T2WPlan& S, const int* list, int n, long long zblk,
                       int* err, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  g_t1u_launches += 2;
  k_t2w_vstore<<<std::min(n, 152 * 8), 256, 0, s>>>(P, X, S, list, n);
  k_t2w_umma<<<std::min(n, num_sms()), kT2Threads, S.smem, s>>>(P, X, S, list, n, zblk, err);
  return cudaGetLastError();
}

cudaError_t launch_t1_umma(const DevPlan& P, const MixPlan& X, const T1UPlan& U, int sp, const int* qlist, int n,
                           size_t smem, int* work, int* err, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  ++g_t1u_launches;
  const int grid = std::min(n * U.nsplit, num_sms());
  cudaError_t e = cudaMemsetAsync(work, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  t1_kern(sp, U.sub != 0)<<<grid, kThreads, smem, s>>>(P, X, U, qlist, n, work, err);
  return cudaGetLastError();
}

}  // namespace hfx
