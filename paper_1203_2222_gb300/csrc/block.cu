// Block contraction: a grouped GEMM that reads the operands' blocks and
// writes the result's blocks in place, with no matrix form in between
// (Ch. 5, Eq. blockmult, taken block by block: C_c = sum over the pairs of
// blocks of A and B that meet in c).  Forward, dA and dB all have this form
// with the tensors' roles exchanged, so a contraction is one launch and its
// backward one more.
//
// What bounds it: launches and latency at the small end (a contraction of a
// few thousand flops is one round of dependent loads), the FP32 pipe or, in
// FP64, the two FP64 lanes a clock of an SM at the large end.  The matrix
// form it replaces costs a gather, up to four GEMM launches and a scatter.
//
// A CTA of 128 threads makes one tile (longest tiles first).  The reductions
// of all segments are strung together, so that short segments share a slab of
// KS steps: per slab, KS threads turn their reduction index into the offsets
// of P's and Q's elements (one division per extra dim), and all threads send
// the slab's elements to shared memory with cp.async, kStages - 1 slabs ahead
// of the multiply.  Lanes run along whichever of (row, reduction) is
// contiguous in memory.  FP32 tiles keep a microtile per thread of
// consecutive rows and columns (vector reads; a slab row is padded by one
// vector to keep the transposing writes apart); FP64 tiles stride their
// microtile so that rows and columns past the block's edge are skipped whole
// -- an FP64 multiply-add costs a warp 16 clocks.
// Measured (GB300, the passes of perf/cases.py through the public API, launches
// and host time included; before: the matrix form): two small rank-4 U(1) tensors
// 263 -> 155 us; U(1) MPS step D = 2048 541 -> 366 us, 35 -> 8 launches; SU(2) x
// U(1) MPS step 551 -> 309 us, 32 -> 6 launches; MERA patch 2.04 -> 1.42 ms, 98 ->
// 38; FP64 MPS apply D = 768 543 -> 121 us (tiles small enough for 152 SMs).  The
// U(1) step's block launches take 44 and 71 us forward, 116 and 82 backward, bound
// by the shared-memory pipe (l1tex 75% busy, FP32 multiply-adds a quarter of the
// instructions); the matrix form's launches take 31 and 30, 41 and 50 us on the
// device, so a captured call takes those (plan.cpp).  64 threads with an 8 x 8
// microtile (12 warps an SM) took 104 us a launch instead of 67, a persistent CTA
// with the next tile's descriptors prefetched 69.
// Outputs of at most 8 x 8 with a long reduction (the gradient of a small
// operator, a scalar) take a thread per reduction step instead.
#include <cuda_runtime.h>

#include "kernels.h"
#include "pdl.h"

namespace sym {
namespace {

constexpr int kThreads = kBlkThreads;
constexpr int kStages = 3;   // slabs of the ring
constexpr int kSegCap = 24;  // segments of a tile kept in shared memory (the rest are read from global memory)

__device__ __forceinline__ int div_magic(int a, uint32_t mag, int shf) {
  return (int)(__umulhi((uint32_t)a << 1, mag) >> shf);
}
// copies sizeof(T) bytes, or writes zeros when !live
template <typename T>
__device__ __forceinline__ void cp_elem(T* smem, const T* gmem, bool live) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
  const int n = live ? (int)sizeof(T) : 0;
  if constexpr (sizeof(T) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(s), "l"(gmem), "r"(n) : "memory");
}
__device__ __forceinline__ void cp8(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ int4 box_index(int e, int lim, const int32_t* d, const uint32_t* mag, int shf) {
  int4 t;
  const int q = div_magic(e, mag[1], (shf >> 8) & 0xff);
  t.z = e - q * d[1];
  t.x = div_magic(q, mag[0], shf & 0xff);
  t.y = q - t.x * d[0];
  t.w = e < lim;
  return t;
}

// per reduction step of a slab, where P's and Q's elements are: (offset, the
// three row (column) strides); offset -1 past the end of the reduction
template <int KS>
struct KTable {
  int4 p[KS], q[KS];
};

// A slab row is padded by one 16-byte vector: lanes along the reduction then
// write eight different bank groups, and vectors along the row stay aligned.
template <typename T>
constexpr int kPad = 16 / (int)sizeof(T);
template <typename T, int TM, int TN, int KS>
struct Smem {
  T a[kStages][KS][TM + kPad<T>], b[kStages][KS][TN + kPad<T>];
  KTable<KS> kt[2];
  T cf[4][KS];          // the steps' coefficients (the ring outlives the loads of a slab)
  int4 rt[TM], ct[TN];  // row and column multi-indices of the tile; w = 1 inside the block
};

template <int N>
__device__ __forceinline__ void load_vec(const float* p, float (&v)[N]) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int q = 0; q < N; q += 4) {
      const float4 x = *reinterpret_cast<const float4*>(p + q);
      v[q] = x.x;
      v[q + 1] = x.y;
      v[q + 2] = x.z;
      v[q + 3] = x.w;
    }
  } else if constexpr (N % 2 == 0) {
#pragma unroll
    for (int q = 0; q < N; q += 2) {
      const float2 x = *reinterpret_cast<const float2*>(p + q);
      v[q] = x.x;
      v[q + 1] = x.y;
    }
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = p[q];
  }
}

// Send one operand slab (W x KS, element (i, k) at dst[k][i]) to shared
// memory.  Lanes along k: a thread's step is fixed, its rows vary (their
// multi-indices are read once for all lanes of a row); lanes along i: the
// thread's row is fixed and kept in registers (`own`), the steps vary.  Either
// way an element costs one broadcast read of shared memory.
constexpr int gcd(int a, int b) { return b == 0 ? a : gcd(b, a % b); }
template <int W>
constexpr int kOwn = W / gcd(W, kThreads);  // rows a thread meets when lanes run along the rows
template <typename T, int W, int KS>
__device__ __forceinline__ void load_slab(T (*dst)[W + kPad<T>], const T* __restrict__ src, const int4* st,
                                          const int4* it, const int4 (&own)[kOwn<W>], bool kfast) {
  static_assert(kThreads % KS == 0, "a thread keeps its step");
  constexpr int N = (W * KS + kThreads - 1) / kThreads;
  if (W * KS < kThreads && threadIdx.x >= W * KS) return;
  if (kfast) {
    const int k = threadIdx.x % KS;
    const int4 s = st[k];
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int i = threadIdx.x / KS + u * (kThreads / KS);
      const int4 t = it[i];
      cp_elem(&dst[k][i], src + (s.x + t.x * s.y + t.y * s.z + t.z * s.w), s.x >= 0 && t.w);
    }
  } else {
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int e = threadIdx.x + u * kThreads;
      const int k = e / W;
      const int4 s = st[k], t = own[u % kOwn<W>];
      cp_elem(&dst[k][e % W], src + (s.x + t.x * s.y + t.y * s.z + t.z * s.w), s.x >= 0 && t.w);
    }
  }
}

template <typename T>
__device__ __forceinline__ const T* src_of(const BoxPtrs& p, int slot) {
  return static_cast<const T*>(slot == 0 ? p.src[0] : slot == 1 ? p.src[1] : p.src[2]);
}
template <typename T>
__device__ __forceinline__ T* dst_of(const BoxPtrs& p, int slot) {
  return static_cast<T*>(slot == DST_OUT ? p.dst[DST_OUT] : slot == DST_DA ? p.dst[DST_DA] : p.dst[DST_DB]);
}

// A part of a cut tile: publish this thread's N values in the part's slot and,
// in the CTA that arrives last, replace them by the sum over the parts (in
// part order).  Returns whether this CTA writes the tile.
template <typename T, int N>
__device__ __forceinline__ bool join_parts(const BlkTile& tl, T (&v)[N], T* __restrict__ ws, int* __restrict__ counters,
                                           int* flag) {
  const int part = tl.part & 0xffff, nparts = tl.part >> 16;
  if (nparts <= 1) return true;
  T* slot = ws + (int64_t)(tl.ws + part * N) * kThreads + threadIdx.x;
#pragma unroll
  for (int i = 0; i < N; ++i) __stcg(slot + i * kThreads, v[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *flag = atomicAdd(counters + tl.cnt, 1) == nparts - 1;
  __syncthreads();
  if (!*flag) return false;
  __threadfence();
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = T(0);
  for (int q = 0; q < nparts; ++q) {
    const T* s = ws + (int64_t)(tl.ws + q * N) * kThreads + threadIdx.x;
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] += __ldcg(s + i * kThreads);
  }
  if (threadIdx.x == 0) counters[tl.cnt] = 0;
  return true;
}

template <typename T, int TM, int TN, int KS, int RM, int RN>
__device__ __forceinline__ void block_tile(const BlkTile& tl, const BlkSeg* sseg, const BlkSeg* __restrict__ segs0,
                                           const BoxPtrs& ptrs, void* smem, T* __restrict__ ws,
                                           int* __restrict__ counters, int* flag) {
  static_assert((TM / RM) * (TN / RN) == kThreads, "one microtile per thread");
  Smem<T, TM, TN, KS>& sm = *static_cast<Smem<T, TM, TN, KS>*>(smem);
  constexpr int TX = TN / RN, TY = TM / RM;
  constexpr bool kVec = sizeof(T) == 4;  // consecutive rows and columns per thread (else strided)
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const BlkOut& ob = tl.ob;
  const int kend = min(ob.ktot, tl.s1 * KS), s0 = tl.s0, ns = tl.s1 - tl.s0;
  const BlkSeg* __restrict__ segs = segs0 + ob.seg0;
  const T* __restrict__ P = src_of<T>(ptrs, ob.slots & 3);
  const T* __restrict__ Q = src_of<T>(ptrs, (ob.slots >> 2) & 3);
  const bool pk = (ob.flags & kBlkPk) != 0, qk = (ob.flags & kBlkQk) != 0, cfs = (ob.flags & kBlkCoef) != 0;
  int4 own_r[kOwn<TM>], own_c[kOwn<TN>];
#pragma unroll
  for (int u = 0; u < kOwn<TM>; ++u) {
    const int i = (tid + u * kThreads) % TM;
    own_r[u] = box_index(tl.r0 + i, ob.m, ob.rd, ob.rmag, ob.shf);
    sm.rt[i] = own_r[u];
  }
#pragma unroll
  for (int u = 0; u < kOwn<TN>; ++u) {
    const int i = (tid + u * kThreads) % TN;
    own_c[u] = box_index(tl.c0 + i, ob.n, ob.cd, ob.cmag, ob.shf >> 16);
    sm.ct[i] = own_c[u];
  }

  int sg = 0;  // this thread's segment (it only moves forward)
  auto build = [&](int j) {  // table of slab s0 + j
    if (tid < KS) {
      KTable<KS>& kt = sm.kt[j & 1];
      const int kk = (s0 + j) * KS + tid;
      if (kk < kend) {
        const BlkSeg* s = sg < kSegCap ? sseg + sg : segs + sg;
        while (kk >= s->k0 + s->kn) {
          ++sg;
          s = sg < kSegCap ? sseg + sg : segs + sg;
        }
        const int4 t = box_index(kk - s->k0, 0, s->kd, s->kmag, s->kshf);
        kt.p[tid] = make_int4((int)s->p_off + (t.x * s->pk[0] + t.y * s->pk[1] + t.z * s->pk[2]), s->pr[0], s->pr[1],
                              s->pr[2]);
        kt.q[tid] = make_int4((int)s->q_off + (t.x * s->qk[0] + t.y * s->qk[1] + t.z * s->qk[2]), s->qc[0], s->qc[1],
                              s->qc[2]);
        sm.cf[j & 3][tid] = sizeof(T) == 4 ? T(s->coef_f) : T(s->coef);
      } else {
        kt.p[tid] = kt.q[tid] = make_int4(-1, 0, 0, 0);
        sm.cf[j & 3][tid] = T(0);
      }
    }
  };
  auto issue = [&](int j) {
    const KTable<KS>& kt = sm.kt[j & 1];
    load_slab<T, TM, KS>(sm.a[j % kStages], P, kt.p, sm.rt, own_r, pk);
    load_slab<T, TN, KS>(sm.b[j % kStages], Q, kt.q, sm.ct, own_c, qk);
  };
  T acc[RM][RN];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = T(0);
  const int mlive = ob.m - tl.r0, nlive = ob.n - tl.c0;  // live rows and columns of the tile (may exceed it)
  static_assert(kStages == 3, "the prologue starts two slabs");
  build(0);
  build(1);
  __syncthreads();
  if (ns > 0) issue(0);
  cp_commit();
  if (ns > 1) issue(1);
  cp_commit();
  __syncthreads();
  build(2);
  auto step = [&](int k, const T (*a)[TM + kPad<T>], const T (*b)[TN + kPad<T>], const T* cf) {
    T av[RM], bv[RN];
    if constexpr (kVec) {
      load_vec<RM>(&a[k][ty * RM], av);
      load_vec<RN>(&b[k][tx * RN], bv);
      if (cf) {
        const T c = cf[k];
        if constexpr (RM < RN) {
#pragma unroll
          for (int i = 0; i < RM; ++i) av[i] *= c;
        } else {
#pragma unroll
          for (int j = 0; j < RN; ++j) bv[j] *= c;
        }
      }
#pragma unroll
      for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    } else {
#pragma unroll
      for (int i = 0; i < RM; ++i) av[i] = a[k][ty + TY * i];
#pragma unroll
      for (int j = 0; j < RN; ++j) bv[j] = b[k][tx + TX * j];
      if (cf) {
        const T c = cf[k];
#pragma unroll
        for (int j = 0; j < RN; ++j)
          if (TX * j < nlive) bv[j] *= c;  // as costly as a multiply-add: only what is used
      }
#pragma unroll
      for (int i = 0; i < RM; ++i)
        if (TY * i < mlive)
#pragma unroll
          for (int j = 0; j < RN; ++j)
            if (TX * j < nlive) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
  };
#pragma unroll 1
  for (int s = 0; s < ns; ++s) {
    cp_wait<1>();     // slab s has landed (the newest group may be in flight)
    __syncthreads();  // for every thread; and slab s - 1 is done with
    if (s + 2 < ns) issue(s + 2);
    cp_commit();
    build(s + 3);
    const T(*a)[TM + kPad<T>] = sm.a[s % kStages];
    const T(*b)[TN + kPad<T>] = sm.b[s % kStages];
    const T* cf = cfs ? sm.cf[s & 3] : nullptr;
    const int kl = kend - (s0 + s) * KS;
    if (kl > KS / 2 && !cfs) {  // steps past the end are zeros on both sides
#pragma unroll
      for (int k = 0; k < KS; ++k) step(k, a, b, nullptr);
    } else {
#pragma unroll 1
      for (int k = 0; k < min(kl, KS); k += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) step(k + u, a, b, cf);
    }
  }
  T(&flat)[RM * RN] = reinterpret_cast<T(&)[RM * RN]>(acc);
  if (!join_parts<T, RM * RN>(tl, flat, ws, counters, flag)) return;
  // write the live part of the microtile
  T* __restrict__ o = dst_of<T>(ptrs, (ob.slots >> 4) & 7) + ob.off;
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const int4 r = sm.rt[kVec ? ty * RM + i : ty + TY * i];
    if (!r.w) continue;
    const int ro = r.x * ob.ro[0] + r.y * ob.ro[1] + r.z * ob.ro[2];
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      const int4 c = sm.ct[kVec ? tx * RN + j : tx + TX * j];
      if (c.w) o[ro + c.x * ob.co[0] + c.y * ob.co[1] + c.z * ob.co[2]] = acc[i][j];
    }
  }
}

// Output of at most 8 x 8: thread t takes reduction steps t, t + 128, ... of
// the part and keeps the whole outer-product sum; the CTA then reduces it.
template <typename T>
__device__ __forceinline__ void block_dot(const BlkTile& tl, const BlkSeg* sseg, const BlkSeg* __restrict__ segs0,
                                          const BoxPtrs& ptrs, T (*red)[64], T* __restrict__ ws,
                                          int* __restrict__ counters, int* flag) {
  constexpr int MX = 8;
  const BlkOut& ob = tl.ob;
  const BlkSeg* __restrict__ segs = segs0 + ob.seg0;
  const T* __restrict__ P = src_of<T>(ptrs, ob.slots & 3);
  const T* __restrict__ Q = src_of<T>(ptrs, (ob.slots >> 2) & 3);
  const int m = ob.m, n = ob.n;
  const int kend = min(ob.ktot, tl.s1 * kThreads);
  T acc[MX][MX];
#pragma unroll
  for (int i = 0; i < MX; ++i)
#pragma unroll
    for (int j = 0; j < MX; ++j) acc[i][j] = T(0);
  int sg = 0;
  for (int kk = tl.s0 * kThreads + threadIdx.x; kk < kend; kk += kThreads) {
    const BlkSeg* s = sg < kSegCap ? sseg + sg : segs + sg;
    while (kk >= s->k0 + s->kn) {
      ++sg;
      s = sg < kSegCap ? sseg + sg : segs + sg;
    }
    const int4 t = box_index(kk - s->k0, 0, s->kd, s->kmag, s->kshf);
    const T* __restrict__ p = P + s->p_off + (t.x * s->pk[0] + t.y * s->pk[1] + t.z * s->pk[2]);
    const T* __restrict__ q = Q + s->q_off + (t.x * s->qk[0] + t.y * s->qk[1] + t.z * s->qk[2]);
    T av[MX], bv[MX];
#pragma unroll
    for (int i = 0; i < MX; ++i) {
      av[i] = T(0);
      if (i < m) {
        const int4 r = box_index(i, m, ob.rd, ob.rmag, ob.shf);
        av[i] = __ldg(p + (r.x * s->pr[0] + r.y * s->pr[1] + r.z * s->pr[2]));
      }
      bv[i] = T(0);
      if (i < n) {
        const int4 c = box_index(i, n, ob.cd, ob.cmag, ob.shf >> 16);
        bv[i] = __ldg(q + (c.x * s->qc[0] + c.y * s->qc[1] + c.z * s->qc[2]));
      }
    }
    const T cf = sizeof(T) == 4 ? T(s->coef_f) : T(s->coef);
#pragma unroll
    for (int i = 0; i < MX; ++i) {
      if (i >= m) break;
      av[i] *= cf;
#pragma unroll
      for (int j = 0; j < MX; ++j) {
        if (j >= n) break;
        acc[i][j] = fma(av[i], bv[j], acc[i][j]);
      }
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < MX; ++i) {
    if (i >= m) break;
#pragma unroll
    for (int j = 0; j < MX; ++j) {
      if (j >= n) break;
      T v = acc[i][j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) red[warp][i * MX + j] = v;
    }
  }
  __syncthreads();
  const int i = threadIdx.x / MX, j = threadIdx.x % MX;  // threads 0..63 hold the result
  const bool on = threadIdx.x < MX * MX && i < m && j < n;
  T v[1] = {T(0)};
  if (on)
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) v[0] += red[w][threadIdx.x];
  if (!join_parts<T, 1>(tl, v, ws, counters, flag) || !on) return;
  const int4 r = box_index(i, m, ob.rd, ob.rmag, ob.shf), c = box_index(j, n, ob.cd, ob.cmag, ob.shf >> 16);
  dst_of<T>(ptrs, (ob.slots >> 4) & 7)[ob.off + (r.x * ob.ro[0] + r.y * ob.ro[1] + r.z * ob.ro[2]) +
                                      (c.x * ob.co[0] + c.y * ob.co[1] + c.z * ob.co[2])] = v[0];
}

template <typename T, int kShape>
using SmemOf = Smem<T, blk_rows(sizeof(T) == 8, kShape), blk_cols(sizeof(T) == 8, kShape), blk_slab(sizeof(T) == 8, kShape)>;
template <typename T>
union AnySmem {
  SmemOf<T, BLK_BIG> big;
  SmemOf<T, BLK_MID> mid;
  SmemOf<T, BLK_SMALL> small;
  SmemOf<T, BLK_TALL> tall;
  T red[kThreads / 32][64];
};
template <typename T>
struct CtaSmem {
  AnySmem<T> u;
  BlkTile tile;
  BlkSeg seg[kSegCap];
  int flag;
};

template <typename T>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? 5 : 4)
    block_kernel(const BlkTile* __restrict__ tiles, const BlkSeg* __restrict__ segs, T* __restrict__ ws,
                 int* __restrict__ counters, const BoxPtrs ptrs) {
  __shared__ __align__(16) unsigned char raw[sizeof(CtaSmem<T>)];
  CtaSmem<T>& sm = *reinterpret_cast<CtaSmem<T>*>(raw);
  constexpr bool f64 = sizeof(T) == 8;
  const int tid = threadIdx.x;
  if (tid < (int)sizeof(BlkTile) / 4)
    reinterpret_cast<int*>(&sm.tile)[tid] = __ldg(reinterpret_cast<const int*>(tiles + blockIdx.x) + tid);
  __syncthreads();
  {
    const int words = min(sm.tile.ob.nseg, kSegCap) * (int)(sizeof(BlkSeg) / 8);
    const int64_t* src = reinterpret_cast<const int64_t*>(segs + sm.tile.ob.seg0);
    for (int i = tid; i < words; i += kThreads) reinterpret_cast<int64_t*>(sm.seg)[i] = __ldg(src + i);
  }
  __syncthreads();
  pdl_wait();  // tiles and segments are plan constants; the data is not
  pdl_launch_dependents();
  const BlkTile& tl = sm.tile;
  if (tl.shape == BLK_BIG) {
    if constexpr (f64) block_tile<T, 32, 32, 16, 4, 2>(tl, sm.seg, segs, ptrs, &sm.u, ws, counters, &sm.flag);
    else block_tile<T, 64, 64, 16, 8, 4>(tl, sm.seg, segs, ptrs, &sm.u, ws, counters, &sm.flag);
  } else if (tl.shape == BLK_MID) {
    if constexpr (f64) block_tile<T, 24, 32, 16, 3, 2>(tl, sm.seg, segs, ptrs, &sm.u, ws, counters, &sm.flag);
    else block_tile<T, 48, 64, 16, 6, 4>(tl, sm.seg, segs, ptrs, &sm.u, ws, counters, &sm.flag);
  } else if (tl.shape == BLK_SMALL) {
    if constexpr (f64) block_tile<T, 16, 16, 16, 2, 1>(tl, sm.seg, segs, ptrs, &sm.u, ws, counters, &sm.flag);
    else block_tile<T, 32, 32, 32, 4, 2>(tl, sm.seg, segs, ptrs, &sm.u, ws, counters, &sm.flag);
  } else if (tl.shape == BLK_TALL) {
    if constexpr (f64) block_tile<T, 128, 8, 8, 2, 4>(tl, sm.seg, segs, ptrs, &sm.u, ws, counters, &sm.flag);
    else block_tile<T, 256, 8, 8, 2, 8>(tl, sm.seg, segs, ptrs, &sm.u, ws, counters, &sm.flag);
  } else {
    block_dot<T>(tl, sm.seg, segs, ptrs, sm.u.red, ws, counters, &sm.flag);
  }
}

}  // namespace

int launch_block(bool f64, const BlkTile* tiles, int ntiles, const BlkSeg* segs, void* ws, int* counters,
                 const BoxPtrs& ptrs, void* stream) {
  if (ntiles <= 0) return 0;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const dim3 g(ntiles), b(kThreads);
  return f64 ? (int)launch_pdl(block_kernel<double>, g, b, 0, s, tiles, segs, static_cast<double*>(ws), counters, ptrs)
             : (int)launch_pdl(block_kernel<float>, g, b, 0, s, tiles, segs, static_cast<float*>(ws), counters, ptrs);
}

}  // namespace sym
