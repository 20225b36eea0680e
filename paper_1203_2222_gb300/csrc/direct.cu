// Direct contraction of sectors with a tiny matrix on one side.
//
// Blockwise matrix multiply of Ch. 5, Eq. blockmult, T_j = M_j N_j, for the
// sectors j whose N_j is at most kMaxDirect x kMaxDirect (an MPO or a
// physical leg on the contracted side).  Moving such a sector into matrix
// form and back would cost two extra passes over the large operand for a
// GEMM that is itself a pure stream, so the product is taken on the blocks:
// a work item is one row group of the sector (the blocks of the large
// operand that share the charges of their free legs), its box the free legs,
// its source and destination columns the positions of the contracted and of
// the other operand's free legs inside those blocks.
//
//   apply  C_d[t] = sum_s N(s, d) A_s[t]   (forward, and dA = dC N^T)
//   outer  dN(s, d) += sum_t A_s[t] dC_d[t] (dB = A^T dC), reduced across the
//          warp with butterfly shuffles and added into the zero-filled
//          gradient blocks with atomics
//   both   dA and dB of an outer item from one read of dC (and of A)
//
// Persistent and warp-independent: a warp copies one 512-byte descriptor
// (columns inline) into its shared-memory slot while the previous item runs,
// and streams the box with coalesced loads along its last dim, 64 bytes of
// them a lane and step in flight, in registers.  What bounds it is the
// instructions and round trips around short streams, so: columns are read
// from the descriptor as they are used (few registers, 24 to 32 warps an SM),
// a position's index is formed once for loads and stores, and an item shorter
// than a step takes smaller ones.  Every item form is a function of its own
// (inlined into one another they spilled 1 KB a thread).  Items come longest
// first (plan.cpp) and go to the CTAs in turn.  128 two-site problems of 64 <=
// D <= 1024, 154 MB in and out per step: apply 107 -> 86 us (3.6 TB/s), both
// gradients 255 -> 115 us (4.0 TB/s) against apply and outer launches with two
// cp.async stages in shared memory (with items in the order of the sectors 92
// and 186 us); one FP64 problem of D = 768, latency-bound: 33 -> 28 us.
// Items of one kind run as launches of their own.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "pdl.h"

namespace sym {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
// positions of a step: COLS values each, 64 bytes of them a lane, at most 8
template <typename T, int COLS>
constexpr int kSteps = 64 / (int)sizeof(T) / COLS >= 8   ? 8
                       : 64 / (int)sizeof(T) / COLS >= 4 ? 4
                       : 64 / (int)sizeof(T) / COLS >= 2 ? 2
                                                         : 1;

template <typename T>
__device__ __forceinline__ const T* src_ptr(const BoxPtrs& p, int slot) {
  return static_cast<const T*>(slot == 0 ? p.src[0] : slot == 1 ? p.src[1] : slot == 2 ? p.src[2] : p.src[3]);
}

template <typename T>
__device__ __forceinline__ T* dst_ptr(const BoxPtrs& p, int slot) {
  return static_cast<T*>(slot == DST_OUT ? p.dst[DST_OUT] : slot == DST_DA ? p.dst[DST_DA] : p.dst[DST_DB]);
}

// Box index of position p (last dim fastest): floor(r / n) = umulhi(2r, mag) >> shf.
// ND = the item's number of dims (1..3); one dim needs no division.
template <int ND>
struct DirectShape {
  int n[ND], shf[ND];
  uint32_t mag[ND];
  __device__ __forceinline__ explicit DirectShape(const DirectItem& it) {
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      n[d] = it.dims[d];
      mag[d] = it.mag[d];
      shf[d] = (it.shf >> (8 * d)) & 0xff;
    }
  }
  __device__ __forceinline__ void index(int p, int (&t)[ND]) const {
    int rem = p;
#pragma unroll
    for (int d = ND - 1; d > 0; --d) {
      const int q = (int)(__umulhi((uint32_t)rem << 1, mag[d]) >> shf[d]);
      t[d] = rem - q * n[d];
      rem = q;
    }
    t[0] = rem;
  }
};

// One step of an item: the H positions p0 + lane + 32 h.  Columns are walked
// one by one, each one's offset and strides read from the descriptor in shared
// memory (the barrier keeps the compiler from holding all of them, which
// spilled): column c at box index t is base[off + <t, str>], the relative
// offset below 2^31 (host check).
template <int ND, int H>
struct Positions {
  int t[H][ND];
  __device__ __forceinline__ Positions(const DirectShape<ND>& sh, int p, int last) {
#pragma unroll
    for (int h = 0; h < H; ++h) sh.index(min(p + 32 * h, last), t[h]);
    asm volatile("" ::: "memory");
  }
  __device__ __forceinline__ int off(const int (&str)[ND], int h) const {
    int o = 0;
#pragma unroll
    for (int d = 0; d < ND; ++d) o += t[h][d] * str[d];
    return o;
  }
  template <typename T, int NC>
  __device__ __forceinline__ void load(T (&x)[H][NC], const T* __restrict__ p, const DirectCol* cols, int n) const {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (c < n) {
        const T* __restrict__ b = p + cols[c].off;
        int str[ND];
#pragma unroll
        for (int d = 0; d < ND; ++d) str[d] = cols[c].str[d];
#pragma unroll
        for (int h = 0; h < H; ++h) x[h][c] = __ldg(b + off(str, h));
      } else {
#pragma unroll
        for (int h = 0; h < H; ++h) x[h][c] = T(0);
      }
    }
  }
  // column c of `cols` at the positions: sum_s cf[c * cs + s * ss] x[.][s], in the order of s
  template <typename T, int NX, int NC>
  __device__ __forceinline__ void store(T* __restrict__ p, const DirectCol* cols, int n, const T (&x)[H][NX],
                                        const T* cf, int cs, int ss, int left) const {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (c >= n) break;
      T* __restrict__ b = p + cols[c].off;
      int str[ND];
      T k[NX];
#pragma unroll
      for (int d = 0; d < ND; ++d) str[d] = cols[c].str[d];
#pragma unroll
      for (int i = 0; i < NX; ++i) k[i] = cf[c * cs + i * ss];
#pragma unroll
      for (int h = 0; h < H; ++h) {
        T v = T(0);
#pragma unroll
        for (int i = 0; i < NX; ++i) v = fma(k[i], x[h][i], v);
        if (32 * h <= left) b[off(str, h)] = v;
      }
    }
  }
};

// Steps of H positions a lane as long as they are whole, then of fewer: a small
// item does not pay for the positions it does not have.  step(Positions, u, left).
template <int ND, int H, typename Step>
__device__ __forceinline__ void steps(const DirectShape<ND>& sh, int p, int lane, int last, const Step& step) {
  for (; p + 32 * (H - 1) <= last; p += 32 * H) step(Positions<ND, H>(sh, p + lane, last), last - p - lane);
  if constexpr (H > 1) {
    if (p <= last) steps<ND, H / 2>(sh, p, lane, last, step);
  }
}

// apply: NS source and NQ destination columns (exact counts when the item has
// them, else upper bounds with the actual counts ns <= NS, nq <= NQ)
template <typename T, int ND, int NS, int NQ>
struct ApplyStep {
  const DirectItem& it;
  const T* slot;
  const T* src;
  T* dst;
  int ns, nq;
  template <int H>
  __device__ __forceinline__ void operator()(const Positions<ND, H>& t, int left) const {
    T x[H][NS];
    t.load(x, src, it.src, ns);
    t.template store<T, NS, NQ>(dst, it.dst, nq, x, slot, kMaxDirect, 1, left);
  }
};
template <typename T, int ND, int NS, int NQ>
__device__ __noinline__ void apply_item(const DirectItem& it, const T* __restrict__ slot, const T* __restrict__ src,
                                        T* __restrict__ dst, int lane) {
  const ApplyStep<T, ND, NS, NQ> step{it, slot, src, dst, it.ns, it.nd};
  steps<ND, kSteps<T, NS>>(DirectShape<ND>(it), it.start, lane, it.start + it.count - 1, step);
}

// outer: out(s, d) = sum_t A_s[t] dC_d[t] over the item's positions, scaled
// by kc and added into the destination at koff.  kBoth: also dA_s[t] = sum_d
// N(s, d) dC_d[t], at A's columns in dA, in the order of an apply item of dA.
template <typename T, int ND, int NS, int NQ, bool kBoth>
struct OuterStep {
  const DirectItem& it;
  const T* slot;
  const T* src;
  const T* qsrc;
  T* da;
  int ns, nq;
  T (&acc)[NS][NQ];
  template <int H>
  __device__ __forceinline__ void operator()(const Positions<ND, H>& t, int left) const {
    T a[H][NS], q[H][NQ];
    t.load(a, src, it.src, ns);
    t.load(q, qsrc, it.dst, nq);
#pragma unroll
    for (int h = 0; h < H; ++h) {
      if (32 * h > left) continue;  // positions past the last one repeat it: they add nothing
#pragma unroll
      for (int c = 0; c < NS; ++c)
#pragma unroll
        for (int d = 0; d < NQ; ++d) acc[c][d] = fma(a[h][c], q[h][d], acc[c][d]);
    }
    if (kBoth) t.template store<T, NQ, NS>(da, it.src, ns, q, slot, 1, kMaxDirect, left);
  }
};
template <typename T, int ND, int NS, int NQ, bool kBoth>
__device__ __noinline__ void outer_item(const DirectItem& it, const T* __restrict__ slot, const T* __restrict__ src,
                                        const T* __restrict__ qsrc, T* __restrict__ dst, T* __restrict__ da,
                                        int lane) {
  const int ns = it.ns, nq = it.nd;
  T acc[NS][NQ];
#pragma unroll
  for (int c = 0; c < NS; ++c)
#pragma unroll
    for (int d = 0; d < NQ; ++d) acc[c][d] = T(0);
  const OuterStep<T, ND, NS, NQ, kBoth> step{it, slot, src, qsrc, da, ns, nq, acc};
  steps<ND, kSteps<T, NS + NQ>>(DirectShape<ND>(it), it.start, lane, it.start + it.count - 1, step);
  // butterfly: every lane ends with the warp's sums
#pragma unroll
  for (int c = 0; c < NS; ++c)
#pragma unroll
    for (int d = 0; d < NQ; ++d)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[c][d] += __shfl_xor_sync(0xffffffffu, acc[c][d], o);
  // lane c * NQ + d adds out(c, d)
  const int c0 = lane / NQ, d0 = lane % NQ;
  if (lane < NS * NQ && c0 < ns && d0 < nq) {
    T v = T(0);
#pragma unroll
    for (int c = 0; c < NS; ++c)
#pragma unroll
      for (int d = 0; d < NQ; ++d)
        if (c == c0 && d == d0) v = acc[c][d];
    const int e = d0 * kMaxDirect + c0;
    const double k = it.kc[e];
    if (k != 0.0) atomicAdd(dst + it.koff[e], T(k) * v);
  }
}

// the item's column counts pick an exact variant (the MPO and physical legs
// of a tensor network give 1 or 4 columns per side), else the bounded one
template <typename T, int kOp, int ND, int NS, int NQ>
__device__ __forceinline__ void run_cols(const DirectItem& it, const T* __restrict__ slot, const BoxPtrs& ptrs,
                                         int lane) {
  if constexpr (kOp == kDirectApply)
    apply_item<T, ND, NS, NQ>(it, slot, src_ptr<T>(ptrs, it.slots & 3), dst_ptr<T>(ptrs, (it.slots >> 4) & 7), lane);
  else
    outer_item<T, ND, NS, NQ, kOp == kDirectBoth>(it, slot, src_ptr<T>(ptrs, it.slots & 3),
                                                  src_ptr<T>(ptrs, (it.slots >> 2) & 3),
                                                  dst_ptr<T>(ptrs, (it.slots >> 4) & 7), dst_ptr<T>(ptrs, DST_DA), lane);
}

template <typename T, int kOp, int ND>
__device__ __forceinline__ void run_item(const DirectItem& it, const T* __restrict__ slot, const BoxPtrs& ptrs,
                                         int lane) {
  const int key = ND == 3 ? 0 : it.ns * 8 + it.nd;  // three-dim boxes take the bounded variant only
  if (key == 4 * 8 + 4) run_cols<T, kOp, ND, 4, 4>(it, slot, ptrs, lane);
  else if (key == 1 * 8 + 1) run_cols<T, kOp, ND, 1, 1>(it, slot, ptrs, lane);
  else if (key == 1 * 8 + 4) run_cols<T, kOp, ND, 1, 4>(it, slot, ptrs, lane);
  else if (key == 4 * 8 + 1) run_cols<T, kOp, ND, 4, 1>(it, slot, ptrs, lane);
  else run_cols<T, kOp, ND, kMaxDirect, kMaxDirect>(it, slot, ptrs, lane);
}

// One kernel per item kind, so that each gets the registers of its own loop.
// A warp keeps the next item's descriptor in flight (one 16-byte load per
// lane) while it runs the current one, so an item's set-up costs one round
// trip: the apply coefficients, loaded by one lane each.
template <typename T, int kOp>
__global__ void __launch_bounds__(kThreads, kOp == kDirectApply ? (sizeof(T) == 4 ? 4 : 3) : 3)
    direct_kernel(const DirectItem* __restrict__ items, int nitems, BoxPtrs ptrs) {
  static_assert(sizeof(DirectItem) == 32 * sizeof(int4), "one 16-byte descriptor word per lane");
  __shared__ __align__(16) DirectItem desc[kWarps];
  __shared__ T cfs[kWarps][kMaxDirect * kMaxDirect];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stride = gridDim.x * kWarps;
  int w = warp * gridDim.x + blockIdx.x;  // the longest items, which come first, spread over the CTAs
  int4 next = make_int4(0, 0, 0, 0);
  if (w < nitems) next = __ldg(reinterpret_cast<const int4*>(items + w) + lane);
  pdl_wait();
  pdl_launch_dependents();
  for (; w < nitems; w += stride) {
    __syncwarp();
    reinterpret_cast<int4*>(desc + warp)[lane] = next;
    __syncwarp();
    if (w + stride < nitems) next = __ldg(reinterpret_cast<const int4*>(items + w + stride) + lane);
    const DirectItem& it = desc[warp];
    if (kOp != kDirectOuter && lane < kMaxDirect * kMaxDirect) {  // N(s, d), one lane each
      const double k = it.kc[lane];
      cfs[warp][lane] = k != 0.0 ? T(k) * __ldg(src_ptr<T>(ptrs, 1) + it.koff[lane]) : T(0);
    }
    __syncwarp();
    if (it.ndim == 1)
      run_item<T, kOp, 1>(it, cfs[warp], ptrs, lane);
    else if (it.ndim == 2)
      run_item<T, kOp, 2>(it, cfs[warp], ptrs, lane);
    else
      run_item<T, kOp, 3>(it, cfs[warp], ptrs, lane);
  }
}

template <typename T, int kOp>
int ctas_per_sm() {
  static const int n = [] {
    int v = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, direct_kernel<T, kOp>, kThreads, 0) != cudaSuccess || v < 1)
      v = 1;
    return v;
  }();
  return n;
}

template <typename T, int kOp>
int launch_op(const DirectItem* items, int nitems, const BoxPtrs& ptrs, cudaStream_t s) {
  if (nitems <= 0) return 0;
  const int ctas = std::min((nitems + kWarps - 1) / kWarps, tc_num_sms() * ctas_per_sm<T, kOp>());
  return (int)launch_pdl(direct_kernel<T, kOp>, dim3(ctas), dim3(kThreads), 0, s, items, nitems, ptrs);
}

template <typename T>
int launch_t(int op, const DirectItem* items, int nitems, const BoxPtrs& ptrs, cudaStream_t s) {
  return op == kDirectApply   ? launch_op<T, kDirectApply>(items, nitems, ptrs, s)
         : op == kDirectOuter ? launch_op<T, kDirectOuter>(items, nitems, ptrs, s)
                              : launch_op<T, kDirectBoth>(items, nitems, ptrs, s);
}

}  // namespace

int launch_direct(bool f64, int op, const DirectItem* items, int nitems, const BoxPtrs& ptrs, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  return f64 ? launch_t<double>(op, items, nitems, ptrs, s) : launch_t<float>(op, items, nitems, ptrs, s);
}

}  // namespace sym
