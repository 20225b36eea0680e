// Blockwise singular value decomposition of a symmetric tensor seen as a
// matrix (Ch. 5, "Factorization of a matrix", Eq. svd0 and svd1; Ch. 6,
// "Matrix multiplication and factorizations").
//
// The matrix is block diagonal in the fused label x of its row legs, so every
// diagonal block M_x is decomposed on its own.  The blocks are read straight
// from the tensor's blocks (each one a row-major sub-matrix of its M_x,
// because the row legs lead), so there is no separate move into matrix form.
//
// svd_jacobi_kernel: one cluster of 16 CTAs per block, one-sided Jacobi
//   (Hestenes) in FP32.  A = M_x (m >= n) or M_x^T, R x C with R >= C, is
//   copied column-major into the workspace.  A sweep visits every column pair
//   once, in the round-robin order of a tournament; a pair whose columns are
//   not orthogonal to within sqrt(R) ulp is rotated so that they are, and the
//   same rotation is applied to V (V = I at the start).  Blocks with at least
//   64 columns take the pairs by column blocks, a block pair in a CTA's shared
//   memory through its Gram matrix (jacobi_sweeps_gram), others a warp per pair
//   with a cluster barrier between rounds.  V is the starting point of
// svd_av_kernel, svd_gram_kernel, svd_correction_kernel, svd_update_kernel:
//   up to kMaxRefine Newton steps in FP64 (below), each a few products over all
//   blocks that spread over every SM.  A V = W then has orthogonal columns: S =
//   their norms, U = W / S.
// svd_sweep_kernel: FP64 Jacobi sweeps for the blocks that the refinement did
//   not finish: values that decay past what the FP32 sweeps separate (seven decades
//   of singular values, four to five of eigenvalues), rank-deficient blocks of an SVD,
//   clusters.  They are bounded (kMaxSweeps); a block that has not converged by
//   then sets the device error word to SYM_ERR_NUMERIC.
// svd_place_kernel, svd_rank_kernel: norms, and the columns ranked by norm
//   (descending, ties by index) into S and a permutation.
// svd_factor_kernel: one CTA per block writes the kept singular vectors into
//   the blocks of U (row legs, bond) and V (bond, column legs), optionally
//   scaled by S.
//
// Measured (GB300, two-site tensor D = 2048: 41 blocks up to 272 x 272, normal
// entries): execute and factors 19.3 -> 6.6 ms; the two-site density matrix (42
// blocks) 25.6 -> 8.0 ms.  Before, two FP64 sweeps (eig: four) in serial rounds on
// each block's own cluster took 14 ms (20 ms); the refinement takes 2.6 ms, bound
// by FP64 (two multiply-adds a clock of an SM; 70% of it), the FP32 sweeps 3.8
// to 4.7 ms, bound by the latencies of a round.  Where all blocks end in FP64 sweeps,
// the sweeps are what they were: geometric values to 1e-8 61 -> 62 ms.
//
// The same kernels give the blockwise eigendecomposition of a symmetric
// tensor seen as a square matrix (Ch. 5, Eq. spectral, by blocks as the
// thesis prescribes after Eq. svd1; blocks flagged `eig`).  The block is
// replaced by its symmetric part B = (M + M^T)/2.  The FP32 sweeps run on B
// plus a shift that makes it positive definite (then the one-sided Jacobi
// result's V holds the eigenvectors), the refinement on V^T B V itself, whose
// diagonal gives the eigenvalues.  The FP64 sweeps, where a block needs them,
// run on B + sigma I with sigma the Frobenius norm (>= the spectral norm), so
// that |w_j| = lambda_j + sigma.  Eigenvalues are ranked by |lambda|
// descending (ties: the larger lambda, then the column), and U = V, V^T.
// The workspace stays L2-resident for the sizes of tensor-network bonds
// (a 300 x 300 block is 1.4 MB), so the sweeps run from L2, not HBM.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cfloat>
#include <cmath>
#include <cstdlib>
#include <memory>
#include <string>
#include <unordered_map>
#include <vector>

#include "../../include/symtensor.h"
#include "handles.h"
#include "plan.h"
#include "structure.h"

namespace cg = cooperative_groups;

namespace sym {
namespace {

constexpr int kMaxGram = 14;  // columns of a block the FP32 sweeps through Gram matrices take (C <= 448)
constexpr int kSvdThreads = 256;  // FP64 sweeps (128 registers a thread, two CTAs an SM)
// FP32 sweeps: a round has up to 12 column pairs a CTA, one a warp -- with 8
// warps the 9 pairs of a 272-column block took two passes
constexpr int kThreads32 = 384;
// CTAs per diagonal block (16: a cluster size above the portable 8, allowed
// by a function attribute; two CTAs of the kernel fit on an SM)
constexpr int kSvdCluster = 16;
// dynamic shared memory a CTA may take for the FP32 and the FP64 sweeps by
// column blocks, so that two share an SM (with one, 41 blocks take waves of
// clusters: 6.7 against 3.8 ms)
constexpr int kSvdSmem32Max = 112 * 1024;
constexpr int kSvdSmem64Max = 100 * 1024;
constexpr int kMaxSweeps = 64;    // FP64 sweeps before a block counts as not converged
constexpr int kMaxSweeps32 = 40;  // FP32 sweeps (their result only seeds the FP64 ones)
// An FP64 sweep ends the sweeps if all its rotations had a coupling |w_p.w_q| <=
// kBigRotation |w_p| |w_q|, and either none an angle above kBigAngle or none a
// coupling above rounding (16 times the threshold of a rotation).  What it leaves
// is the product of the angles and the couplings, plus the rotations' own residual (the angle
// is formed to FP32 accuracy, about 6e-8 of the coupling): near the FP64
// rounding level, so a further sweep would find nothing to rotate.  The angles
// count on their own: in a cluster of values that are close on the columns'
// scale -- the small eigenvalues of a density matrix, next to the shift -- they
// are of order 1 down to rounding, and carry the couplings of other pairs along.
// With the first condition alone eigenvectors of decaying values (k^-4 to k^-8) had
// residuals |B v - lambda v| of 1e-9 |B|; with all it takes 3 to 6 more sweeps
// there and none on values that are apart.
constexpr double kBigRotation = 1e-8;
constexpr double kBigAngle = 1e-6;
// The FP32 sweeps stop on the coupling alone, at 1e-4: what they leave (1e-8) is
// below FP32's own rounding of the pair products.
constexpr float kBigRotation32 = 1e-4f;

struct SvdBlock {
  int m, n;    // M_x is m x n
  int R, C;    // working matrix A (R x C, R >= C): M_x, or M_x^T when trans
  int trans;   // A = M_x^T (m < n)
  int keep;    // singular vectors the factor kernel writes
  int t0, nt;  // pieces of T
  int u0, nu;  // pieces of U
  int v0, nv;  // pieces of V
  int slot;    // position of the block in ascending x
  int ks;      // first kept singular value of the block in the bond order
  double vscale;  // SU(2): sqrt(2j+1) (the factors carry it, S is divided by it), else 1
  int eig;        // eigendecomposition of the symmetric part (square block) instead of the SVD
  double sgn;     // eig, SU(2) with an incoming row leg: (-1)^{2j}, the sign of the dense block; else 1
  int bw;         // FP32 sweeps by column blocks of bw columns (0: by column pairs)
  int bw64;       // the same for the FP64 sweeps
  int64_t w;   // workspace offset (SvdWork; matrices column-major)
  int64_t s;   // first singular value of the block in S and in the permutation
};

// FP64 refinement steps after the FP32 sweeps before a block goes on to FP64 sweeps
constexpr int kMaxRefine = 5;
// squared norm of a column of sa A V below which an SVD block goes to the FP64
// sweeps: its angles to the large columns are out of FP32's reach
constexpr double kMinNorm2 = 1e-36;
// What the kernels of one call hand on per block (blocks in launch order).
struct SvdState {
  double sa, unsa;  // power-of-two scale of A, and its inverse
  double norm;      // Frobenius norm of sa A (eig: sa sigma)
  unsigned xmax[kMaxRefine];  // bits of the largest squared column norm of a step's correction X (FP32)
  int nulls[kMaxRefine];      // SVD: a step left pairs of columns at the rounding level alone
  int done;         // refinement step after which the block counts as converged (0: not, -1: given up)
};
// One 32 x 32 tile of a refinement product; kind 0: W or V^T W, 1: V^T V or the other factor (see the kernels)
struct SvdTile {
  int block, i0, j0, kind;
};

// The parts of a block's workspace.
struct SvdWork {
  double *W, *V, *nrm, *Ss, *A, *G, *E;
  float *W32, *V32, *X, *F0, *F1;
  __host__ __device__ static int64_t elems(int64_t R, int64_t C) {
    const int64_t rc = R * C, cc = C * C;
    return 2 * rc + 3 * cc + 2 * C + (rc + 4 * cc + 1) / 2 + 1;
  }
  __device__ SvdWork(double* w, int64_t R, int64_t C) {
    const int64_t rc = R * C, cc = C * C;
    W = w;  // the factor kernel reads W, V, the norms and Ss at these places
    V = W + rc;
    nrm = V + cc;
    Ss = nrm + C;
    A = Ss + C;
    G = A + rc;
    E = G + cc;
    W32 = reinterpret_cast<float*>(E + cc);
    V32 = W32 + rc;
    X = V32 + cc;
    F0 = X + cc;
    F1 = F0 + cc;
  }
};

// A tensor block inside its M_x: rows r0.., columns c0.. (row-major, rows x cols).
struct SvdPiece {
  int64_t off;
  int r0, c0, rows, cols;
};

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
  // xor butterfly: every lane ends with the same sum (each step adds the same
  // two values on both partners)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The Jacobi angle of a column pair (p, q) with a = |w_p|^2, bb = |w_q|^2,
// g = w_p.w_q: if the pair is not orthogonal to within tol, the rotation by
// t = tan(theta), the smaller root of t^2 + 2 zeta t - 1 = 0 with
// zeta = (bb - a) / (2 g), makes it so.  Every lane takes the same decision
// (identical butterfly sums).
template <typename T>
struct JacobiArith;

// Approximate root of x (of 0 for x < 0, where a rotated Gram matrix's diagonal can end up).
__device__ __forceinline__ float sqrt_approx(float x) {
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(fmaxf(x, 0.0f)));
  return x;
}
// tan(theta) of a pair in FP32, d = bb - a and h = 2 g: 1 / (zeta + sign(zeta)
// sqrt(zeta^2 + 1)), zeta = d / h.  Only ratios are squared: the squares of d and
// h underflow for columns below 1e-10 of max |A| (equal ones, d = 0, then made
// t = h / 0).  h is normal (kMinCoupling).
__device__ __forceinline__ float tangent(float d, float h) {
  const float zeta = __fdividef(d, h), z = fabsf(zeta);
  return copysignf(__fdividef(1.0f, z + sqrt_approx(fmaf(z, z, 1.0f))), zeta);  // 0 where z^2 is infinite
}
constexpr float kMinCoupling = FLT_MIN;  // |w_p.w_q| below this is underflow, not an angle

template <>
struct JacobiArith<float> {
  // the FP32 sweeps only choose a starting point: approximate roots and quotients
  // |w_p| |w_q| (the product of the squared norms underflows before they do; with
  // approximate roots here the pair loop spills twice as much: 7% at D = 96)
  static __device__ __forceinline__ float norms(float a, float bb) { return sqrtf(a) * sqrtf(bb); }
  static __device__ __forceinline__ bool angle(float a, float bb, float g, float sab, float tol, float& c,
                                               float& s) {
    if (!(fabsf(g) > tol * sab && fabsf(g) > kMinCoupling)) return false;
    const float t = tangent(bb - a, 2.0f * g);
    c = rsqrtf(fmaf(t, t, 1.0f));
    s = c * t;
    return true;
  }
};

template <>
struct JacobiArith<double> {
  static __device__ __forceinline__ double norms(double a, double bb) { return sqrt(a * bb); }
  // The angle itself needs only FP32 accuracy: an inexact angle is still an
  // exact rotation (c^2 + s^2 = 1 to FP64 precision), it just leaves the
  // pair slightly non-orthogonal for the next sweep.  So t = sign(d) h /
  // (|d| + sqrt(d^2 + h^2)) (d = bb - a, h = 2 g; the same root) is formed in
  // FP32 after scaling d and h by a power of two, and c = (1 + t^2)^(-1/2)
  // by two Newton steps in FP64 from the FP32 estimate -- GB300's FP64 units
  // are few, and FP64 square roots and divisions cost many of their cycles.
  static __device__ __forceinline__ bool angle(double a, double bb, double g, double sab, double tol, double& c,
                                               double& s) {
    if (!(fabs(g) > tol * sab)) return false;
    const double d = bb - a, h = 2.0 * g;
    const double m = fmax(fabs(d), fabs(h));
    const int ex = (__double2hiint(m) >> 20) & 0x7ff;  // biased exponent of m
    float tf = 0.0f;
    if (ex > 0 && ex < 2046) {
      const double sc = __hiloint2double((2046 - ex) << 20, 0);  // 2^(1023 - e): m * sc in [1, 2)
      const float df = (float)(d * sc), hf = (float)(h * sc);
      tf = copysignf(1.0f, df) * hf / (fabsf(df) + sqrtf(fmaf(df, df, hf * hf)));
    }
    double t;
    if (fabsf(tf) >= FLT_MIN && isfinite(tf)) {
      t = (double)tf;
    } else {  // out of FP32's reach (a subnormal tf has few digits: no sweep would end): the angle in FP64
      const double zeta = d / h;
      t = fabs(zeta) > 1e150 ? 0.5 / zeta : copysign(1.0, zeta) / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0)));
    }
    const double x = fma(t, t, 1.0);
    double y = (double)rsqrtf((float)x);
    y = y * fma(-0.5 * x * y, y, 1.5);  // Newton steps for x^(-1/2): y (3 - x y^2) / 2
    y = y * fma(-0.5 * x * y, y, 1.5);
    c = y;
    s = y * t;
    return true;
  }
};

// What a rotation says about convergence (bits; or'ed over a sweep): kRotated, kBig
// (another sweep has to follow), and in FP64 kAngle, kCoupling (another one if the
// sweep has seen both).
constexpr int kRotated = 1, kBig = 2, kAngle = 4, kCoupling = 8;
template <typename T>
__device__ __forceinline__ int rotated(T g, T sab, T sn, T tol, T big) {
  int r = kRotated;
  if (fabs(g) > big * sab) r |= kBig;
  if constexpr (sizeof(T) == 8) {
    if (fabs(sn) > kBigAngle) r |= kAngle;
    if (fabs(g) > T(16) * tol * sab) r |= kCoupling;
  }
  return r;
}
// what the CTA's threads have seen
template <typename T>
__device__ __forceinline__ int seen_by_all(int seen) {
  int f = (__syncthreads_or(seen & kRotated) ? kRotated : 0) | (__syncthreads_or(seen & kBig) ? kBig : 0);
  if constexpr (sizeof(T) == 8)
    f |= (__syncthreads_or(seen & kAngle) ? kAngle : 0) | (__syncthreads_or(seen & kCoupling) ? kCoupling : 0);
  return f;
}
__device__ __forceinline__ bool sweeps_done(int seen) {
  return !(seen & kBig) && (seen & (kAngle | kCoupling)) != (kAngle | kCoupling);
}

// Rotate one column pair (p, q) of W (length R) and V (length C) if needed.
// NR rows per lane held in registers (R <= 32 NR); V's columns are loaded
// with W's, so a pair costs one round trip to L2.
template <typename T, int NR>
// With na, nb (the pair's squared column norms, carried as in
// rotate_pair_smem below) one dot product a pair instead of three.
__device__ __forceinline__ int rotate_pair(T* wp, T* wq, T* vp, T* vq, T* na, T* nb, int R, int C, int lane, T tol,
                                           T big) {
  T xw[NR], yw[NR], xv[NR], yv[NR];
  T a = 0, bb = 0;
  if (na) {
    a = __ldcg(na);
    bb = __ldcg(nb);
  }
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int i = lane + 32 * u;
    xw[u] = i < R ? __ldcg(wp + i) : T(0);
    yw[u] = i < R ? __ldcg(wq + i) : T(0);
    xv[u] = i < C ? __ldcg(vp + i) : T(0);
    yv[u] = i < C ? __ldcg(vq + i) : T(0);
  }
  T g = 0;
  if (!na) {
#pragma unroll
    for (int u = 0; u < NR; ++u) {
      a = fma(xw[u], xw[u], a);
      bb = fma(yw[u], yw[u], bb);
    }
    a = warp_sum(a);
    bb = warp_sum(bb);
  }
#pragma unroll
  for (int u = 0; u < NR; ++u) g = fma(xw[u], yw[u], g);
  g = warp_sum(g);
  const T sab = JacobiArith<T>::norms(a, bb);
  T c, s;
  if (!JacobiArith<T>::angle(a, bb, g, sab, tol, c, s)) return 0;
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int i = lane + 32 * u;
    if (i < R) {
      __stcg(wp + i, c * xw[u] - s * yw[u]);
      __stcg(wq + i, s * xw[u] + c * yw[u]);
    }
    if (i < C) {
      __stcg(vp + i, c * xv[u] - s * yv[u]);
      __stcg(vq + i, s * xv[u] + c * yv[u]);
    }
  }
  if (na && lane == 0) {
    const T cs2g = T(2) * c * s * g, cc = c * c, ss = s * s;
    __stcg(na, fma(cc, a, fma(ss, bb, -cs2g)));
    __stcg(nb, fma(ss, a, fma(cc, bb, cs2g)));
  }
  return rotated(g, sab, s, tol, big);
}

// Any R: the columns streamed twice (products, then the rotation).
template <typename T>
__device__ __noinline__ int rotate_pair_stream(T* wp, T* wq, T* vp, T* vq, int R, int C, int lane, T tol, T big) {
  T a = 0, bb = 0, g = 0;
  for (int i = lane; i < R; i += 32) {
    const T x = __ldcg(wp + i), y = __ldcg(wq + i);
    a = fma(x, x, a);
    bb = fma(y, y, bb);
    g = fma(x, y, g);
  }
  a = warp_sum(a);
  bb = warp_sum(bb);
  g = warp_sum(g);
  const T sab = JacobiArith<T>::norms(a, bb);
  T c, s;
  if (!JacobiArith<T>::angle(a, bb, g, sab, tol, c, s)) return 0;
  for (int i = lane; i < R; i += 32) {
    const T x = __ldcg(wp + i), y = __ldcg(wq + i);
    __stcg(wp + i, c * x - s * y);
    __stcg(wq + i, s * x + c * y);
  }
  for (int i = lane; i < C; i += 32) {
    const T x = __ldcg(vp + i), y = __ldcg(vq + i);
    __stcg(vp + i, c * x - s * y);
    __stcg(vq + i, s * x + c * y);
  }
  return rotated(g, sab, s, tol, big);
}

// Per-cluster state of the sweeps (shared memory of every CTA; rank 0's
// flags are the cluster's).
struct SweepCtl {
  int flag[2];
  int any;
};

// Sweeps of one-sided Jacobi on (W, V), at most max_sweeps; returns the
// sweeps taken, conv = the last sweep rotated nothing.  The C/2 pairs of a
// round (tournament order, an odd C playing against a bye) go to the
// cluster's warps; cluster barriers separate the rounds.
template <typename T, int NT>
__device__ int jacobi_sweeps(T* W, T* V, T* nrm2, int R, int C, int max_sweeps, T tol, cg::cluster_group& cluster,
                             SweepCtl* ctl, int* flag0, int crank, int cw, int lane, int& gsweep,
                             unsigned long long& myrot, bool& conv, T big_tol) {
  constexpr int kCW = kSvdCluster * (NT / 32);
  const int Ce = C + (C & 1);
  const int rpl = (R + 31) / 32;
  const int nr = rpl <= 1 ? 1 : rpl <= 2 ? 2 : rpl <= 4 ? 4 : rpl <= 8 ? 8 : rpl <= 9 ? 9 : rpl <= 12 ? 12 : 0;
  int sweeps = 0;
  conv = C < 2;
  while (!conv && sweeps < max_sweeps) {
    ++sweeps;
    const int gs = ++gsweep;  // sweeps so far over both precisions (same in every thread): picks the flag
    int seen = 0;
    if (nrm2 && nr) {  // the squared column norms, exact at the sweep's start, carried by the rotations
      for (int j = cw; j < C; j += kCW) {
        const T* wj = W + (int64_t)j * R;
        T a = 0;
        for (int i = lane; i < R; i += 32) {
          const T x = __ldcg(wj + i);
          a = fma(x, x, a);
        }
        a = warp_sum(a);
        if (lane == 0) __stcg(nrm2 + j, a);
      }
      cluster.sync();
    }
    T* const carry = nr ? nrm2 : nullptr;
    for (int r = 0; r < Ce - 1; ++r) {
      for (int k = cw; k < Ce / 2; k += kCW) {
        int p = k == 0 ? r : (r + k) % (Ce - 1);
        int q = k == 0 ? Ce - 1 : (r - k + Ce - 1) % (Ce - 1);
        if (p > q) {
          const int t = p;
          p = q;
          q = t;
        }
        if (q >= C) continue;
        T* wp = W + (int64_t)p * R;
        T* wq = W + (int64_t)q * R;
        T* vp = V + (int64_t)p * C;
        T* vq = V + (int64_t)q * C;
        int rot;
        T* na = carry ? carry + p : nullptr;
        T* nb = carry ? carry + q : nullptr;
        switch (nr) {
          case 1: rot = rotate_pair<T, 1>(wp, wq, vp, vq, na, nb, R, C, lane, tol, big_tol); break;
          case 2: rot = rotate_pair<T, 2>(wp, wq, vp, vq, na, nb, R, C, lane, tol, big_tol); break;
          case 4: rot = rotate_pair<T, 4>(wp, wq, vp, vq, na, nb, R, C, lane, tol, big_tol); break;
          case 8: rot = rotate_pair<T, 8>(wp, wq, vp, vq, na, nb, R, C, lane, tol, big_tol); break;
          case 9: rot = rotate_pair<T, 9>(wp, wq, vp, vq, na, nb, R, C, lane, tol, big_tol); break;
          case 12: rot = rotate_pair<T, 12>(wp, wq, vp, vq, na, nb, R, C, lane, tol, big_tol); break;
          default: rot = rotate_pair_stream<T>(wp, wq, vp, vq, R, C, lane, tol, big_tol); break;
        }
        seen |= rot;
        myrot += rot != 0;
      }
      cluster.sync();  // the next round's pairs read columns this round wrote
    }
    // did any warp of the cluster rotate?  flags alternate between sweeps, so
    // the one read now is never the one being cleared for the next sweep
    const int f = seen_by_all<T>(seen);
    if (f && threadIdx.x == 0) atomicOr(flag0 + (gs & 1), f);
    cluster.sync();
    if (threadIdx.x == 0) {
      ctl->any = flag0[gs & 1];
      if (crank == 0) ctl->flag[(gs + 1) & 1] = 0;
    }
    __syncthreads();
    conv = sweeps_done(ctl->any);
    __syncthreads();  // any and gsweep are rewritten by the next sweep
  }
  return sweeps;
}

// Rotate one column pair of W (length R) and V (length C) held in shared
// memory; NR rows per lane.  The squared column norms *na, *nb are carried
// from rotation to rotation (recomputed at every sweep's start), so a pair
// costs one dot product (w_p . w_q), not three; the rotation updates them
// exactly as it rotates the columns: |w_p'|^2 = c^2 a - 2 c s g + s^2 b,
// |w_q'|^2 = s^2 a + 2 c s g + c^2 b.  Returns 0 (no rotation)
// or what `rotated` says of it.
template <typename T, int NR>
__device__ __forceinline__ int rotate_pair_smem(T* wp, T* wq, T* vp, T* vq, T* na, T* nb, int R, int C, int lane,
                                                T tol, T big) {
  T xw[NR], yw[NR];
  T g = 0;
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int i = lane + 32 * u;
    xw[u] = i < R ? wp[i] : T(0);
    yw[u] = i < R ? wq[i] : T(0);
    g = fma(xw[u], yw[u], g);
  }
  g = warp_sum(g);
  const T a = *na, bb = *nb;
  const T sab = JacobiArith<T>::norms(a, bb);
  T c, sn;
  if (!JacobiArith<T>::angle(a, bb, g, sab, tol, c, sn)) return 0;
#pragma unroll
  for (int u = 0; u < NR; ++u) {
    const int i = lane + 32 * u;
    if (i < R) {
      wp[i] = c * xw[u] - sn * yw[u];
      wq[i] = sn * xw[u] + c * yw[u];
    }
    if (i < C) {
      const T x = vp[i], y = vq[i];
      vp[i] = c * x - sn * y;
      vq[i] = sn * x + c * y;
    }
  }
  const T cs2g = T(2) * c * sn * g, cc = c * c, ss = sn * sn;
  __syncwarp();  // every lane has read the old norms
  if (lane == 0) {
    *na = fma(cc, a, fma(ss, bb, -cs2g));
    *nb = fma(ss, a, fma(cc, bb, cs2g));
  }
  return rotated(g, sab, sn, tol, big);
}

// FP64 sweeps by column blocks: the C columns form kColBlocks blocks of bw
// (the last ones ragged or empty), and a sweep is the tournament over the
// blocks (kColBlocks - 1 rounds of kSvdCluster disjoint block pairs).  In a
// round, CTA k of the cluster takes block pair k -- the columns of W and V
// -- into its shared memory, rotates every cross pair (p in P, q in Q; in
// the first round also the pairs inside P and inside Q) in bw inner rounds
// of disjoint pairs separated by CTA barriers, and writes the columns back;
// a cluster barrier separates the rounds.  Every column pair is visited once
// a sweep, as in the order by pairs, but a sweep needs kColBlocks - 1 cluster
// barriers instead of C - 1, and the pairs' columns come from shared memory.
constexpr int kColBlocks = 2 * kSvdCluster;
// n contiguous values between L2 and shared memory, eight loads in flight a thread
template <int NT, typename T>
__device__ __forceinline__ void copy_in(T* dst, const T* src, int n) {
  int i = threadIdx.x;
  for (; i + 7 * NT < n; i += 8 * NT) {
    T x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = __ldcg(src + i + u * NT);
#pragma unroll
    for (int u = 0; u < 8; ++u) dst[i + u * NT] = x[u];
  }
#pragma unroll 4
  for (; i < n; i += NT) dst[i] = __ldcg(src + i);
}
template <int NT, typename T>
__device__ __forceinline__ void copy_out(T* dst, const T* src, int n) {
#pragma unroll 8
  for (int i = threadIdx.x; i < n; i += NT) __stcg(dst + i, src[i]);
}
template <typename T, int NR, int NT>
__device__ int jacobi_sweeps_blocked(T* W, T* V, T* nrm2, int R, int C, int bw, int max_sweeps, T tol,
                                     cg::cluster_group& cluster, SweepCtl* ctl, int* flag0, int crank, int lane,
                                     int& gsweep, unsigned long long& myrot, bool& conv, T big_tol, T* sm) {
  const int warp = threadIdx.x >> 5;
  constexpr int kWarps = NT / 32, kCW = kSvdCluster * kWarps;
  const int cw = crank * kWarps + warp;
  T* Wp = sm;  // bw columns of R, then Q's, then V's columns of P and Q (C each), then their squared norms
  T* Wq = Wp + (int64_t)bw * R;
  T* Vp = Wq + (int64_t)bw * R;
  T* Vq = Vp + (int64_t)bw * C;
  T* Np = Vq + (int64_t)bw * C;
  T* Nq = Np + bw;
  const int bwe = bw + (bw & 1);  // a block's own tournament: bwe - 1 rounds of bwe / 2 pairs
  int sweeps = 0;
  conv = C < 2;
  while (!conv && sweeps < max_sweeps) {
    ++sweeps;
    const int gs = ++gsweep;
    int seen = 0;
    for (int j = cw; j < C; j += kCW) {  // the squared column norms, exact at the sweep's start
      const T* wj = W + (int64_t)j * R;
      T a = 0;
      for (int i = lane; i < R; i += 32) {
        const T x = __ldcg(wj + i);
        a = fma(x, x, a);
      }
      a = warp_sum(a);
      if (lane == 0) __stcg(nrm2 + j, a);
    }
    cluster.sync();
    auto rot = [&](T* wp, T* wq, T* vp, T* vq, T* na, T* nb) {
      const int r = rotate_pair_smem<T, NR>(wp, wq, vp, vq, na, nb, R, C, lane, tol, big_tol);
      seen |= r;
      myrot += r != 0;
    };
    for (int r = 0; r < kColBlocks - 1; ++r) {
      const int k = crank;
      const int P = k == 0 ? r : (r + k) % (kColBlocks - 1);
      const int Q = k == 0 ? kColBlocks - 1 : (r - k + kColBlocks - 1) % (kColBlocks - 1);
      const int p0 = P * bw, np = max(0, min(bw, C - p0));
      const int q0 = Q * bw, nq = max(0, min(bw, C - q0));
      // the two blocks' columns are contiguous in the column-major W and V
      copy_in<NT>(Wp, W + (int64_t)p0 * R, np * R);
      copy_in<NT>(Wq, W + (int64_t)q0 * R, nq * R);
      copy_in<NT>(Vp, V + (int64_t)p0 * C, np * C);
      copy_in<NT>(Vq, V + (int64_t)q0 * C, nq * C);
      copy_in<NT>(Np, nrm2 + p0, np);
      copy_in<NT>(Nq, nrm2 + q0, nq);
      __syncthreads();
      if (r == 0) {  // the pairs inside P and inside Q: each block's own tournament, side by side
        for (int ir = 0; ir < bwe - 1; ++ir) {
          for (int t = warp; t < bwe; t += kWarps) {
            const int side = t < bwe / 2 ? 0 : 1, kk = side ? t - bwe / 2 : t;
            int a = kk == 0 ? ir : (ir + kk) % (bwe - 1);
            int c = kk == 0 ? bwe - 1 : (ir - kk + bwe - 1) % (bwe - 1);
            const int n = side ? nq : np;
            if (a < n && c < n) {
              T* w0 = side ? Wq : Wp;
              T* v0 = side ? Vq : Vp;
              T* n0 = side ? Nq : Np;
              rot(w0 + (int64_t)a * R, w0 + (int64_t)c * R, v0 + (int64_t)a * C, v0 + (int64_t)c * C, n0 + a, n0 + c);
            }
          }
          __syncthreads();
        }
      }
      for (int ir = 0; ir < bw; ++ir) {  // the cross pairs (i, (i + ir) mod bw)
        for (int i = warp; i < bw; i += kWarps) {
          const int j = (i + ir) % bw;
          if (i < np && j < nq)
            rot(Wp + (int64_t)i * R, Wq + (int64_t)j * R, Vp + (int64_t)i * C, Vq + (int64_t)j * C, Np + i, Nq + j);
        }
        __syncthreads();
      }
      copy_out<NT>(W + (int64_t)p0 * R, Wp, np * R);
      copy_out<NT>(W + (int64_t)q0 * R, Wq, nq * R);
      copy_out<NT>(V + (int64_t)p0 * C, Vp, np * C);
      copy_out<NT>(V + (int64_t)q0 * C, Vq, nq * C);
      copy_out<NT>(nrm2 + p0, Np, np);
      copy_out<NT>(nrm2 + q0, Nq, nq);
      cluster.sync();  // the next round reads columns this round wrote, on other CTAs
    }
    const int f = seen_by_all<T>(seen);
    if (f && threadIdx.x == 0) atomicOr(flag0 + (gs & 1), f);
    cluster.sync();
    if (threadIdx.x == 0) {
      ctl->any = flag0[gs & 1];
      if (crank == 0) ctl->flag[(gs + 1) & 1] = 0;
    }
    __syncthreads();
    conv = sweeps_done(ctl->any);
    __syncthreads();
  }
  return sweeps;
}

// FP32 sweeps by column blocks through Gram matrices.  The order of the pairs
// is that of jacobi_sweeps_blocked (a CTA takes a block pair, N = 2 BW columns
// or fewer, a round), but the rotations of a round act on the N x N Gram
// matrix of the block pair's W columns and are collected in Q, which then
// multiplies the columns of W and V once: a pair costs a few operations on
// shared values instead of a pass over its columns in shared memory, and a
// set of disjoint pairs one barrier.  The starting point needs no more than
// that: rotated Gram entries carry FP32's rounding relative to their columns'
// norms, and every round forms them afresh.  The FP32 kernel on the blocks of
// a U(1) two-site tensor of D = 2048 took 4.98 ms with the columns rotated a pair a warp
// (a pass over both columns in shared memory a pair) and takes 3.78 ms; on the
// density matrix of the eigendecomposition 5.82 and 4.69 ms.  A round is bound
// by latencies: 1.2-2.4 us for the columns from L2, 1.6 the Gram matrix, 3 the
// nine sets of rotations, 2-4 the product, 1.2 the cluster's barrier.
template <int BW>
struct GramSmem {
  static constexpr int N = 2 * BW, GP = N + 1, QP = (N + 3) / 4 * 4;
};
// W columns are gram_pitch apart: eight rows of four column pairs, what a warp
// reads for the Gram matrix, fall on different banks
__host__ __device__ inline int gram_pitch(int R) { return (R + 3) / 8 * 8 + 4; }
__host__ __device__ inline int64_t gram_floats(int R, int C, int bw) {
  const int64_t n = 2 * bw, qp = (n + 3) / 4 * 4;
  return n * gram_pitch(R) + n * qp + 2 * n * (n + 1) + n * C;
}
// The angles of a set are a chain of latencies, so what is squared there is kept
// in range by constants rather than by the ratio d / h (two-site tensor of D =
// 2048, six inputs: 6.62 -> 6.57 ms an execute; with squares out of range 6.52):
// squared norms are below 2^21 (max |A| < 2), so 2^40 d, 2^40 h and 2^60 a b have
// finite squares, and a coupling of at least kGramMinCoupling gives normal ones.
// Smaller couplings (columns below 1e-14 of max |A|) are left to FP64.
constexpr float kGramScale = 1099511627776.0f, kGramScaleAb = 1152921504606846976.0f, kGramRoot = 1073741824.0f;
constexpr float kGramMinCoupling = 1e-28f;
template <int BW>
__device__ int jacobi_sweeps_gram(float* W, float* V, int R, int C, int bw, int max_sweeps, float tol,
                                  cg::cluster_group& cluster, SweepCtl* ctl, int* flag0, int crank, int lane,
                                  int& gsweep, unsigned long long& myrot, bool& conv, float big_tol, float* sm) {
  using GS = GramSmem<BW>;
  constexpr int N = GS::N, GP = GS::GP, QP = GS::QP, NT = kThreads32, NW = NT / 32;
  const int RP = gram_pitch(R);
  float* Ws = sm;
  float* Qt = Ws + (size_t)N * RP;  // Q transposed: row j holds column j's coefficients (RP, N QP multiples of 4)
  float* G0 = Qt + N * QP;
  float* Vs = G0 + 2 * N * GP;
  // warps 0 .. GW-1 rotate the Gram matrix, GW .. GW+QW-1 Q
  constexpr int GW = (BW * BW + 31) / 32, QW = (BW * QP / 4 + 31) / 32;
  static_assert(GW + QW <= NW, "threads of a set");
  static_assert(QP % 4 == 0 && (N * QP) % 4 == 0, "Qt's rows and what follows start on 16 bytes (as does N * gram_pitch)");
  const int tid = threadIdx.x, warp = tid >> 5;
  const int gx = tid / BW, gy = tid % BW;
  const float tols = tol / kGramRoot, bigs = big_tol / kGramRoot;
  const int qx = tid < 32 * GW ? BW : (tid - 32 * GW) / (QP / 4), qy = tid < 32 * GW ? 0 : (tid - 32 * GW) % (QP / 4);
  int sweeps = 0;
  conv = C < 2;
  while (!conv && sweeps < max_sweeps) {
    ++sweeps;
    const int gs = ++gsweep;
    int did = 0, big = 0;
    for (int r = 0; r < kColBlocks - 1; ++r) {
      const int k = crank;
      const int P = k == 0 ? r : (r + k) % (kColBlocks - 1);
      const int Q = k == 0 ? kColBlocks - 1 : (r - k + kColBlocks - 1) % (kColBlocks - 1);
      const int p0 = P * bw, np = max(0, min(bw, C - p0));
      const int q0 = Q * bw, nq = max(0, min(bw, C - q0));
      if (np + nq >= 2) {
        // columns of W and V (absent ones: zeros, which nothing rotates)
        for (int c = warp; c < N; c += NW) {
          const int n = c < BW ? np : nq, d = c < BW ? c : c - BW;
          const int64_t col = (c < BW ? p0 : q0) + d;
          const float *w = W + col * R, *v = V + col * C;
          if (d < n) {
            float x[12], y[12];
            for (int i = lane; i < max(R, C); i += 384) {
#pragma unroll
              for (int u = 0; u < 12; ++u) {
                x[u] = i + 32 * u < R ? __ldcg(w + i + 32 * u) : 0.0f;
                y[u] = i + 32 * u < C ? __ldcg(v + i + 32 * u) : 0.0f;
              }
#pragma unroll
              for (int u = 0; u < 12; ++u) {
                if (i + 32 * u < R) Ws[c * RP + i + 32 * u] = x[u];
                if (i + 32 * u < C) Vs[c * C + i + 32 * u] = y[u];
              }
            }
          } else {
            for (int i = lane; i < R; i += 32) Ws[c * RP + i] = 0.0f;
            for (int i = lane; i < C; i += 32) Vs[c * C + i] = 0.0f;
          }
        }
        for (int i = tid; i < N * QP; i += NT) Qt[i] = i / QP == i % QP ? 1.0f : 0.0f;
        __syncthreads();
        // Gram matrix: eight lanes per 2 x 2 tile of its upper triangle
        for (int t = tid >> 3; t < (BW * (BW + 1) / 2 + 3) / 4 * 4; t += NT / 8) {
          int ti = 0, rest = min(t, BW * (BW + 1) / 2 - 1);
          while (rest >= BW - ti) rest -= BW - ti, ++ti;
          const int i0 = 2 * ti, j0 = 2 * (ti + rest);
          const float *a = Ws + i0 * RP, *b = Ws + j0 * RP;
          float g[4] = {};
#pragma unroll 4
          for (int row = lane & 7; row < R; row += 8) {
            const float a0 = a[row], a1 = a[row + RP], b0 = b[row], b1 = b[row + RP];
            g[0] = fmaf(a0, b0, g[0]);
            g[1] = fmaf(a0, b1, g[1]);
            g[2] = fmaf(a1, b0, g[2]);
            g[3] = fmaf(a1, b1, g[3]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) g[u] += __shfl_xor_sync(0xffffffffu, g[u], o);
          }
          if ((lane & 7) < 4) {
            const int u = lane & 7, x = i0 + (u >> 1), y = j0 + (u & 1);
            const float v = u == 0 ? g[0] : u == 1 ? g[1] : u == 2 ? g[2] : g[3];
            G0[x * GP + y] = v;
            G0[y * GP + x] = v;
          }
        }
        __syncthreads();
        // Round 0: every pair of the N columns (a tournament); later rounds:
        // the cross pairs.  Every thread forms the angles it needs from the
        // old Gram matrix and writes the new one: one barrier a set.
        const int inner = r == 0 ? N - 1 : BW;
        int rotated = 0;
        for (int ir = 0; ir < inner && tid < 32 * (GW + QW); ++ir) {
          const float* G = G0 + (ir & 1) * N * GP;
          float* H = G0 + (~ir & 1) * N * GP;
          auto pair = [&](int t, int& p, int& q) {
            if (r == 0) {
              p = t == 0 ? ir : ir + t >= N - 1 ? ir + t - (N - 1) : ir + t;
              q = t == 0 ? N - 1 : ir - t < 0 ? ir - t + N - 1 : ir - t;
            } else {
              p = t;
              q = BW + (t + ir >= BW ? t + ir - BW : t + ir);
            }
          };
          // no branches: a warp's threads look at different pairs, a thread at two
          auto angle = [&](int i, int j, float& c, float& s) {  // 0: no rotation, 1, or 2: a large one
            const float a = G[i * GP + i], b = G[j * GP + j], g = G[i * GP + j];
            const float sab = sqrt_approx(kGramScaleAb * a * b);  // 2^30 |w_p| |w_q|
            const float d = kGramScale * (b - a), h = 2.0f * kGramScale * g;
            const float t = __fdividef(copysignf(1.0f, d) * h, fabsf(d) + sqrt_approx(fmaf(d, d, h * h)));
            const bool on = fabsf(g) > fmaxf(tols * sab, kGramMinCoupling);
            c = on ? rsqrtf(fmaf(t, t, 1.0f)) : 1.0f;
            s = on ? c * t : 0.0f;
            return on ? (fabsf(g) > bigs * sab ? 2 : 1) : 0;
          };
          int p, q;
          float c, s;
          if (gx < BW) {  // a 2 x 2 block of the Gram matrix: both sides' rotations
            int u, v;
            float d, t;
            pair(gx, p, q);
            pair(gy, u, v);
            const int did_pair = angle(p, q, c, s);
            angle(u, v, d, t);
            const float gpu = G[p * GP + u], gpv = G[p * GP + v], gqu = G[q * GP + u], gqv = G[q * GP + v];
            const float pu = c * gpu - s * gqu, pv = c * gpv - s * gqv;
            const float qu = s * gpu + c * gqu, qv = s * gpv + c * gqv;
            H[p * GP + u] = d * pu - t * pv;
            H[p * GP + v] = t * pu + d * pv;
            H[q * GP + u] = d * qu - t * qv;
            H[q * GP + v] = t * qu + d * qv;
            if (gx == gy) {
              rotated += did_pair != 0;
              big |= did_pair == 2;
            }
          } else if (qx < BW) {  // four rows of a pair's columns of Q
            pair(qx, p, q);
            angle(p, q, c, s);
            float4 *qp = reinterpret_cast<float4*>(Qt + p * QP) + qy, *qq = reinterpret_cast<float4*>(Qt + q * QP) + qy;
            const float4 a = *qp, b = *qq;
            *qp = make_float4(c * a.x - s * b.x, c * a.y - s * b.y, c * a.z - s * b.z, c * a.w - s * b.w);
            *qq = make_float4(s * a.x + c * b.x, s * a.y + c * b.y, s * a.z + c * b.z, s * a.w + c * b.w);
          }
          // only the warps at work wait for one another
          asm volatile("bar.sync 1, %0;" ::"n"(32 * (GW + QW)) : "memory");
        }
        myrot += rotated;
        if (__syncthreads_or(rotated)) {
          // columns of W and V times Q: a warp per 32 rows and half of the columns
          did = 1;
          const int gw = (R + 31) / 32, gv = (C + 31) / 32;
          for (int t = warp; t < 2 * (gw + gv); t += NW) {
            const int h = t & 1, gr = t >> 1;
            const bool w = gr < gw;
            const int ld = w ? R : C, pitch = w ? RP : C, i = 32 * (w ? gr : gr - gw) + lane;
            if (i >= ld) continue;
            const float* src = (w ? Ws : Vs) + i;
            float* dst = (w ? W : V) + (int64_t)(h ? q0 : p0) * ld + i;
            const int n = h ? nq : np;
            float x[QP];
#pragma unroll
            for (int c = 0; c < QP; ++c) x[c] = c < N ? src[c * pitch] : 0.0f;
#pragma unroll 3
            for (int j = 0; j < n; ++j) {
              const float* y = Qt + (h * BW + j) * QP;
              float acc[2] = {};
#pragma unroll
              for (int c = 0; c < QP; c += 4) {
                const float4 z = *reinterpret_cast<const float4*>(y + c);
                acc[0] = fmaf(z.x, x[c], acc[0]);
                acc[1] = fmaf(z.y, x[c + 1], acc[1]);
                acc[0] = fmaf(z.z, x[c + 2], acc[0]);
                acc[1] = fmaf(z.w, x[c + 3], acc[1]);
              }
              __stcg(dst + (int64_t)j * ld, acc[0] + acc[1]);
            }
          }
        }
      }
      cluster.sync();  // the next round reads columns this round wrote, on other CTAs
    }
    const int f = (__syncthreads_or(did) ? 1 : 0) | (__syncthreads_or(big) ? 2 : 0);
    if (f && tid == 0) atomicOr(flag0 + (gs & 1), f);
    cluster.sync();
    if (tid == 0) {
      ctl->any = flag0[gs & 1];
      if (crank == 0) ctl->flag[(gs + 1) & 1] = 0;
    }
    __syncthreads();
    conv = !(ctl->any & 2);
    __syncthreads();
  }
  return sweeps;
}

// out[:, j] = scale * sum_i X[i, j] Aop[:, i]  (column-major: Aop rows x C,
// X C x C, out rows x C); a warp per (column j, 128 rows).
__device__ void gemm_cols(const double* Aop, int rows, int C, const double* X, double* out, double scale, int cw,
                          int lane) {
  constexpr int kCW = kSvdCluster * (kSvdThreads / 32);
  const int nrb = (rows + 127) / 128;
  for (int task = cw; task < C * nrb; task += kCW) {
    const int j = task / nrb, r0 = (task - j * nrb) * 128;
    const double* xj = X + (int64_t)j * C;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int i = 0; i < C; ++i) {
      const double x = __ldcg(xj + i);
      const double* ai = Aop + (int64_t)i * rows;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = r0 + lane + 32 * u;
        if (r < rows) acc[u] = fma(x, __ldcg(ai + r), acc[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = r0 + lane + 32 * u;
      if (r < rows) __stcg(out + (int64_t)j * rows + r, scale * acc[u]);
    }
  }
}

// G = 1.5 I - 0.5 Q^T Q (Q: C x C column-major), the factor of one
// Newton-Schulz step Q <- Q G towards the orthogonal polar factor of Q; a
// warp per (row i, four columns j).
__device__ void newton_schulz_factor(const double* Q, int C, double* G, int cw, int lane) {
  constexpr int kCW = kSvdCluster * (kSvdThreads / 32);
  const int nj = (C + 3) / 4;
  for (int task = cw; task < C * nj; task += kCW) {
    const int i = task / nj, j0 = (task - i * nj) * 4;
    const double* qi = Q + (int64_t)i * C;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int k = lane; k < C; k += 32) {
      const double x = __ldcg(qi + k);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (j0 + u < C) acc[u] = fma(x, __ldcg(Q + (int64_t)(j0 + u) * C + k), acc[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const double v = warp_sum(acc[u]);
      if (lane == 0 && j0 + u < C) __stcg(G + i + (int64_t)(j0 + u) * C, (i == j0 + u ? 1.5 : 0.0) - 0.5 * v);
    }
  }
}

// eig: a shift that makes the block B (here sa B in FP32, W) positive definite
// but hardly larger than that needs.  One-sided Jacobi finds a column of
// norm |lambda + shift| to FP32 accuracy relative to that norm, so with the
// Frobenius norm as the shift the eigenvectors of close small eigenvalues (a
// density matrix has many) come out mixed; 17 of the 42 blocks of the two-site
// density matrix then failed the refinement.  kLanczos Lanczos steps bound
// the spectrum: shift = max(0, -smallest Ritz value) + 10% of its extent (of
// the 42 blocks: 1% takes 14 FP32 sweeps and 3 refinement steps, 10% 12 and 3,
// 100% 10 and 5; 10.5, 9.6 and 9.4 ms in all).  A shift that is still too
// small only costs accuracy of the starting point.
constexpr int kLanczos = 32;
__device__ float lanczos_shift(const float* W, int C, float* v, float* vp, float* y, cg::cluster_group& cluster,
                               float* red, float* sh, int crank, int cw, int lane) {
  // v, vp, y: C floats each (global); red: (kThreads32 / 32) + 1 floats, sh: 2 kLanczos + 1 floats of this CTA
  constexpr int kCW = kSvdCluster * (kThreads32 / 32);
  const int tid = threadIdx.x;
  auto block_sum = [&](float x) {
    x = warp_sum(x);
    __syncthreads();
    if (lane == 0) red[tid >> 5] = x;
    __syncthreads();
    float t = 0.0f;
    for (int w = 0; w < (kThreads32 / 32); ++w) t += red[w];
    return t;
  };
  const int K = min(kLanczos, C);
  if (crank == 0) {  // a fixed start vector without structure
    float n = 0.0f;
    for (int i = tid; i < C; i += kThreads32) {
      const unsigned h = (unsigned)(i + 1) * 2654435761u;
      const float x = (float)(int)(h ^ (h >> 15)) * 4.656612873077393e-10f;
      n = fmaf(x, x, n);
      __stcg(v + i, x);
      __stcg(vp + i, 0.0f);
    }
    n = rsqrtf(block_sum(n));
    for (int i = tid; i < C; i += kThreads32) __stcg(v + i, n * __ldcg(v + i));
  }
  float beta = 0.0f;
  for (int k = 0; k < K; ++k) {
    cluster.sync();
    for (int j = cw; j < C; j += kCW) {  // y = W v (W symmetric)
      const float* wj = W + (int64_t)j * C;
      float a = 0.0f;
      for (int i = lane; i < C; i += 32) a = fmaf(__ldcg(wj + i), __ldcg(v + i), a);
      a = warp_sum(a);
      if (lane == 0) __stcg(y + j, a);
    }
    cluster.sync();
    if (crank == 0) {
      float a = 0.0f;
      for (int i = tid; i < C; i += kThreads32) a = fmaf(__ldcg(y + i), __ldcg(v + i), a);
      const float alpha = block_sum(a);
      float n = 0.0f;
      for (int i = tid; i < C; i += kThreads32) {
        const float r = __ldcg(y + i) - alpha * __ldcg(v + i) - beta * __ldcg(vp + i);
        n = fmaf(r, r, n);
        __stcg(vp + i, __ldcg(v + i));
        __stcg(v + i, r);
      }
      beta = sqrtf(block_sum(n));
      const float inv = beta > 1e-6f ? 1.0f / beta : 0.0f;  // an invariant subspace: the rest adds Ritz values 0
      for (int i = tid; i < C; i += kThreads32) __stcg(v + i, inv * __ldcg(v + i));
      if (inv == 0.0f) beta = 0.0f;
      if (tid == 0) {
        sh[k] = alpha;
        sh[kLanczos + k] = beta;  // between k and k + 1
      }
      __syncthreads();
    }
  }
  if (crank == 0 && tid == 0) {  // smallest eigenvalue of the tridiagonal matrix by bisection (Sturm counts)
    float lo = 0.0f, hi = 0.0f;
    for (int k = 0; k < K; ++k) {
      const float r = (k > 0 ? sh[kLanczos + k - 1] : 0.0f) + (k + 1 < K ? sh[kLanczos + k] : 0.0f);
      lo = fminf(lo, sh[k] - r);
      hi = fmaxf(hi, sh[k] + r);
    }
    const float extent = fmaxf(-lo, hi);
    float top = 0.0f;  // only a negative smallest value matters
    for (int it = 0; it < 24; ++it) {
      const float x = 0.5f * (lo + top);
      int below = 0;
      float d = 1.0f;
      for (int k = 0; k < K; ++k) {
        const float bk = k > 0 ? sh[kLanczos + k - 1] : 0.0f;
        d = sh[k] - x - bk * bk / d;
        if (d == 0.0f) d = -1e-30f;
        below += d < 0.0f;
      }
      if (below) top = x;
      else lo = x;
    }
    sh[2 * kLanczos] = -top + 0.1f * extent;
  }
  cluster.sync();
  return *cluster.map_shared_rank(sh + 2 * kLanczos, 0);
}

// A block for the sweeps: A from the tensor's blocks (eig: its symmetric part), sa A
// and I in FP32 (eig: sa A plus the shift), and the block's state.  A function of
// its own: inlined, its values cost the sweeps registers (6% at D = 96).
__device__ __noinline__ void load_block(const SvdBlock* __restrict__ block, const SvdPiece* __restrict__ pieces,
                                        const double* __restrict__ T, double* __restrict__ work,
                                        SvdState* __restrict__ state) {
  __shared__ unsigned long long wmax[kThreads32 / 32], amax;  // the largest |A| of the warps, of this CTA
  __shared__ double wsum[kThreads32 / 32];
  __shared__ double fpart;  // this CTA's part of the squared Frobenius norm
  __shared__ float lred[(kThreads32 / 32) + 1], lsh[2 * kLanczos + 1];
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int kCT = kSvdCluster * kThreads32;
  const int crank = (int)cluster.block_rank(), tid = threadIdx.x, lane = tid & 31;
  const int ct = crank * kThreads32 + tid, cw = ct >> 5;  // thread, warp of the cluster
  const SvdBlock& b = *block;
  const int R = b.R, C = b.C;
  const int64_t RC = (int64_t)R * C, CC = (int64_t)C * C;
  const SvdWork ws(work + b.w, R, C);
  double* A = ws.A;
  float *W32 = ws.W32, *V32 = ws.V32;

  // A (m >= n: M_x, else M_x^T) in FP64, column-major, and max |A|
  for (int64_t i = ct; i < RC; i += kCT) __stcg(A + i, 0.0);
  cluster.sync();
  unsigned long long mx = 0;
  for (int k = 0; k < b.nt; ++k) {
    const SvdPiece pc = pieces[b.t0 + k];
    const int64_t n = (int64_t)pc.rows * pc.cols;
    for (int64_t e = ct; e < n; e += kCT) {
      const int i = (int)(e / pc.cols), j = (int)(e - (int64_t)i * pc.cols);
      const int64_t r = pc.r0 + i, c = pc.c0 + j;
      const double v = T[pc.off + e];
      __stcg(b.trans ? A + c + r * R : A + r + c * R, v);
      mx = max(mx, (unsigned long long)__double_as_longlong(fabs(v)));  // |v| >= 0 orders as its bits
    }
  }
  cluster.sync();  // the whole block is in A
  // eig: the symmetric part, in place (the thread of (r, c), r < c, writes both halves)
  if (b.eig) {
    mx = 0;
    for (int64_t e = ct; e < RC; e += kCT) {
      const int r = (int)(e % R), c = (int)(e / R);
      if (r > c) continue;
      double v = __ldcg(A + e);
      if (r < c) {
        const int64_t t = c + (int64_t)r * R;
        v = 0.5 * (v + __ldcg(A + t));
        __stcg(A + e, v);
        __stcg(A + t, v);
      }
      mx = max(mx, (unsigned long long)__double_as_longlong(fabs(v)));
    }
  }
  // the largest |A| of all CTAs, read from each of them (64-bit atomics on
  // another CTA's shared memory lost the larger value now and then: a block
  // with one large entry was then scaled out of FP32's range)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) wmax[tid >> 5] = mx;
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kThreads32 / 32; ++w) mx = max(mx, wmax[w]);
    amax = mx;
  }
  cluster.sync();
  mx = 0;
  for (int r = 0; r < kSvdCluster; ++r) mx = max(mx, *cluster.map_shared_rank(&amax, r));
  const double amx = __longlong_as_double((long long)mx);
  // scale sa = 2^-e with 2^e <= max |A| < 2^(e+1); 1 for a zero or non-finite block
  const int ex = (__double2hiint(amx) >> 20) & 0x7ff;
  const bool scaled = ex > 0 && ex < 2046;
  const double sa = scaled ? __hiloint2double((2046 - ex) << 20, 0) : 1.0;
  const double unsa = scaled ? __hiloint2double(ex << 20, 0) : 1.0;  // 1 / sa

  // sa A in FP32, and its squared Frobenius norm in FP64: of the scaled values,
  // whose squares neither overflow nor underflow, at any scale of the block
  double f2 = 0.0;
  for (int64_t i = ct; i < RC; i += kCT) {
    const double v = sa * __ldcg(A + i);
    f2 = fma(v, v, f2);
    __stcg(W32 + i, (float)v);
  }
  for (int64_t i = ct; i < CC; i += kCT) __stcg(V32 + i, (i % (C + 1) == 0) ? 1.0f : 0.0f);
  f2 = warp_sum(f2);
  if (lane == 0) wsum[tid >> 5] = f2;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < (kThreads32 / 32); ++w) t += wsum[w];
    fpart = t;
  }
  cluster.sync();  // every CTA's part, and W32, are written
  f2 = 0.0;  // the same sum, in the same order, in every thread
  for (int r = 0; r < kSvdCluster; ++r) f2 += *cluster.map_shared_rank(&fpart, r);
  const double norm = sqrt(f2);  // of sa A
  if (b.eig) {  // the FP32 sweeps run on B + a shift; A keeps B
    const double s = C >= 4 ? (double)lanczos_shift(W32, C, ws.F0, ws.F0 + C, ws.F0 + 2 * C, cluster, lred, lsh, crank, cw, lane)
                            : norm;
    for (int j = ct; j < C; j += kCT)
      __stcg(W32 + j + (int64_t)j * R, (float)(sa * __ldcg(A + j + (int64_t)j * R) + s));
    cluster.sync();
  }
  if (crank == 0 && tid == 0) {
    SvdState& st = *state;
    st.sa = sa;
    st.unsa = unsa;
    st.norm = norm;
    st.done = 0;
    for (int i = 0; i < kMaxRefine; ++i) {
      st.xmax[i] = 0;
      st.nulls[i] = 0;
    }
  }
}

// One cluster of kSvdCluster CTAs per block: the pairs of a round are spread
// over the cluster's warps and the rounds are separated by cluster barriers
// (their release / acquire order the workspace writes; the workspace is read
// and written at L2, bypassing L1, so no SM keeps a stale copy).
//
// Mixed precision.  GB300 runs FP32 at many times its FP64 rate, so the
// sweeps that do most of the work run in FP32 on A scaled by a power of two
// (max |A| in [1/2, 1): no FP32 overflow or underflow of the bulk).  Their V
// is only the starting point: the refinement below takes it to FP64.
__global__ void __cluster_dims__(kSvdCluster, 1, 1) __launch_bounds__(kThreads32, 2)
    svd_jacobi_kernel(const SvdBlock* __restrict__ blocks, const SvdPiece* __restrict__ pieces,
                      const double* __restrict__ T, double* __restrict__ work, SvdState* __restrict__ state,
                      int* __restrict__ sweeps, long long* __restrict__ rotations) {
  __shared__ unsigned long long nrot;  // rotations of this CTA
  __shared__ SweepCtl ctl;
  // the sweeps by column blocks: a block pair of W and V (16-byte vectors in jacobi_sweeps_gram)
  extern __shared__ __align__(16) double sm_pair[];
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = (int)cluster.block_rank();
  const int bi = blockIdx.x / kSvdCluster;
  const SvdBlock b = blocks[bi];
  const int R = b.R, C = b.C;
  const int64_t CC = (int64_t)C * C;
  const SvdWork ws(work + b.w, R, C);
  float *W32 = ws.W32, *V32 = ws.V32;
  const int tid = threadIdx.x, lane = tid & 31;
  const int ct = crank * kThreads32 + tid;       // thread of the cluster
  const int cw = crank * (kThreads32 / 32) + (tid >> 5);  // warp of the cluster
  constexpr int kCT = kSvdCluster * kThreads32;
  if (tid == 0) {
    nrot = 0;
    ctl.flag[0] = ctl.flag[1] = 0;
    ctl.any = 0;
    if (crank == 0) rotations[2 * b.slot] = rotations[2 * b.slot + 1] = 0;
  }
  cluster.sync();  // shared state initialised before any remote access, the counts before they are added to
  load_block(blocks + bi, pieces, T, work, state + bi);

  int* flag0 = cluster.map_shared_rank(ctl.flag, 0);
  unsigned long long rot32 = 0;
  bool conv32;
  int gsweep = 0;
  const float tol32 = sqrtf((float)R) * FLT_EPSILON;
  float* nrm32 = reinterpret_cast<float*>(ws.nrm);
  int sw32;
  switch (b.bw) {  // the columns of a block, up to the bound of an instance
#define SYM_GRAM(BW)                                                                                              \
  case BW:                                                                                                        \
    sw32 = jacobi_sweeps_gram<BW>(W32, V32, R, C, b.bw, kMaxSweeps32, tol32, cluster, &ctl, flag0, crank, lane,   \
                                  gsweep, rot32, conv32, kBigRotation32, reinterpret_cast<float*>(sm_pair));      \
    break;
    SYM_GRAM(2)
    SYM_GRAM(3)
    SYM_GRAM(4)
    SYM_GRAM(5)
    SYM_GRAM(6)
    SYM_GRAM(7)
    SYM_GRAM(8)
    SYM_GRAM(9)
    SYM_GRAM(10)
    SYM_GRAM(11)
    SYM_GRAM(12)
    SYM_GRAM(13)
    SYM_GRAM(14)
#undef SYM_GRAM
    default:
      sw32 = jacobi_sweeps<float, kThreads32>(W32, V32, nrm32, R, C, kMaxSweeps32, tol32, cluster, &ctl, flag0, crank, cw, lane,
                                  gsweep, rot32, conv32, kBigRotation32);
  }
  if (b.bw ? rot32 != 0 : lane == 0 && rot32) atomicAdd(&nrot, rot32);
  for (int64_t i = ct; i < CC; i += kCT) __stcg(ws.V + i, (double)__ldcg(V32 + i));
  cluster.sync();  // no CTA leaves while its shared memory is read
  if (tid == 0 && nrot) atomicAdd(reinterpret_cast<unsigned long long*>(rotations + 2 * b.slot + 1), nrot);
  if (crank == 0 && tid == 0) {
    sweeps[2 * b.slot + 1] = sw32;
    sweeps[2 * b.slot] = 0;
  }
}

// ------------------------------------------------------------- FP64 refinement --
// V (from the FP32 sweeps, or from the step before) is orthogonal and
// diagonalises the block up to a small error; one step removes it to first
// order.  From W = A V, G = W^T W (eig: T = V^T W) and E = V^T V - I, all in
// FP64, the correction X with V' = V (I + X) has X_pq + X_qp = -E_pq and
// makes the off-diagonal element G_pq + a_p X_pq + a_q X_qp vanish (a_p, a_q:
// the diagonal elements): the symmetric part is -E/2, the antisymmetric one
// the Jacobi rotation of the pair with g' = G_pq - E_pq (a_p + a_q) / 2 (its
// sine, and on the diagonal its cosine less one, so that an isolated pair of
// close values is rotated exactly).  This is Newton's iteration for the
// singular value (eigenvalue) problem: what a step leaves is quadratic in X,
// so a step whose columns of X are all at most 1e-8 long ends the block: its
// remainder is 1e-16.  X multiplies V in FP32 (V' = V + V X: the product's
// relative error 6e-8 falls on a term of at most |X|, which the next step
// sees in full; on the last one it is 6e-16 of 1e-8), everything else is FP64.
//
// Against FP64 Jacobi sweeps, which this replaces: 2 RC^2 multiply-adds a
// step in products that spread over every SM, instead of 9/2 RC^2 a sweep in
// serial rounds on the block's own cluster.  FP64 (two multiply-adds a clock
// of an SM) bounds the products.  A block that has not converged after
// kMaxRefine steps (clusters of values the FP32 sweeps could not tell apart)
// starts again from the FP32 V with FP64 sweeps (svd_sweep_kernel).
constexpr int kTile = 32, kSlab = 16, kTileThreads = 128;

// 32 x 32 tile of out = alpha sum_k P(i, k) Q(k, j), Q column-major (ldq), P
// column-major (kTrans = false: P(i, k) = p[i + k ldp]) or transposed
// (p[k + i ldp]).  A thread has 4 x 2 elements 8 rows and 16 columns apart,
// so that rows and columns past the edge are skipped whole: an FP64
// multiply-add occupies a warp's FP64 pipe for 16 clocks.
template <bool kTrans, typename Store>
__device__ __forceinline__ void tile_f64(const double* __restrict__ p, int64_t ldp, int m, const double* __restrict__ q,
                                         int64_t ldq, int n, int K, int i0, int j0, Store store) {
  __shared__ double ps[2][kSlab][kTile + 1], qs[2][kSlab][kTile + 1];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int ml = min(kTile, m - i0), nl = min(kTile, n - j0);
  double rp[4], rq[4];
  auto load = [&](int k0) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + kTileThreads * u;
      const int kk = k0 + (kTrans ? e % kSlab : e / kTile), i = kTrans ? e / kSlab : e % kTile;
      rp[u] = kk < K && i < ml ? __ldcg(p + (kTrans ? kk + (int64_t)(i0 + i) * ldp : i0 + i + (int64_t)kk * ldp)) : 0.0;
      const int kq = k0 + e % kSlab, j = e / kSlab;
      rq[u] = kq < K && j < nl ? __ldcg(q + kq + (int64_t)(j0 + j) * ldq) : 0.0;
    }
  };
  auto put = [&](int s) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + kTileThreads * u;
      ps[s][kTrans ? e % kSlab : e / kTile][kTrans ? e / kSlab : e % kTile] = rp[u];
      qs[s][e % kSlab][e / kSlab] = rq[u];
    }
  };
  double acc[4][2] = {};
  const int ns = (K + kSlab - 1) / kSlab;
  load(0);
  put(0);
  __syncthreads();
  for (int s = 0; s < ns; ++s) {
    if (s + 1 < ns) load((s + 1) * kSlab);
#pragma unroll
    for (int k = 0; k < kSlab; ++k) {
      double a[4], b[2];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = ps[s & 1][k][ty + 8 * i];
#pragma unroll
      for (int j = 0; j < 2; ++j) b[j] = qs[s & 1][k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (8 * i < ml)
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (16 * j < nl) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (s + 1 < ns) put((s + 1) & 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (ty + 8 * i < ml && tx + 16 * j < nl) store(i0 + ty + 8 * i, j0 + tx + 16 * j, acc[i][j]);
}

__device__ __forceinline__ float* refine_f(const SvdWork& ws, int step) {
  return step == 0 ? ws.V32 : step & 1 ? ws.F0 : ws.F1;
}

// W = sa A V, and its FP32 copy (for W X of a last step)
__global__ void __launch_bounds__(kTileThreads)
    svd_av_kernel(const SvdBlock* __restrict__ blocks, const SvdTile* __restrict__ tiles, double* __restrict__ work,
                  const SvdState* __restrict__ state, int step) {
  const SvdTile t = tiles[blockIdx.x];
  if (state[t.block].done) return;
  const SvdBlock& b = blocks[t.block];
  const SvdWork ws(work + b.w, b.R, b.C);
  const double sa = state[t.block].sa;
  const int R = b.R;
  const bool eig = b.eig != 0;
  tile_f64<false>(ws.A, R, R, ws.V, b.C, b.C, b.C, t.i0, t.j0, [&](int i, int j, double v) {
    ws.W[i + (int64_t)j * R] = sa * v;
    if (!eig) ws.W32[i + (int64_t)j * R] = (float)(sa * v);
  });
}

// lower triangles of G = W^T W (eig: T = V^T W) and of V^T V
__global__ void __launch_bounds__(kTileThreads)
    svd_gram_kernel(const SvdBlock* __restrict__ blocks, const SvdTile* __restrict__ tiles, double* __restrict__ work,
                    const SvdState* __restrict__ state, int step) {
  const SvdTile t = tiles[blockIdx.x];
  if (state[t.block].done) return;
  const SvdBlock& b = blocks[t.block];
  const SvdWork ws(work + b.w, b.R, b.C);
  const double* V = ws.V;
  const int C = b.C;
  double* out = t.kind ? ws.E : ws.G;
  auto store = [&](int i, int j, double v) { out[i + (int64_t)j * C] = v; };
  if (t.kind)
    tile_f64<true>(V, C, C, V, C, C, C, t.i0, t.j0, store);
  else if (b.eig)
    tile_f64<true>(V, C, C, ws.W, C, C, C, t.i0, t.j0, store);
  else
    tile_f64<true>(ws.W, b.R, C, ws.W, b.R, C, b.R, t.i0, t.j0, store);
}

// X, a warp per column q.  The rotation's angle is formed in FP32 from d =
// a_q - a_p and h = 2 g' (X is FP32 anyway, and GB300's FP64 square roots and
// divisions are slow).  Pairs whose off-diagonal element is at FP64's rounding
// level are left alone, as in the Jacobi sweeps: |g'| <= sqrt(R) ulp of
// |w_p| |w_q| (eig: 4 ulp of the block's norm).  Many large angles at once do
// not make an orthogonal I + X, so pairs that the error of V so far cannot
// tell apart are left alone too: in a null space (g' no larger than that error
// squared times the norm: 1e-5 in step 0, 1e-9 in step 1, the rounding level
// 3e-14 after that) and in a cluster of equal values (difference and g' within
// 1e-6, then 1e-11 of them) -- as V becomes orthogonal their g' vanishes by
// itself.  In steps 0 and 1 such a pair asks for a further step; the columns of
// an SVD that stay at the rounding level (a block of less than full rank) are
// left to FP64 sweeps that start from the refined V.
__global__ void __launch_bounds__(256)
    svd_correction_kernel(const SvdBlock* __restrict__ blocks, const int2* __restrict__ cols, int ncols,
                          double* __restrict__ work, SvdState* __restrict__ state, int step) {
  const int w = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (w >= ncols) return;
  const int2 bq = cols[w];  // (block, column)
  SvdState& st = state[bq.x];
  if (st.done) return;
  const SvdBlock& b = blocks[bq.x];
  const SvdWork ws(work + b.w, b.R, b.C);
  const int C = b.C, q = bq.y;
  const double aq = ws.G[q + (int64_t)q * C], eqq = ws.E[q + (int64_t)q * C] - 1.0;
  const double tol = b.eig ? 4.0 * DBL_EPSILON * st.norm : sqrt((double)b.R) * DBL_EPSILON;
  const float sq = sqrtf((float)aq);
  // a null space's off-diagonal elements: of W^T W they are squares of the
  // error of V times the squared norm, of V^T B V times the norm
  const double null_level = (step == 0 ? 1e-10 : step == 1 ? 1e-18 : 1e-27) * st.norm * (b.eig ? 1.0 : st.norm);
  const double near = step == 0 ? 1e-6 : step == 1 ? 1e-11 : 0.0;
  bool skipped = false;
  float n2 = 0.0f, diag = 0.0f;
  for (int p = lane; p < C; p += 32) {
    if (p == q) continue;
    const int64_t at = p > q ? p + (int64_t)q * C : q + (int64_t)p * C;  // lower triangle
    const double ap = ws.G[p + (int64_t)p * C], e = ws.E[at];
    const double g = ws.G[at] - 0.5 * e * (ap + aq);
    float s = 0.0f;
    if (fabs(g) > (b.eig ? tol : tol * (double)(sq * sqrtf((float)ap)))) {
      const double d = aq - ap, h = 2.0 * g;
      const double m = fmax(fabs(d), fabs(h));
      const int ex = (__double2hiint(m) >> 20) & 0x7ff;
      float t = 0.0f;
      if (ex > 0 && ex < 2046) {
        const double sc = __hiloint2double((2046 - ex) << 20, 0);  // m * sc in [1, 2)
        const float df = (float)(d * sc), hf = (float)(h * sc);
        const float sgn = df > 0.0f || (df == 0.0f && p < q) ? 1.0f : -1.0f;
        t = sgn * hf / (fabsf(df) + sqrtf(fmaf(df, df, hf * hf)));
      } else {
        t = (float)(h / d);  // out of range: what comes of it fails the step's test
      }
      const double big = fmax(aq, ap);
      if ((fabs(g) <= null_level && (fabsf(t) > 0.05f || (b.eig ? fabs(d) : big) <= null_level)) ||
          m <= near * (b.eig ? st.norm : big)) {
        skipped = true;
      } else {
        const float c = rsqrtf(fmaf(t, t, 1.0f));
        s = c * t;
        diag -= s * s / (1.0f + c);  // c - 1
      }
    }
    const float x = s - 0.5f * (float)e;
    ws.X[p + (int64_t)q * C] = x;
    n2 = fmaf(x, x, n2);
  }
  n2 = warp_sum(n2);
  diag = warp_sum(diag);
  skipped = __any_sync(0xffffffffu, skipped);
  if (skipped && lane == 0) st.nulls[step] = 1;
  if (lane == 0) {
    const float x = diag - 0.5f * (float)eqq;
    ws.X[q + (int64_t)q * C] = x;
    n2 = fmaf(x, x, n2);
    if (skipped && step < 2) n2 = fmaxf(n2, 1e-15f);  // not the last step
    // a column of an SVD block this far below the others: X and W X, in FP32, no
    // longer carry its corrections.  One-sided sweeps find such values (of graded
    // columns) to full relative accuracy
    if (!b.eig && aq > 0.0 && aq < kMinNorm2) n2 = 1.0f;
    atomicMax(&st.xmax[step], __float_as_uint(n2));  // n2 >= 0 orders as its bits, a NaN above all
    if (b.eig) ws.nrm[q] = st.unsa * (aq / (1.0 + eqq));  // lambda: the Rayleigh quotient
  }
}

__device__ __forceinline__ bool last_step(const SvdState& st, int step) {
  return __uint_as_float(st.xmax[step]) <= 1e-16f;  // every column of X at most 1e-8 long
}

// the refinement ended with nothing left to do
__device__ __forceinline__ bool refined(const SvdState& st, const SvdBlock& b) {
  return st.done > 0 && (b.eig || !st.nulls[st.done - 1]);
}

// V' = V + V X (kind 0), and on a block's last step W' = W + W X (kind 1): in place,
// since the products read the FP32 copies
__global__ void __launch_bounds__(kTileThreads)
    svd_update_kernel(const SvdBlock* __restrict__ blocks, const SvdTile* __restrict__ tiles, double* __restrict__ work,
                      SvdState* __restrict__ state, int step) {
  __shared__ float ps[32][kTile + 1], xs[32][kTile + 1];
  const SvdTile t = tiles[blockIdx.x];
  SvdState& st = state[t.block];
  const int done = *reinterpret_cast<volatile int*>(&st.done);
  if (done && done != step + 1) return;  // this launch's own mark may be there already
  const SvdBlock& b = blocks[t.block];
  const bool last = last_step(st, step);
  const bool lost = !(__uint_as_float(st.xmax[step]) <= 0.25f);  // no longer a small correction (or a NaN)
  if (threadIdx.x == 0 && t.kind == 0 && t.i0 == 0 && t.j0 == 0 && (last || lost))
    *reinterpret_cast<volatile int*>(&st.done) = last ? step + 1 : -1;
  if (lost || (t.kind && (!last || b.eig))) return;
  const SvdWork ws(work + b.w, b.R, b.C);
  const int C = b.C, m = t.kind ? b.R : C;
  double* out = t.kind ? ws.W : ws.V;
  const float* srcf = t.kind ? ws.W32 : refine_f(ws, step);
  float* dstf = t.kind ? nullptr : refine_f(ws, step + 1);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int ml = min(kTile, m - t.i0), nl = min(kTile, C - t.j0);
  float acc[4][2] = {};
  for (int k0 = 0; k0 < C; k0 += 32) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = tid + kTileThreads * u;
      const int hi = e >> 5, lo = e & 31;
      ps[hi][lo] = k0 + hi < C && lo < ml ? __ldcg(srcf + t.i0 + lo + (int64_t)(k0 + hi) * m) : 0.0f;
      xs[lo][hi] = k0 + lo < C && hi < nl ? __ldcg(ws.X + k0 + lo + (int64_t)(t.j0 + hi) * C) : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 32; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) acc[i][j] = fmaf(ps[k][ty + 8 * i], xs[k][tx + 16 * j], acc[i][j]);
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ty + 8 * i, c = tx + 16 * j;
      if (r >= ml || c >= nl) continue;
      const int64_t at = t.i0 + r + (int64_t)(t.j0 + c) * m;
      const double v = out[at] + (double)acc[i][j];
      out[at] = v;
      if (dstf) dstf[at] = (float)v;
    }
}

// Columns of W at the rounding level of the block, |w| <= R eps |A|, can be exact
// multiples of one another (a block with equal rows): rotations then shrink them
// by eps a sweep without an end.  Sets such columns to 0 and returns whether the
// others are orthogonal.
__device__ bool drop_null_columns(double* W, int R, int C, double norm, cg::cluster_group& cluster, int* bad, int cw,
                                  int lane) {
  constexpr int kCW = kSvdCluster * (kSvdThreads / 32);
  const double level = (double)R * DBL_EPSILON * norm;
  auto dot = [&](int p, int q) {
    double g = 0.0;
    for (int i = lane; i < R; i += 32) g = fma(__ldcg(W + (int64_t)p * R + i), __ldcg(W + (int64_t)q * R + i), g);
    return warp_sum(g);
  };
  for (int j = cw; j < C; j += kCW)
    if (dot(j, j) <= level * level)
      for (int i = lane; i < R; i += 32) __stcg(W + (int64_t)j * R + i, 0.0);
  cluster.sync();
  int b = 0;
  for (int p = cw; p < C; p += kCW) {
    const double a = dot(p, p);
    for (int q = p + 1; q < C && a > 0.0; ++q) b |= !(fabs(dot(p, q)) <= 1e-13 * sqrt(a) * sqrt(dot(q, q)));
  }
  b = __syncthreads_or(b);
  if (threadIdx.x == 0) *bad = b;
  cluster.sync();
  for (int r = 0; r < kSvdCluster; ++r) b |= *cluster.map_shared_rank(bad, r);
  return !b;
}

// Blocks the refinement did not finish.  Where it converged but left columns
// at the rounding level (SVD), FP64 sweeps on its W and V, which mostly find
// nothing to rotate.  Else the FP32 V made orthogonal in FP64 by two
// Newton-Schulz steps (an orthogonality error e becomes ~1.5 e^2), W = A V
// (eig: A = B + sigma I), and FP64 sweeps to convergence.  Leaves W and V in
// place, the scaling undone, and the values (eig: |w_j| - sigma) in nrm.
__global__ void __cluster_dims__(kSvdCluster, 1, 1) __launch_bounds__(kSvdThreads, 2)
    svd_sweep_kernel(const SvdBlock* __restrict__ blocks, double* __restrict__ work,
                     const SvdState* __restrict__ state, int* __restrict__ sweeps, long long* __restrict__ rotations,
                     int* __restrict__ err) {
  __shared__ unsigned long long nrot;
  __shared__ SweepCtl ctl;
  __shared__ int bad;
  // the sweeps by column blocks: a block pair of W and V (16-byte vectors in jacobi_sweeps_gram)
  extern __shared__ __align__(16) double sm_pair[];
  cg::cluster_group cluster = cg::this_cluster();
  const int crank = (int)cluster.block_rank();
  const int bi = blockIdx.x / kSvdCluster;
  const int done = state[bi].done;  // the same for the whole cluster
  const SvdBlock b = blocks[bi];
  if (refined(state[bi], b)) return;
  const double sa = state[bi].sa, unsa = state[bi].unsa;
  const double shift = b.eig ? state[bi].norm : 0.0;  // sa sigma
  const int R = b.R, C = b.C;
  const int64_t CC = (int64_t)C * C;
  const SvdWork ws(work + b.w, R, C);
  double *W = ws.W, *V = ws.V, *A = ws.A, *G = ws.G, *nrm = ws.nrm;
  const int tid = threadIdx.x, lane = tid & 31;
  const int ct = crank * kSvdThreads + tid;
  const int cw = crank * (kSvdThreads / 32) + (tid >> 5);
  constexpr int kCT = kSvdCluster * kSvdThreads;
  constexpr int kCW = kSvdCluster * (kSvdThreads / 32);
  if (tid == 0) {
    nrot = 0;
    ctl.flag[0] = ctl.flag[1] = 0;
    ctl.any = 0;
  }
  cluster.sync();  // shared state initialised before any remote access
  if (done <= 0) {  // else the refined V and W are in place
    // two Newton-Schulz steps through the G buffer, the first one's product in
    // W's buffer (free until W = A V)
    for (int64_t i = ct; i < CC; i += kCT) __stcg(V + i, (double)__ldcg(ws.V32 + i));
    if (b.eig)  // sa (B + sigma I)
      for (int64_t i = ct; i < CC; i += kCT) __stcg(A + i, sa * __ldcg(A + i) + (i % (C + 1) == 0 ? shift : 0.0));
    cluster.sync();
    newton_schulz_factor(V, C, G, cw, lane);
    cluster.sync();
    gemm_cols(V, C, C, G, W, 1.0, cw, lane);
    cluster.sync();
    newton_schulz_factor(W, C, G, cw, lane);
    cluster.sync();
    gemm_cols(W, C, C, G, V, 1.0, cw, lane);
    cluster.sync();
    gemm_cols(A, R, C, V, W, b.eig ? 1.0 : sa, cw, lane);  // W = (sa A) V
    cluster.sync();
  }

  int* flag0 = cluster.map_shared_rank(ctl.flag, 0);
  unsigned long long rot64 = 0;
  bool conv;
  int gsweep = 0;
  const double tol64 = sqrt((double)R) * DBL_EPSILON;
  int sw64;
  switch (b.bw64 ? (R + 31) / 32 : 0) {
#define SYM_BLOCKED(NR)                                                                                          \
  case NR:                                                                                                        \
    sw64 = jacobi_sweeps_blocked<double, NR, kSvdThreads>(W, V, nrm, R, C, b.bw64, kMaxSweeps, tol64, cluster, &ctl, flag0,   \
                                             crank, lane, gsweep, rot64, conv, kBigRotation, sm_pair);          \
    break;
    SYM_BLOCKED(1)
    SYM_BLOCKED(2)
    SYM_BLOCKED(3)
    SYM_BLOCKED(4)
    SYM_BLOCKED(5)
    SYM_BLOCKED(6)
    SYM_BLOCKED(7)
    SYM_BLOCKED(8)
    SYM_BLOCKED(9)
    SYM_BLOCKED(10)
    SYM_BLOCKED(11)
    SYM_BLOCKED(12)
#undef SYM_BLOCKED
    default:
      sw64 = jacobi_sweeps<double, kSvdThreads>(W, V, nrm, R, C, kMaxSweeps, tol64, cluster, &ctl, flag0, crank, cw, lane, gsweep,
                                   rot64, conv, kBigRotation);
  }
  if (lane == 0 && rot64) atomicAdd(&nrot, rot64);
  if (!conv && !b.eig) conv = drop_null_columns(W, R, C, state[bi].norm, cluster, &bad, cw, lane);

  // take the column norms (of the scaled columns: their squares stay in range)
  // and undo the scaling (a power of two: exact)
  for (int j = cw; j < C; j += kCW) {
    double* wj = W + (int64_t)j * R;
    double a = 0.0;
    for (int i = lane; i < R; i += 32) {
      const double x = __ldcg(wj + i);
      __stcg(wj + i, unsa * x);
      a = fma(x, x, a);
    }
    a = warp_sum(a);
    if (lane == 0) __stcg(nrm + j, unsa * (sqrt(a) - shift));
  }
  cluster.sync();  // no CTA leaves while its shared memory is read
  if (tid == 0 && nrot) atomicAdd(reinterpret_cast<unsigned long long*>(rotations + 2 * b.slot), nrot);
  if (crank == 0 && tid == 0) {
    if (!conv) atomicExch(err, SYM_ERR_NUMERIC);
    sweeps[2 * b.slot] = sw64;
  }
}

// Refined blocks: the scaling of W undone, and its column norms (as in
// svd_sweep_kernel); a warp per column.
__global__ void __launch_bounds__(256)
    svd_place_kernel(const SvdBlock* __restrict__ blocks, const int2* __restrict__ cols, int ncols,
                     double* __restrict__ work, const SvdState* __restrict__ state, int* __restrict__ sweeps) {
  const int w = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (w >= ncols) return;
  const int2 bq = cols[w];
  const SvdState& st = state[bq.x];
  const SvdBlock& b = blocks[bq.x];
  if (!refined(st, b)) return;
  const SvdWork ws(work + b.w, b.R, b.C);
  const int R = b.R, C = b.C, j = bq.y;
  if (!b.eig) {
    double a = 0.0;
    for (int i = lane; i < R; i += 32) {
      const double x = ws.W[i + (int64_t)j * R];
      ws.W[i + (int64_t)j * R] = st.unsa * x;
      a = fma(x, x, a);
    }
    a = warp_sum(a);
    if (lane == 0) ws.nrm[j] = st.unsa * sqrt(a);
  }
  if (j == 0 && lane == 0) sweeps[2 * b.slot] = st.done;
}

// Values in descending order (eig: of |lambda|; ties: the larger lambda, then
// the column) with their permutation; a thread per column.
__global__ void __launch_bounds__(128)
    svd_rank_kernel(const SvdBlock* __restrict__ blocks, double* __restrict__ work, double* __restrict__ S,
                    int* __restrict__ perm) {
  const SvdBlock& b = blocks[blockIdx.x];
  const SvdWork ws(work + b.w, b.R, b.C);
  const int C = b.C;
  for (int j = blockIdx.y * 128 + threadIdx.x; j < C; j += gridDim.y * 128) {
    const double v = ws.nrm[j], av = fabs(v);
    int rank = 0;
    for (int i = 0; i < C; ++i) {
      const double u = ws.nrm[i], au = fabs(u);
      rank += (au > av) || (au == av && (u > v || (u == v && i < j)));
    }
    S[b.s + rank] = (b.eig ? b.sgn : 1.0) * v / b.vscale;
    ws.Ss[rank] = v;
    perm[b.s + rank] = j;
  }
}

// From A V = W with orthogonal columns: M = (W / S) diag(S) V^T when A = M,
// and M = V diag(S) (W / S)^T when A = M^T.
__global__ void __launch_bounds__(kSvdThreads)
    svd_factor_kernel(const SvdBlock* __restrict__ blocks, const SvdPiece* __restrict__ pieces,
                      const double* __restrict__ work, const int* __restrict__ perm, double* __restrict__ U,
                      double* __restrict__ Vt, double* __restrict__ Sk, int absorb) {
  const SvdBlock b = blocks[blockIdx.x];
  const int R = b.R, C = b.C, k = b.keep;
  if (k == 0) return;
  const double* W = work + b.w;
  const double* V = W + (int64_t)R * C;
  const double* Ss = V + (int64_t)C * C + C;
  const int* pm = perm + b.s;
  const int tid = threadIdx.x;
  // SU(2): the factors are vscale times the orthonormal ones and the values
  // are divided by it; absorbing S gives the orthonormal factor times sigma
  const double vs = b.vscale;
  if (b.eig) {  // M = Q diag(lambda) Q^T: U = vs Q, V = sgn vs Q^T, values sgn lambda / vs
    const double sg = b.sgn;
    if (Sk)
      for (int j = tid; j < k; j += kSvdThreads) Sk[b.ks + j] = sg * Ss[j] / vs;
    for (int q = 0; q < b.nu; ++q) {
      const SvdPiece pc = pieces[b.u0 + q];
      const int64_t n = (int64_t)pc.rows * k;
      for (int64_t e = tid; e < n; e += kSvdThreads) {
        const int i = (int)(e / k), j = (int)(e - (int64_t)i * k);
        U[pc.off + e] = V[pc.r0 + i + (int64_t)pm[j] * C] * (absorb == 1 ? sg * Ss[j] : vs);
      }
    }
    for (int q = 0; q < b.nv; ++q) {
      const SvdPiece pc = pieces[b.v0 + q];
      const int64_t n = (int64_t)k * pc.cols;
      for (int64_t e = tid; e < n; e += kSvdThreads) {
        const int j = (int)(e / pc.cols);
        const int64_t c = pc.c0 + (e - (int64_t)j * pc.cols);
        Vt[pc.off + e] = V[c + (int64_t)pm[j] * C] * (absorb == 2 ? Ss[j] : sg * vs);
      }
    }
    return;
  }
  if (Sk)
    for (int j = tid; j < k; j += kSvdThreads) Sk[b.ks + j] = Ss[j] / vs;
  for (int q = 0; q < b.nu; ++q) {
    const SvdPiece pc = pieces[b.u0 + q];
    const int64_t n = (int64_t)pc.rows * k;
    for (int64_t e = tid; e < n; e += kSvdThreads) {
      const int i = (int)(e / k), j = (int)(e - (int64_t)i * k);
      const int64_t r = pc.r0 + i, pj = pm[j];
      const double s = Ss[j];
      double v;
      if (!b.trans) {
        const double w = W[r + pj * R];
        v = absorb == 1 ? w : (s > 0.0 ? vs * w / s : 0.0);
      } else {
        v = V[r + pj * C];
        v *= absorb == 1 ? s : vs;
      }
      U[pc.off + e] = v;
    }
  }
  for (int q = 0; q < b.nv; ++q) {
    const SvdPiece pc = pieces[b.v0 + q];
    const int64_t n = (int64_t)k * pc.cols;
    for (int64_t e = tid; e < n; e += kSvdThreads) {
      const int j = (int)(e / pc.cols);
      const int64_t c = pc.c0 + (e - (int64_t)j * pc.cols), pj = pm[j];
      const double s = Ss[j];
      double v;
      if (!b.trans) {
        v = V[c + pj * C];
        v *= absorb == 2 ? s : vs;
      } else {
        const double w = W[c + pj * R];
        v = absorb == 2 ? w : (s > 0.0 ? vs * w / s : 0.0);
      }
      Vt[pc.off + e] = v;
    }
  }
}

struct TupleEntry {
  int x;
  int64_t first, extent;
};
using TupleMap = std::unordered_map<std::vector<int>, TupleEntry, VecHash>;

int fused_label(int group, const std::vector<Leg>& legs, int l0, const std::vector<int>& pos) {
  if (group == SYM_SU2) return legs[l0].labels[pos[0]];  // rank 2: the spin of the one leg
  int k = 0;
  for (size_t i = 0; i < pos.size(); ++i) {
    const Leg& L = legs[l0 + i];
    k = group == SYM_Z2F ? (k ^ L.labels[pos[i]]) : k + L.dir * L.labels[pos[i]];
  }
  return k;
}

// Every label tuple of legs [l0, l1), lexicographic (first leg slowest),
// grouped by the block label x = partner(fused label), with its first
// row (column) inside the block.
TupleMap enumerate_tuples(int group, const std::vector<Leg>& legs, int l0, int l1, bool columns, int total,
                          std::unordered_map<int, int64_t>& extent) {
  TupleMap out;
  const int k = l1 - l0;
  std::vector<int> pos(k, 0);
  while (true) {
    const int f = fused_label(group, legs, l0, pos);
    const int x = !columns || group == SYM_SU2 ? f : group == SYM_Z2F ? (total ^ f) : total - f;
    int64_t e = 1;
    for (int i = 0; i < k; ++i) e *= legs[l0 + i].degens[pos[i]];
    int64_t& acc = extent[x];
    out[pos] = TupleEntry{x, acc, e};
    acc += e;
    int i = k - 1;
    while (i >= 0 && ++pos[i] == (int)legs[l0 + i].labels.size()) pos[i--] = 0;
    if (i < 0) break;
  }
  return out;
}

}  // namespace

struct SvdPlan {
  Tensor T;
  int nrow = 0;
  bool eig = false;  // eigendecomposition plan (sym_eig_plan)
  std::vector<int> xs;            // block labels, ascending
  std::vector<SvdBlock> blocks;   // ascending x
  std::vector<SvdPiece> tpieces;  // grouped by block
  TupleMap rows, cols;
  int64_t nsv = 0, work_elems = 0;
  int64_t smem32 = 0;      // dynamic shared memory of the Jacobi launch (FP32 sweeps by column blocks)
  std::vector<int> order;  // launch order: blocks by decreasing work
  bool dry = false;
  bool bonded = false;

  std::vector<SvdTile> tiles[3];  // refinement products: W; the two Gram matrices; V' and W'
  std::vector<int2> columns;      // (block, column)

  DeviceArena arena;
  SvdBlock* d_blocks = nullptr;
  SvdTile* d_tiles[3] = {nullptr, nullptr, nullptr};
  int2* d_cols = nullptr;
  SvdState* state = nullptr;
  double* work = nullptr;
  int* perm = nullptr;
  int* sweeps = nullptr;
  long long* rotations = nullptr;
  SvdPiece* d_pieces = nullptr;  // T pieces, then U and V pieces of the last bond
  size_t pieces_cap = 0;

  ~SvdPlan() {
    if (d_pieces) cudaFree(d_pieces);
  }

  void upload_blocks() {
    std::vector<SvdBlock> launch;
    for (int i : order) launch.push_back(blocks[i]);
    cudaError_t e = cudaMemcpy(d_blocks, launch.data(), launch.size() * sizeof(SvdBlock), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) fail(SYM_ERR_CUDA, std::string("svd plan upload: ") + cudaGetErrorString(e));
  }

  void upload_pieces(const std::vector<SvdPiece>& all) {
    cudaError_t e = cudaDeviceSynchronize();  // no launch of this plan may still read the old lists
    if (e != cudaSuccess) fail(SYM_ERR_CUDA, std::string("svd plan upload: ") + cudaGetErrorString(e));
    if (all.size() > pieces_cap) {
      if (d_pieces) cudaFree(d_pieces);
      d_pieces = nullptr;
      pieces_cap = 0;
      e = cudaMalloc(&d_pieces, all.size() * sizeof(SvdPiece));
      if (e != cudaSuccess) {
        d_pieces = nullptr;
        cudaGetLastError();
        fail(e == cudaErrorMemoryAllocation ? SYM_ERR_OOM : SYM_ERR_CUDA,
             std::string("cudaMalloc failed: ") + cudaGetErrorString(e));
      }
      pieces_cap = all.size();
    }
    e = cudaMemcpy(d_pieces, all.data(), all.size() * sizeof(SvdPiece), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) fail(SYM_ERR_CUDA, std::string("svd plan upload: ") + cudaGetErrorString(e));
  }
};

std::unique_ptr<SvdPlan> plan_svd(const Tensor& T, int nrow, bool eig) {
  const char* what = eig ? "blockwise eigendecomposition" : "blockwise SVD";
  if (T.group == SYM_SU2U1) fail(SYM_ERR_UNSUPPORTED, std::string(what) + " of SU(2) x U(1) tensors is not built");
  if (T.group == SYM_SU2 && T.rank != 2)
    fail(SYM_ERR_UNSUPPORTED, std::string(what) + " of SU(2) tensors is built for rank 2 (the block-diagonal form)");
  if (T.rank < 2 || nrow < 1 || nrow >= T.rank) fail(SYM_ERR_ARG, "SVD needs rank >= 2 and 1 <= nrow < rank");
  if (eig) {  // a square matrix: the column legs are the row legs reversed, total label 0
    if (T.rank != 2 * nrow) fail(SYM_ERR_ARG, "eigendecomposition needs rank = 2 nrow");
    for (int l = 0; l < nrow; ++l)
      if (!T.legs[l].same_content(T.legs[nrow + l]) || T.legs[l].dir != -T.legs[nrow + l].dir)
        fail(SYM_ERR_INCOMPATIBLE_LEGS,
             "eigendecomposition: column leg " + std::to_string(nrow + l) + " must be row leg " + std::to_string(l) +
                 " reversed (same labels and degeneracies, opposite direction)");
    if (T.group != SYM_SU2 && T.total != 0) fail(SYM_ERR_ARG, "eigendecomposition needs total label 0");
  }
  auto P = std::make_unique<SvdPlan>();
  P->T = T;
  P->nrow = nrow;
  P->eig = eig;
  std::unordered_map<int, int64_t> mext, next;
  P->rows = enumerate_tuples(T.group, T.legs, 0, nrow, false, T.total, mext);
  P->cols = enumerate_tuples(T.group, T.legs, nrow, T.rank, true, T.total, next);
  for (auto& kv : mext)
    if (next.count(kv.first)) P->xs.push_back(kv.first);
  std::sort(P->xs.begin(), P->xs.end());
  if (P->xs.empty()) fail(SYM_ERR_ARG, "the tensor has no blocks");
  std::unordered_map<int, int> slot_of;
  for (int x : P->xs) {
    const int64_t m = mext[x], n = next[x];
    if (m >= (int64_t)1 << 31 || n >= (int64_t)1 << 31) fail(SYM_ERR_UNSUPPORTED, "SVD block too large");
    SvdBlock b{};
    b.m = (int)m;
    b.n = (int)n;
    b.trans = m < n;
    b.R = (int)std::max(m, n);
    b.C = (int)std::min(m, n);
    b.slot = (int)P->blocks.size();
    b.vscale = T.group == SYM_SU2 ? std::sqrt((double)x + 1.0) : 1.0;
    b.eig = eig ? 1 : 0;
    // SU(2) with an incoming row leg: the dense block is (-1)^{2j} M_x / sqrt(2j+1) (x) 1
    b.sgn = (eig && T.group == SYM_SU2 && T.legs[0].dir == -1 && (x & 1)) ? -1.0 : 1.0;
    if (eig && m != n) fail(SYM_ERR_ARG, "internal: eigendecomposition block is not square");
    // sweeps by column blocks when a block pair of W and V (FP64: rows up to 12
    // per lane) fits the shared memory two CTAs of an SM can have
    {
      const int bw = (b.C + kColBlocks - 1) / kColBlocks;
      const int64_t bytes = 2 * (int64_t)bw * (b.R + b.C + 1) * (int64_t)sizeof(float);
      const int64_t gram = gram_floats(b.R, b.C, bw) * (int64_t)sizeof(float);
      const bool ok = b.C >= kColBlocks * 2 && b.R <= 32 * 12;  // FP64
      b.bw = (b.C >= kColBlocks * 2 && bw <= kMaxGram && gram <= kSvdSmem32Max) ? bw : 0;
      // FP64 by column blocks for the SVD only: on the shifted symmetric blocks of
      // the eigendecomposition that order took up to 6 FP64 sweeps where the
      // order by pairs takes 4 (two-site density matrix: 29.8 against 29.0 ms;
      // two-site SVD: 20.4 against 22.3 ms)
      b.bw64 = (ok && !eig && 2 * bytes <= kSvdSmem64Max) ? bw : 0;
      P->smem32 = std::max<int64_t>(P->smem32, std::max<int64_t>(b.bw ? gram : 0, b.bw64 ? 2 * bytes : 0));
    }
    b.w = P->work_elems;
    b.s = P->nsv;
    P->work_elems += SvdWork::elems(b.R, b.C);
    P->nsv += b.C;
    slot_of[x] = b.slot;
    P->blocks.push_back(b);
  }
  // tensor blocks, grouped by diagonal block
  std::vector<std::vector<SvdPiece>> per(P->blocks.size());
  for (int64_t s = 0; s < T.nsec(); ++s) {
    std::vector<int> rt(T.pos.begin() + s * T.rank, T.pos.begin() + s * T.rank + nrow);
    std::vector<int> ct(T.pos.begin() + s * T.rank + nrow, T.pos.begin() + (s + 1) * T.rank);
    const TupleEntry& r = P->rows.at(rt);
    const TupleEntry& c = P->cols.at(ct);
    if (r.x != c.x) fail(SYM_ERR_ARG, "internal: block outside the diagonal");
    const SvdBlock& b = P->blocks[slot_of.at(r.x)];
    if (r.first + r.extent > b.m || c.first + c.extent > b.n || r.extent * c.extent != T.block_size(s))
      fail(SYM_ERR_ARG, "internal: block outside its matrix");
    per[b.slot].push_back(SvdPiece{T.offs[s], (int)r.first, (int)c.first, (int)r.extent, (int)c.extent});
  }
  for (auto& b : P->blocks) {
    b.t0 = (int)P->tpieces.size();
    b.nt = (int)per[b.slot].size();
    P->tpieces.insert(P->tpieces.end(), per[b.slot].begin(), per[b.slot].end());
  }
  for (size_t i = 0; i < P->blocks.size(); ++i) P->order.push_back((int)i);
  std::stable_sort(P->order.begin(), P->order.end(), [&](int a, int c) {
    const SvdBlock &A = P->blocks[a], &B = P->blocks[c];
    return (double)A.R * A.C * A.C > (double)B.R * B.C * B.C;
  });
  // refinement tiles, the blocks in launch order (decreasing work)
  for (size_t o = 0; o < P->order.size(); ++o) {
    const SvdBlock& b = P->blocks[P->order[o]];
    for (int j = 0; j < b.C; j += kTile)
      for (int i = 0; i < b.R; i += kTile) {
        P->tiles[0].push_back({(int)o, i, j, 0});
        if (!eig) P->tiles[2].push_back({(int)o, i, j, 1});
      }
    for (int j = 0; j < b.C; j += kTile)
      for (int i = 0; i < b.C; i += kTile) {
        if (i >= j) {
          P->tiles[1].push_back({(int)o, i, j, 0});
          P->tiles[1].push_back({(int)o, i, j, 1});
        }
        P->tiles[2].push_back({(int)o, i, j, 0});
      }
    for (int j = 0; j < b.C; ++j) P->columns.push_back(make_int2((int)o, j));
  }
  const char* dry = std::getenv("SYM_PLAN_DRYRUN");
  P->dry = dry && dry[0] == '1';
  if (!P->dry) {
    for (int k = 0; k < 3; ++k) {
      P->d_tiles[k] = static_cast<SvdTile*>(P->arena.alloc(P->tiles[k].size() * sizeof(SvdTile), false));
      cudaError_t e = cudaMemcpy(P->d_tiles[k], P->tiles[k].data(), P->tiles[k].size() * sizeof(SvdTile),
                                 cudaMemcpyHostToDevice);
      if (e != cudaSuccess) fail(SYM_ERR_CUDA, std::string("svd plan upload: ") + cudaGetErrorString(e));
    }
    P->d_cols = static_cast<int2*>(P->arena.alloc(P->columns.size() * sizeof(int2), false));
    cudaError_t ec = cudaMemcpy(P->d_cols, P->columns.data(), P->columns.size() * sizeof(int2), cudaMemcpyHostToDevice);
    if (ec != cudaSuccess) fail(SYM_ERR_CUDA, std::string("svd plan upload: ") + cudaGetErrorString(ec));
    P->state = static_cast<SvdState*>(P->arena.alloc(P->blocks.size() * sizeof(SvdState), true));
    P->d_blocks = static_cast<SvdBlock*>(P->arena.alloc(P->blocks.size() * sizeof(SvdBlock), false));
    P->work = static_cast<double*>(P->arena.alloc(P->work_elems * sizeof(double), true));
    P->perm = static_cast<int*>(P->arena.alloc(P->nsv * sizeof(int), true));
    P->sweeps = static_cast<int*>(P->arena.alloc(2 * P->blocks.size() * sizeof(int), true));
    P->rotations = static_cast<long long*>(P->arena.alloc(2 * P->blocks.size() * sizeof(long long), true));
    P->upload_blocks();
    P->upload_pieces(P->tpieces);
  }
  return P;
}

}  // namespace sym

struct sym_svd_s {
  std::unique_ptr<sym::SvdPlan> p;
};

namespace {

void need(bool ok, const char* msg) {
  if (!ok) sym::fail(SYM_ERR_ARG, msg);
}

void check_launch(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) sym::fail(SYM_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

}  // namespace

extern "C" {

int sym_svd_plan(sym_tensor T, int nrow, sym_svd* out, int* nblocks, int64_t* nsv) {
  return sym::guard([&] {
    need(T != nullptr && out != nullptr, "T or out is NULL");
    auto P = sym::plan_svd(T->t, nrow, false);
    if (nblocks) *nblocks = (int)P->blocks.size();
    if (nsv) *nsv = P->nsv;
    *out = new sym_svd_s{std::move(P)};
    return SYM_OK;
  });
}

int sym_eig_plan(sym_tensor T, int nrow, sym_svd* out, int* nblocks, int64_t* nev) {
  return sym::guard([&] {
    need(T != nullptr && out != nullptr, "T or out is NULL");
    auto P = sym::plan_svd(T->t, nrow, true);
    if (nblocks) *nblocks = (int)P->blocks.size();
    if (nev) *nev = P->nsv;
    *out = new sym_svd_s{std::move(P)};
    return SYM_OK;
  });
}

int sym_svd_blocks(sym_svd plan, int* x, int* m, int* n) {
  return sym::guard([&] {
    need(plan != nullptr, "plan is NULL");
    const auto& P = *plan->p;
    for (size_t i = 0; i < P.blocks.size(); ++i) {
      if (x) x[i] = P.xs[i];
      if (m) m[i] = P.blocks[i].m;
      if (n) n[i] = P.blocks[i].n;
    }
    return SYM_OK;
  });
}

namespace {
void launch_jacobi(sym::SvdPlan& P, const double* T, double* S, void* stream) {
  if (P.dry) sym::fail(SYM_ERR_UNSUPPORTED, "plan was built with SYM_PLAN_DRYRUN=1 and cannot run");
  static int attr_set = -1;  // dynamic shared memory the kernels are allowed (set once to the maximum)
  if (attr_set < 0) {
    auto allow = [](auto* k) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sym::kSvdSmem32Max);
      return e == cudaSuccess ? cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : e;
    };
    cudaError_t e = allow(sym::svd_jacobi_kernel);
    if (e == cudaSuccess) e = allow(sym::svd_sweep_kernel);
    if (e != cudaSuccess) sym::fail(SYM_ERR_CUDA, std::string("SVD kernel attribute: ") + cudaGetErrorString(e));
    attr_set = 1;
  }
  const cudaStream_t s = static_cast<cudaStream_t>(stream);
  const unsigned nb = (unsigned)P.blocks.size(), ncols = (unsigned)P.columns.size();
  const unsigned warps = (ncols + 7) / 8;  // CTAs of the warp-per-column kernels
  sym::svd_jacobi_kernel<<<nb * sym::kSvdCluster, sym::kThreads32, (size_t)P.smem32, s>>>(
      P.d_blocks, P.d_pieces, T, P.work, P.state, P.sweeps, P.rotations);
  check_launch("svd_jacobi_kernel");
  for (int step = 0; step < sym::kMaxRefine; ++step) {
    sym::svd_av_kernel<<<(unsigned)P.tiles[0].size(), sym::kTileThreads, 0, s>>>(P.d_blocks, P.d_tiles[0], P.work,
                                                                               P.state, step);
    sym::svd_gram_kernel<<<(unsigned)P.tiles[1].size(), sym::kTileThreads, 0, s>>>(P.d_blocks, P.d_tiles[1], P.work,
                                                                                 P.state, step);
    sym::svd_correction_kernel<<<warps, 256, 0, s>>>(P.d_blocks, P.d_cols, (int)ncols, P.work, P.state, step);
    sym::svd_update_kernel<<<(unsigned)P.tiles[2].size(), sym::kTileThreads, 0, s>>>(P.d_blocks, P.d_tiles[2], P.work,
                                                                                   P.state, step);
    check_launch("SVD refinement");
  }
  sym::svd_sweep_kernel<<<nb * sym::kSvdCluster, sym::kSvdThreads, (size_t)P.smem32, s>>>(
      P.d_blocks, P.work, P.state, P.sweeps, P.rotations, sym::device_error_word());
  check_launch("svd_sweep_kernel");
  sym::svd_place_kernel<<<warps, 256, 0, s>>>(P.d_blocks, P.d_cols, (int)ncols, P.work, P.state, P.sweeps);
  int cmax = 1;
  for (const auto& b : P.blocks) cmax = std::max(cmax, b.C);
  sym::svd_rank_kernel<<<dim3(nb, (unsigned)std::min(64, (cmax + 127) / 128)), 128, 0, s>>>(P.d_blocks, P.work, S,
                                                                                          P.perm);
  check_launch("svd_rank_kernel");
}
}  // namespace

int sym_eig_execute(sym_svd plan, const double* T, double* lambda, void* stream) {
  return sym::guard([&] {
    need(plan != nullptr && T != nullptr && lambda != nullptr, "plan, T or lambda is NULL");
    need(plan->p->eig, "not an eigendecomposition plan (sym_eig_plan)");
    launch_jacobi(*plan->p, T, lambda, stream);
    return SYM_OK;
  });
}

int sym_svd_execute(sym_svd plan, const double* T, double* S, void* stream) {
  return sym::guard([&] {
    need(plan != nullptr && T != nullptr && S != nullptr, "plan, T or S is NULL");
    auto& P = *plan->p;
    need(!P.eig, "an eigendecomposition plan runs with sym_eig_execute");
    launch_jacobi(P, T, S, stream);
    return SYM_OK;
  });
}

int sym_svd_stats(sym_svd plan, int fp32, int* sweeps, int64_t* rotations) {
  return sym::guard([&] {
    need(plan != nullptr, "plan is NULL");
    need(fp32 == 0 || fp32 == 1, "fp32 must be 0 (the FP64 sweeps) or 1 (the FP32 sweeps)");
    auto& P = *plan->p;
    if (P.dry) sym::fail(SYM_ERR_UNSUPPORTED, "plan was built with SYM_PLAN_DRYRUN=1 and cannot run");
    const size_t nb = P.blocks.size();
    std::vector<int> sw(2 * nb);
    std::vector<long long> r(2 * nb);
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(sw.data(), P.sweeps, sw.size() * sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(r.data(), P.rotations, r.size() * sizeof(long long), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) sym::fail(SYM_ERR_CUDA, std::string("svd stats: ") + cudaGetErrorString(e));
    const int k = fp32;
    for (size_t i = 0; i < nb; ++i) {
      if (sweeps) sweeps[i] = sw[2 * i + k];
      if (rotations) rotations[i] = r[2 * i + k];
    }
    return SYM_OK;
  });
}

int sym_svd_bond(sym_svd plan, const int* keep, sym_tensor* U, sym_tensor* V) {
  return sym::guard([&] {
    need(plan != nullptr && keep != nullptr && U != nullptr && V != nullptr, "plan, keep, U or V is NULL");
    auto& P = *plan->p;
    const sym::Tensor& T = P.T;
    sym::Leg bu, bv;
    bu.dir = -1;
    bv.dir = 1;
    for (size_t i = 0; i < P.blocks.size(); ++i) {
      need(keep[i] >= 0 && keep[i] <= P.blocks[i].C, "keep[b] must be in 0..min(m, n) of block b");
      if (keep[i] > 0) {
        bu.labels.push_back(P.xs[i]);
        bu.degens.push_back(keep[i]);
      }
    }
    need(!bu.labels.empty(), "at least one singular vector must be kept");
    bv.labels = bu.labels;
    bv.degens = bu.degens;
    std::vector<sym::Leg> lu(T.legs.begin(), T.legs.begin() + P.nrow), lv{bv};
    lu.push_back(bu);
    lv.insert(lv.end(), T.legs.begin() + P.nrow, T.legs.end());
    const sym::Tree tr = T.group == SYM_SU2 ? sym::Tree::comb(2) : sym::Tree{};
    sym::Tensor tu = sym::make_tensor(T.group, lu, 0, tr);
    sym::Tensor tv = sym::make_tensor(T.group, lv, T.total, tr);
    std::unordered_map<int, int> slot_of;
    for (size_t i = 0; i < P.xs.size(); ++i) slot_of[P.xs[i]] = (int)i;
    std::vector<std::vector<sym::SvdPiece>> pu(P.blocks.size()), pv(P.blocks.size());
    for (int64_t s = 0; s < tu.nsec(); ++s) {
      std::vector<int> rt(tu.pos.begin() + s * tu.rank, tu.pos.begin() + s * tu.rank + P.nrow);
      const int x = tu.label(s, P.nrow);
      const auto& r = P.rows.at(rt);
      need(r.x == x, "internal: U block outside the diagonal");
      const int b = slot_of.at(x);
      pu[b].push_back(sym::SvdPiece{tu.offs[s], (int)r.first, 0, (int)r.extent, keep[b]});
    }
    for (int64_t s = 0; s < tv.nsec(); ++s) {
      std::vector<int> ct(tv.pos.begin() + s * tv.rank + 1, tv.pos.begin() + (s + 1) * tv.rank);
      const int x = tv.label(s, 0);
      const auto& c = P.cols.at(ct);
      need(c.x == x, "internal: V block outside the diagonal");
      const int b = slot_of.at(x);
      pv[b].push_back(sym::SvdPiece{tv.offs[s], 0, (int)c.first, keep[b], (int)c.extent});
    }
    std::vector<sym::SvdPiece> all(P.tpieces);
    int ks = 0;
    for (size_t b = 0; b < P.blocks.size(); ++b) {
      auto& B = P.blocks[b];
      B.keep = keep[b];
      B.ks = ks;
      ks += keep[b];
      B.u0 = (int)all.size();
      B.nu = (int)pu[b].size();
      all.insert(all.end(), pu[b].begin(), pu[b].end());
      B.v0 = (int)all.size();
      B.nv = (int)pv[b].size();
      all.insert(all.end(), pv[b].begin(), pv[b].end());
    }
    if (!P.dry) {
      P.upload_pieces(all);
      P.upload_blocks();
    }
    P.bonded = true;
    *U = new sym_tensor_s{std::move(tu)};
    *V = new sym_tensor_s{std::move(tv)};
    return SYM_OK;
  });
}

int sym_svd_factors(sym_svd plan, int absorb, double* U, double* V, double* Sk, void* stream) {
  return sym::guard([&] {
    need(plan != nullptr && U != nullptr && V != nullptr, "plan, U or V is NULL");
    need(absorb >= 0 && absorb <= 2, "absorb must be 0, 1 or 2");
    auto& P = *plan->p;
    if (P.dry) sym::fail(SYM_ERR_UNSUPPORTED, "plan was built with SYM_PLAN_DRYRUN=1 and cannot run");
    if (!P.bonded) sym::fail(SYM_ERR_ARG, "sym_svd_bond must be called before sym_svd_factors");
    sym::svd_factor_kernel<<<(unsigned)P.blocks.size(), sym::kSvdThreads, 0, static_cast<cudaStream_t>(stream)>>>(
        P.d_blocks, P.d_pieces, P.work, P.perm, U, V, Sk, absorb);
    check_launch("svd_factor_kernel");
    return SYM_OK;
  });
}

namespace {
// keep[b] from the values' magnitudes (SVD: the singular values; eig: |lambda|)
void truncate_values(const sym::SvdPlan& P, const double* S, int64_t chi, double cutoff, int* keep) {
  need(cutoff >= 0.0, "cutoff must be >= 0");
  struct Val {
    double v;
    int b, i;
  };
  std::vector<Val> vals;
  vals.reserve(P.nsv);
  for (size_t b = 0; b < P.blocks.size(); ++b)
    for (int i = 0; i < P.blocks[b].C; ++i) {
      const double s = S[P.blocks[b].s + i];
      const double v = P.eig ? std::fabs(s) : s;
      if (!(v >= 0.0) || !std::isfinite(v))
        sym::fail(SYM_ERR_NUMERIC, P.eig ? "eigenvalues must be finite" : "singular values must be finite and >= 0");
      vals.push_back(Val{v, (int)b, i});
    }
  // descending; ties: smaller x first, then the block's own order
  std::sort(vals.begin(), vals.end(), [](const Val& a, const Val& c) {
    if (a.v != c.v) return a.v > c.v;
    return a.b != c.b ? a.b < c.b : a.i < c.i;
  });
  const double vmax = vals.empty() ? 0.0 : vals[0].v;
  for (size_t b = 0; b < P.blocks.size(); ++b) keep[b] = 0;
  int64_t n = 0;
  for (const Val& x : vals) {
    const int w = P.T.group == SYM_SU2 ? P.xs[x.b] + 1 : 1;  // dense values one value stands for
    if (chi >= 0 && n + w > chi) break;
    if (cutoff > 0.0 && x.v <= cutoff * vmax) break;
    ++keep[x.b];
    n += w;
  }
}
}  // namespace

int sym_svd_truncation(sym_svd plan, const double* S, int64_t chi, double cutoff, int* keep) {
  return sym::guard([&] {
    need(plan != nullptr && S != nullptr && keep != nullptr, "plan, S or keep is NULL");
    need(!plan->p->eig, "an eigendecomposition plan truncates with sym_eig_truncation");
    truncate_values(*plan->p, S, chi, cutoff, keep);
    return SYM_OK;
  });
}

int sym_eig_truncation(sym_svd plan, const double* lambda, int64_t chi, double cutoff, int* keep) {
  return sym::guard([&] {
    need(plan != nullptr && lambda != nullptr && keep != nullptr, "plan, lambda or keep is NULL");
    need(plan->p->eig, "not an eigendecomposition plan (sym_eig_plan)");
    truncate_values(*plan->p, lambda, chi, cutoff, keep);
    return SYM_OK;
  });
}

int sym_svd_destroy(sym_svd plan) {
  delete plan;
  return SYM_OK;
}

}  // extern "C"
