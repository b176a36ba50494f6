// Natural-gradient direction of the optimiser (Sec. 4, "Optimizer"): the loss
// gradient g = G^T w of Eq. (30) preconditioned by the damped Fisher information
// of |psi|^2 estimated from the walkers,
//   delta = (Gc^T Gc / B + lambda I)^-1 g = Gc^T (Gc Gc^T / B + lambda I)^-1 w,
// Gc = G - mean over walkers.  The second (sample-space) form needs a B x B
// system only: the Gram matrix Gc Gc^T comes from the 3 x TF32 tensor-core GEMM
// (gemm_tc.cu), the system is solved by conjugate gradients preconditioned with
// its diagonal (walkers' gradient norms span orders of magnitude near the
// nodes), in FP64 with fixed-order reductions (deterministic), and delta =
// Gc^T x is a weighted column sum.  The conjugate gradients run in one cooperative kernel whose
// CTAs meet at one grid barrier per iteration and leave the loop when the residual is small
// enough, so the call needs no host synchronisation and can be captured in a CUDA graph.
#include <float.h>
#include <math.h>

#include "common.cuh"
#include "det_util.cuh"
#include "tc_ptx.cuh"

namespace dq {
namespace {

constexpr int kNgThreads = 256;
constexpr int64_t kNgChunk = 8192;  // K extent of one Gram chunk (FP32 accumulation length)
constexpr int kNgJobs = 16;         // chunks per GEMM launch
constexpr int kNgRowWarps = 8;  // matvec: one warp per row of the Gram matrix

// FP64 adds, multiply-adds and conversions from FP32 issue at 1.7 per clock and SM, 75 times slower
// than FP32 ones: passes over G in FP64 were bound by them (one conversion, one operation per
// element: 1.6 ms for 1024 x 412,656 gradients that memory delivers in 0.25 ms).  The sums below
// (column means 1.62 -> 0.27 ms, centring 2.30 -> 0.59, the last product 1.60 -> 0.66)
// are carried as three FP32 terms instead, hi + c1 + c2: every product and every addition into hi
// and c1 keeps its rounding error exactly (TwoProd and TwoSum of Ogita, Rump, Oishi, "Accurate sum
// and dot product", SIAM J. Sci. Comput. 26, 2005), so that only c2's additions round, at 2^-72 of
// the sum: more than FP64 holds.
struct Sum3 {
  float hi, c1, c2;
  __device__ __forceinline__ void add_c1(float e) {
    const dfloat t = two_sum(c1, e);
    c1 = t.hi;
    c2 = __fadd_rn(c2, t.lo);
  }
  __device__ __forceinline__ void add(float x) {
    const dfloat t = two_sum(hi, x);
    hi = t.hi;
    add_c1(t.lo);
  }
  __device__ __forceinline__ double value() const { return (double)hi + ((double)c1 + (double)c2); }
};
// x as the three FP32 terms whose sum it is
__device__ __forceinline__ float4 split3(double x) {
  const float h = (float)x;
  const double r = x - (double)h;
  const float l = (float)r;
  return make_float4(h, l, (float)(r - (double)l), 0.f);
}

// mean[p] = (1 / B) sum_b G[b][p] in FP64, stored as the three FP32 terms that hold it exactly.  A
// CTA sums 32 columns, warp g the rows g, g + 8, ..; the warps' sums are added in FP64.
__global__ void __launch_bounds__(kNgThreads)
    ng_colmean_kernel(const float* __restrict__ G, int64_t B, int64_t P, float4* __restrict__ mean) {
  __shared__ double sh[kNgThreads / 32][32];
  const int lane = threadIdx.x % 32, g = threadIdx.x / 32;
  const int64_t p = (int64_t)blockIdx.x * 32 + lane;
  Sum3 s = {0.f, 0.f, 0.f};
  if (p < P) {
    const float* q = G + p;
#pragma unroll 8
    for (int64_t b = g; b < B; b += kNgThreads / 32) s.add(__ldg(q + b * P));
  }
  double v = s.value();
  if (!(fabsf(s.hi + (s.c1 + s.c2)) <= FLT_MAX)) {  // a sum past FP32's range (or not a number): in FP64
    v = 0;
    for (int64_t b = g; b < B; b += kNgThreads / 32) v += (double)__ldg(G + b * P + p);
  }
  sh[g][lane] = v;
  __syncthreads();
  if (g == 0 && p < P) {
    double t = 0;
#pragma unroll
    for (int k = 0; k < kNgThreads / 32; ++k) t += sh[k][lane];
    t /= (double)B;
    mean[p] = split3(t);
  }
}

// Gc[b][p] = G[b][p] - mean[p], the FP64 mean's three terms subtracted with one rounding, and row
// pitch Pp (zeros in the padding); a thread per column and 8 rows.  g - mean is formed without error
// as f.hi + f.lo + the rest, and the small parts are added with rounding to odd (the last bit tells
// that more follows), so that f.hi + them rounds as the exact difference does (Boldo, Melquiond,
// "Emulation of a FMA and correctly rounded sums: proved algorithms using rounding to odd", IEEE
// Trans. Comput. 57, 2008).  The three terms and the odd roundings take 0.59 ms for 1024 x 412,656
// gradients where two terms rounded as they come took 0.48, with up to 1.5 times the error.
constexpr int kNgCenterRows = 8;
__device__ __forceinline__ float add_odd(float a, float b) {  // a + b rounded to odd
  const float d = __fadd_rd(a, b), u = __fadd_ru(a, b);  // of two neighbours one is odd
  return (__float_as_int(d) & 1) ? d : u;
}
__device__ __forceinline__ float ng_minus_mean(float g, float4 m) {
  const dfloat d = two_sum(g, -m.x);
  const dfloat f = two_sum(d.hi, -m.y);
  return __fadd_rn(f.hi, add_odd(f.lo, add_odd(d.lo, -m.z)));
}
__global__ void ng_center_kernel(const float* __restrict__ G, const float4* __restrict__ mean, int64_t B, int64_t P,
                                 int64_t Pp, float* __restrict__ Gc) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= Pp) return;
  const int64_t b0 = (int64_t)blockIdx.y * kNgCenterRows;
  const int n = (int)min((int64_t)kNgCenterRows, B - b0);
  float* out = Gc + b0 * Pp + p;
  if (p >= P) {
    for (int k = 0; k < n; ++k) out[k * Pp] = 0.f;
    return;
  }
  const float4 m = mean[p];
  const float* in = G + b0 * P + p;
  float g[kNgCenterRows];
#pragma unroll
  for (int k = 0; k < kNgCenterRows; ++k) g[k] = k < n ? __ldg(in + k * P) : 0.f;
#pragma unroll
  for (int k = 0; k < kNgCenterRows; ++k)
    if (k < n) out[k * Pp] = ng_minus_mean(g[k], m);
}

struct CgScalars {
  double rr, rr0, rz, pAp, beta, lam;
  double tol2;  // (tol ||w||)^2
  double xback;  // 1 / the scale of x in three FP32 terms
  int iter, max_iter, done, pad;
  unsigned int counter;  // arrivals of the CTAs of the current reduction
};

// Block sum in FP64, fixed order (tree over the block's threads).
__device__ double ng_block_sum(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

// Last-arriving CTA adds the per-CTA partials in index order; returns true in that CTA
// (the sum is then in *out).
__device__ bool ng_finish(double part, double* partials, unsigned int* counter, double* out) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = part;
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __shared__ double sh[kNgThreads];
  double s = 0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) s += ((volatile double*)partials)[i];
  // fixed order: strided per thread, then the block tree
  s = ng_block_sum(s, sh);
  if (threadIdx.x == 0) {
    *out = s;
    *counter = 0;
  }
  return true;
}

// x = 0, r = w, p = z = r / diag(A), rr = rr0 = r.r, rz = r.z (one CTA)
__global__ void ng_cg_init_kernel(const float* __restrict__ w, int64_t B, const double* __restrict__ T, double* x,
                                  double* r, double* p, double* dinv, CgScalars* sc, double lam, double tol,
                                  int max_iter) {
  __shared__ double sh[kNgThreads];
  if (lam < 0) {  // relative damping: |lam| x the mean eigenvalue tr(T) / B^2 of T / B
    double tr = 0;
    for (int64_t i = threadIdx.x; i < B; i += blockDim.x) tr += T[i * B + i];
    tr = ng_block_sum(tr, sh);
    lam = -lam * tr / ((double)B * (double)B);
    if (!(lam > 0)) lam = 1.0;  // all-zero gradients: any positive damping gives delta = 0
  }
  double s = 0, sz = 0;
  for (int64_t i = threadIdx.x; i < B; i += blockDim.x) {
    const double v = (double)w[i];
    const double di = 1.0 / (T[i * B + i] / (double)B + lam);
    dinv[i] = di;
    x[i] = 0;
    r[i] = v;
    p[i] = v * di;
    s += v * v;
    sz += v * v * di;
  }
  s = ng_block_sum(s, sh);
  sz = ng_block_sum(sz, sh);
  if (threadIdx.x == 0) {
    sc->rr = s;
    sc->rr0 = s;
    sc->rz = sz;
    sc->pAp = 0;
    sc->beta = 0;
    sc->lam = lam;
    sc->tol2 = tol * tol * s;
    sc->iter = 0;
    sc->max_iter = max_iter;
    sc->done = s == 0.0 || max_iter <= 0;
    sc->counter = 0;
  }
}

// T (+)= sum of the chunks' Gram matrices, in FP64 and chunk order; mirror: only elements i >= j
// are there, and stand for (j, i) as well
__global__ void ng_gram_add_kernel(const float* __restrict__ Tc, int n_chunks, int64_t B, int first, int mirror,
                                   double* __restrict__ T) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, BB = B * B;
  if (e >= BB) return;
  const int64_t i = e / B, j = e - (e / B) * B;
  if (mirror && j > i) return;
  double s = first ? 0.0 : T[e];
  for (int c = 0; c < n_chunks; ++c) s += (double)Tc[(int64_t)c * BB + e];
  T[e] = s;
  if (mirror) T[j * B + i] = s;
}

// T = (T + T^T) / 2: the 3 x TF32 products of T_ij and T_ji drop different low-order
// terms, and conjugate gradients need an exactly symmetric matrix
__global__ void ng_symmetrize_kernel(double* T, int64_t B) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * B) return;
  const int64_t i = e / B, j = e - (e / B) * B;
  if (j <= i) return;
  const double a = 0.5 * (T[i * B + j] + T[j * B + i]);
  T[i * B + j] = a;
  T[j * B + i] = a;
}

// Ap = T p / B + lam p and pAp = p . Ap; one warp per row of T (B x B, FP64)
__global__ void __launch_bounds__(32 * kNgRowWarps)
    ng_cg_matvec_kernel(const double* __restrict__ T, int64_t B, const double* __restrict__ p, double* __restrict__ Ap,
                        CgScalars* sc, double* partials) {
  if (((volatile CgScalars*)sc)->done) return;
  const int lane = threadIdx.x % 32, wq = threadIdx.x / 32;
  const int64_t i = (int64_t)blockIdx.x * kNgRowWarps + wq;
  double part = 0;
  if (i < B) {
    const double* Ti = T + i * B;
    double s = 0;
    for (int64_t j = lane; j < B; j += 32) s += Ti[j] * p[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double a = s / (double)B + sc->lam * p[i];
    if (lane == 0) Ap[i] = a;
    part = lane == 0 ? a * p[i] : 0.0;
  }
  __shared__ double sh[32 * kNgRowWarps];
  const double cta = ng_block_sum(part, sh);
  ng_finish(cta, partials, &sc->counter, &sc->pAp);
}

// alpha = rz / pAp; x += alpha p; r -= alpha Ap; z = r / diag(A); rr' = r.r, rz' = r.z;
// beta = rz' / rz; convergence flag (on ||r|| / ||w||)
__global__ void ng_cg_update_kernel(int64_t B, double* x, double* r, double* z, const double* __restrict__ dinv,
                                    const double* __restrict__ p, const double* __restrict__ Ap, CgScalars* sc,
                                    double* partials, double* partials2) {
  volatile CgScalars* vs = sc;
  if (vs->done) return;
  const double alpha = vs->pAp > 0 ? vs->rz / vs->pAp : 0.0;
  double part = 0, partz = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < B; i += (int64_t)gridDim.x * blockDim.x) {
    x[i] += alpha * p[i];
    const double ri = r[i] - alpha * Ap[i];
    const double zi = ri * dinv[i];
    r[i] = ri;
    z[i] = zi;
    part += ri * ri;
    partz += ri * zi;
  }
  __shared__ double sh[kNgThreads];
  const double cta = ng_block_sum(part, sh);
  const double ctaz = ng_block_sum(partz, sh);
  if (threadIdx.x == 0) partials2[blockIdx.x] = ctaz;  // published before this CTA's arrival in ng_finish
  double rr_new = 0;
  if (ng_finish(cta, partials, &sc->counter, &rr_new)) {
    __shared__ double shz[kNgThreads];
    double s = 0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) s += ((volatile double*)partials2)[i];
    const double rz_new = ng_block_sum(s, shz);
    if (threadIdx.x == 0) {
      const int it = vs->iter;
      sc->beta = vs->rz > 0 ? rz_new / vs->rz : 0.0;
      sc->rz = rz_new;
      sc->rr = rr_new;
      sc->iter = it + 1;
      sc->done = (rr_new <= vs->tol2 || it + 1 >= vs->max_iter || !(vs->pAp > 0)) ? 1 : 0;
    }
  }
}

// p = z + beta p
__global__ void ng_cg_direction_kernel(int64_t B, const double* __restrict__ z, double* p, const CgScalars* sc) {
  const volatile CgScalars* vs = sc;
  if (vs->done) return;
  const double beta = vs->beta;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < B; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = z[i] + beta * p[i];
}

// ---------------------------------------------------------------------------
// All iterations in one cooperative kernel (ng_cg_init_kernel sets the system up).
// What bounds an iteration: the matvec's B^2 FP64 multiply-adds (1.7 per clock
// and SM: 2 us at B = 1024, 33 us at 4096) and the trips to the other SMs, not
// memory (T stays in L2, or in L1 up to B of about 1200).  So every CTA owns rpc
// rows of T, and keeps p, r and 1 / diag of the whole system in shared memory:
// it publishes its rows of A p, meets the others at one grid barrier, and then
// forms pAp, r, rr, rz and the next p of all walkers by itself, as every other
// CTA does.  That spends 6 B redundant multiply-adds per CTA instead of a second
// barrier with its reduction, and every CTA takes the same decisions from the
// same bits.  The sums are added in the order of the kernels above, which serve
// the systems that do not fit here, with their roundings: with either form forced,
// systems of 2 to 2000 walkers gave the same solutions and iteration counts bit for bit.
// Against those (three launches per iteration, always max_iter of them; 17.4 +
// 9.9 + 3.1 us each at B = 1024 until the residual is small) the call on 1024
// walkers x 412,656 parameters took 15.2 ms instead of 17.7, and a LiH training
// step of 1024 walkers 8.0 ms instead of 10.7; 200 iterations at B = 1024 are 2.1 ms.
// The barrier's wait is bounded; on a timeout every CTA leaves and
// DQ_FLAG_TIMEOUT is set.
// ---------------------------------------------------------------------------
constexpr int kCgThreads = 512;
constexpr int kCgWarps = kCgThreads / 32;
constexpr int kCgMaxGroups = 64;                  // groups of kNgThreads walkers: B <= 16384
constexpr size_t kCgStatics = 4096;               // kept for the static arrays

inline size_t ng_solve_smem(int64_t B) { return (size_t)3 * B * sizeof(double); }

// ng_block_sum's tree over kNgThreads = 256 values by one warp, lane l holding the values
// l + 32 m in v[m]; every lane returns the sum.
__device__ __forceinline__ double cg_tree256(double (&v)[8]) {
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] += v[m + 4];
  v[0] += v[2];
  v[1] += v[3];
  double s = v[0] + v[1];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
// The same over n <= 256 values of shared memory (zeros after them).
__device__ __forceinline__ double cg_tree256(const double* a, int n, int lane) {
  double v[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) v[m] = lane + 32 * m < n ? a[lane + 32 * m] : 0.0;
  return cg_tree256(v);
}

__global__ void __launch_bounds__(kCgThreads, 1)
    ng_cg_solve_kernel(const double* __restrict__ T, int B, int rpc, const double* __restrict__ r_in,
                       const double* __restrict__ p_in, const double* __restrict__ dinv_in, double* Ap,
                       double* __restrict__ x, CgScalars* sc, unsigned int* arrivals, unsigned int* status) {
  extern __shared__ __align__(16) unsigned char cg_smem[];
  double* p = reinterpret_cast<double*>(cg_smem);  // [B] direction
  double* r = p + B;                               // [B] residual
  double* dinv = r + B;                            // [B] 1 / diagonal
  __shared__ double s_pap[kNgThreads], s_rr[kCgMaxGroups], s_rz[kCgMaxGroups], s_scal[5];
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
  const int row0 = blockIdx.x * rpc, row1 = min(B, row0 + rpc);
  const int n_oct = (B + kNgRowWarps - 1) / kNgRowWarps;  // groups of eight rows (ng_cg_matvec_kernel's CTAs)
  const int n_grp = (B + kNgThreads - 1) / kNgThreads;    // groups of 256 walkers (ng_cg_update_kernel's CTAs)
  static_assert(kNgRowWarps == 8 && kNgThreads == 256, "cg_tree256 and the octet sums follow these sizes");
  for (int i = tid; i < B; i += kCgThreads) {
    r[i] = r_in[i];
    p[i] = p_in[i];
    dinv[i] = dinv_in[i];
  }
  const double lam = sc->lam, tol2 = sc->tol2;
  const int max_iter = sc->max_iter;
  double rr = sc->rr, rz = sc->rz;
  bool done = sc->done != 0;
  double xi = 0;  // x of walker row0 + tid (tid < row1 - row0)
  int it = 0;
  __syncthreads();
  for (; !done; ++it) {
    double* Ab = Ap + (size_t)(it & 1) * B;  // two buffers: a CTA may still read the last iteration's
    for (int i = row0 + warp; i < row1; i += kCgWarps) {
      const double* Ti = T + (int64_t)i * B;
      double s = 0;
#pragma unroll 8
      for (int j = lane; j < B; j += 32) s = fma(Ti[j], p[j], s);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) __stcg(Ab + i, fma(lam, p[i], s / (double)B));
    }
    __syncthreads();
    if (tid == 0) {  // grid barrier: all rows of A p published
      __threadfence();
      atomicAdd(arrivals, 1u);
      const unsigned int target = (unsigned int)(it + 1) * gridDim.x;
      const long long t0 = clock64();
      int ok = 1;
      while ((int)(*(volatile unsigned int*)arrivals - target) < 0)
        if (clock64() - t0 > tcp::kWaitCycles) {
          ok = 0;
          break;
        }
      __threadfence();
      s_ok = ok;
    }
    __syncthreads();
    if (!s_ok) {
      if (tid == 0) atomicOr(status, (unsigned)DQ_FLAG_TIMEOUT);
      break;
    }
    if (tid < kNgThreads) {  // p . A p: octets of rows, strided over 256 threads, then the tree
      double s = 0;
      for (int c = tid; c < n_oct; c += kNgThreads) {
        double t[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int i = c * 8 + q;
          t[q] = i < B ? __ldcg(Ab + i) * p[i] : 0.0;
        }
        s += ((t[0] + t[4]) + (t[2] + t[6])) + ((t[1] + t[5]) + (t[3] + t[7]));
      }
      s_pap[tid] = s;
    }
    __syncthreads();
    // sums of sums and the scalars by one warp: an FP64 instruction holds the SM's pipe for 19 clocks
    // whatever its lanes do, so that all 16 warps doing them cost 8 us per iteration
    if (warp == 0) {
      const double v = cg_tree256(s_pap, kNgThreads, lane);
      if (lane == 0) {
        s_scal[0] = v;
        s_scal[1] = v > 0 ? rz / v : 0.0;
      }
    }
    __syncthreads();
    const double pAp = s_scal[0], alpha = s_scal[1];
    if (tid < row1 - row0) xi = fma(alpha, p[row0 + tid], xi);
    for (int g = warp; g < n_grp; g += kCgWarps) {  // r -= alpha A p; the group's r.r and r.z
      double vr[8], vz[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int i = g * kNgThreads + lane + 32 * m;
        vr[m] = vz[m] = 0;
        if (i < B) {
          const double ri = fma(-alpha, __ldcg(Ab + i), r[i]);
          r[i] = ri;
          vr[m] = ri * ri;
          vz[m] = ri * (ri * dinv[i]);
        }
      }
      const double a = cg_tree256(vr), b = cg_tree256(vz);
      if (lane == 0) {
        s_rr[g] = a;
        s_rz[g] = b;
      }
    }
    __syncthreads();
    if (warp == 0) {
      const double a = cg_tree256(s_rr, n_grp, lane), b = cg_tree256(s_rz, n_grp, lane);
      if (lane == 0) {
        s_scal[2] = a;
        s_scal[3] = b;
        s_scal[4] = rz > 0 ? b / rz : 0.0;
      }
    }
    __syncthreads();
    rr = s_scal[2];
    rz = s_scal[3];
    const double beta = s_scal[4];
    done = rr <= tol2 || it + 1 >= max_iter || !(pAp > 0);
    for (int i = tid; i < B; i += kCgThreads) p[i] = fma(beta, p[i], r[i] * dinv[i]);
    __syncthreads();
  }
  if (tid < row1 - row0) x[row0 + tid] = xi;
  if (blockIdx.x == 0 && tid == 0) {
    sc->rr = rr;
    sc->iter = it;
  }
}

// The coefficients of ng_apply_kernel: x as three FP32 terms, scaled by the power of two that takes
// the largest |x| to 2^40: its products with FP32 gradients then neither overflow (gradients past 2^64
// already overflow the Gram matrix's FP32 sums) nor lose their rounding errors to underflow, whatever
// the size of x.  Every CTA finds the largest exponent by itself.
constexpr int kNgScaleExp = 40;
__global__ void __launch_bounds__(kNgThreads)
    ng_split_x_kernel(const double* __restrict__ x, int64_t B, CgScalars* sc, float4* __restrict__ x3) {
  __shared__ int s_e;
  if (threadIdx.x == 0) s_e = 0;
  __syncthreads();
  int e = 0;
  for (int64_t i = threadIdx.x; i < B; i += blockDim.x) e = max(e, (__double2hiint(x[i]) >> 20) & 0x7ff);
  atomicMax(&s_e, e);
  __syncthreads();
  e = max(s_e, kNgScaleExp + 1);              // biased exponent (clamped: the scale stays below 2^1023)
  if (e == 0x7ff) e = 1023 + kNgScaleExp;     // not finite: no scale
  const double up = __hiloint2double((2 * 1023 + kNgScaleExp - e) << 20, 0);
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B) x3[b] = split3(x[b] * up);
  if (b == 0) sc->xback = __hiloint2double((e - kNgScaleExp) << 20, 0);
}

// delta[p] = sum_b x_b Gc[b][p] (fixed order): a CTA 32 columns, warp g the rows g, g + 8, ..
__global__ void __launch_bounds__(kNgThreads)
    ng_apply_kernel(const float* __restrict__ Gc, int64_t B, int64_t P, int64_t Pp, const float4* __restrict__ x3,
                    const CgScalars* __restrict__ sc, float* __restrict__ delta) {
  __shared__ double sh[kNgThreads / 32][32];
  const int lane = threadIdx.x % 32, g = threadIdx.x / 32;
  const int64_t q = (int64_t)blockIdx.x * 32 + lane;
  Sum3 s = {0.f, 0.f, 0.f};
  if (q < P) {
#pragma unroll 8
    for (int64_t b = g; b < B; b += kNgThreads / 32) {
      const float v = __ldg(Gc + b * Pp + q);
      const float4 c = __ldg(x3 + b);
      const float p = __fmul_rn(c.x, v);
      const float e = __fmaf_rn(c.x, v, -p);
      const float p2 = __fmul_rn(c.y, v);
      s.add(p);
      s.add_c1(e);
      s.add_c1(p2);
      s.c2 = __fadd_rn(s.c2, __fmaf_rn(c.z, v, __fmaf_rn(c.y, v, -p2)));
    }
  }
  sh[g][lane] = s.value();
  __syncthreads();
  if (g == 0 && q < P) {
    double t = 0;
#pragma unroll
    for (int k = 0; k < kNgThreads / 32; ++k) t += sh[k][lane];
    delta[q] = (float)(t * sc->xback);
  }
}

__global__ void ng_stats_kernel(const CgScalars* sc, double* stats) {
  stats[0] = (double)sc->iter;
  stats[1] = sc->rr0 > 0 ? sqrt(sc->rr / sc->rr0) : 0.0;
  stats[2] = sqrt(sc->rr0);
  stats[3] = sc->lam;
}

inline unsigned ng_blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }
inline size_t ng_align(size_t x) { return (x + 255) / 256 * 256; }

// Launches the one-kernel iteration; false where it does not serve the system (its vectors exceed
// shared memory, or the device cannot hold the grid at once), *e: a launch error.
bool ng_solve(const double* T, int64_t B, const double* r, const double* p, const double* dinv, double* Ap, double* x,
              CgScalars* sc, unsigned int* arrivals, unsigned int* status, cudaStream_t s, cudaError_t* e) {
  *e = cudaSuccess;
  const size_t smem = ng_solve_smem(B);
  if (smem > kMaxSmem - kCgStatics) return false;  // B > 9514
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  *e = allow_smem(ng_cg_solve_kernel, smem, kCgStatics);
  if (*e == cudaSuccess)
    *e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ng_cg_solve_kernel, kCgThreads, smem);
  if (*e != cudaSuccess) return true;
  int b = (int)B, rpc = (int)((B + sms - 1) / sms);  // rows per CTA, spread over every SM
  if (per_sm < 1 || rpc > kCgThreads) return false;
  const unsigned grid = ng_blocks(B, rpc);
  *e = cudaMemsetAsync(arrivals, 0, sizeof(unsigned int), s);
  if (*e != cudaSuccess) return true;
  void* args[] = {&T, &b, &rpc, &r, &p, &dinv, &Ap, &x, &sc, &arrivals, &status};
  *e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(ng_cg_solve_kernel), dim3(grid), dim3(kCgThreads),
                                   args, smem, s);
  return true;
}

}  // namespace

// Workspace layout of natgrad_run (bytes), for B walkers and P parameters.
size_t natgrad_workspace(int64_t B, int64_t P) {
  const int64_t Pp = (P + 3) / 4 * 4;
  const int64_t mv_ctas = (B + kNgRowWarps - 1) / kNgRowWarps;
  size_t o = 0;
  o += ng_align((size_t)P * 16);                // mean in three FP32 terms
  o += ng_align((size_t)B * Pp * 4);            // Gc
  o += ng_align((size_t)kNgJobs * B * B * 4);  // Gram matrices of the chunks of one launch
  o += ng_align((size_t)B * B * 8);             // Gram matrix (FP64)
  o += 5 * ng_align((size_t)B * 8);             // x, r, p, z, 1 / diag
  o += ng_align((size_t)2 * B * 8);             // Ap, two buffers
  o += 2 * ng_align((size_t)(mv_ctas + 1024) * 8);  // partials
  o += ng_align(sizeof(CgScalars));
  o += ng_align(sizeof(unsigned int));          // arrivals at the solve's grid barrier
  o += ng_align((size_t)B * 16);                // x in three FP32 terms
  return o;
}

cudaError_t natgrad_run(const float* G, const float* w, int64_t B, int64_t P, double lam, int max_iter, double tol,
                        float* delta, double* stats, unsigned char* ws, unsigned int* status, cudaStream_t s) {
  const int64_t Pp = (P + 3) / 4 * 4;
  const int64_t mv_ctas = (B + kNgRowWarps - 1) / kNgRowWarps;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    unsigned char* q = ws + o;
    o += ng_align(bytes);
    return q;
  };
  float4* mean = reinterpret_cast<float4*>(take((size_t)P * 16));
  float* Gc = reinterpret_cast<float*>(take((size_t)B * Pp * 4));
  float* Tc = reinterpret_cast<float*>(take((size_t)kNgJobs * B * B * 4));
  double* T = reinterpret_cast<double*>(take((size_t)B * B * 8));
  double* x = reinterpret_cast<double*>(take((size_t)B * 8));
  double* r = reinterpret_cast<double*>(take((size_t)B * 8));
  double* p = reinterpret_cast<double*>(take((size_t)B * 8));
  double* Ap = reinterpret_cast<double*>(take((size_t)2 * B * 8));
  double* z = reinterpret_cast<double*>(take((size_t)B * 8));
  double* dinv = reinterpret_cast<double*>(take((size_t)B * 8));
  double* partials = reinterpret_cast<double*>(take((size_t)(mv_ctas + 1024) * 8));
  double* partials2 = reinterpret_cast<double*>(take((size_t)(mv_ctas + 1024) * 8));
  CgScalars* sc = reinterpret_cast<CgScalars*>(take(sizeof(CgScalars)));
  unsigned int* arrivals = reinterpret_cast<unsigned int*>(take(sizeof(unsigned int)));
  float4* x3 = reinterpret_cast<float4*>(take((size_t)B * 16));

  ng_colmean_kernel<<<ng_blocks(P, 32), kNgThreads, 0, s>>>(G, B, P, mean);
  const dim3 cgrid(ng_blocks(Pp, kNgThreads), ng_blocks(B, kNgCenterRows));
  ng_center_kernel<<<cgrid, kNgThreads, 0, s>>>(G, mean, B, P, Pp, Gc);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // T = Gc Gc^T (B x B), in chunks of kNgChunk columns (each accumulated in FP32 on the tensor
  // cores), the chunks added in FP64.  Both operands are split in shared memory.  Half the tiles
  // (row >= column) and as many chunks per launch as leave the last wave of its tiles fullest:
  // 1024 walkers have 32 tiles per chunk, 20 in the triangle; 51 chunks are 13 waves of 152 CTAs in
  // launches of 16 chunks, 7 as triangles in launches of 15.  The triangle is taken where it saves
  // a wave; where it does not (a few chunks fill one wave either way) both halves are computed and
  // averaged.  (5.3 ms of launches with W split in memory first, 1.2 ms more, are 2.8 ms so.)
  // The triangle costs no accuracy: T_ij and T_ji carry the same error of the FP32 sums, so that their
  // average does not reduce it (largest and rms errors against 64 bits equal to four digits for N2, LiH
  // and H2O gradients and random ones; N2, 1024 walkers: 7.16e-5 and 4.70e-5 of sqrt(T_ii T_jj)).
  const int64_t n_chunks = (Pp + kNgChunk - 1) / kNgChunk;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  bool tri = false;
  int per_launch = 0;
  int64_t waves = 0;
  for (int t = 0; t < 2; ++t) {
    const int64_t tiles = gemm_tf32x3_tiles(B, B, t == 1);
    for (int nj = kNgJobs; nj >= 1; --nj) {
      const int64_t rest = n_chunks % nj;
      const int64_t n = n_chunks / nj * ((nj * tiles + sms - 1) / sms) + (rest * tiles + sms - 1) / sms;
      if (per_launch == 0 || n < waves) {
        waves = n;
        per_launch = nj;
        tri = t == 1;
      }
    }
  }
  for (int64_t c0 = 0; c0 < n_chunks; c0 += per_launch) {
    T3JobDesc jd[kNgJobs];
    int nj = 0;
    for (int64_t c = c0; c < n_chunks && nj < per_launch; ++c, ++nj) {
      const int64_t k0 = c * kNgChunk, kc = Pp - k0 < kNgChunk ? Pp - k0 : kNgChunk;
      jd[nj] = T3JobDesc{Gc + k0, B, 1, 0, (int)kc, Pp, Gc + k0, nullptr, (int)B, nullptr, 1,
                         Tc + (int64_t)nj * B * B, B, 0, false, Pp, true, tri};
    }
    e = gemm_tf32x3_tc_jobs(jd, nj, status, s);
    if (e != cudaSuccess) return e;
    ng_gram_add_kernel<<<ng_blocks(B * B, kNgThreads), kNgThreads, 0, s>>>(Tc, nj, B, c0 == 0 ? 1 : 0, tri ? 1 : 0, T);
  }
  if (!tri) ng_symmetrize_kernel<<<ng_blocks(B * B, kNgThreads), kNgThreads, 0, s>>>(T, B);
  ng_cg_init_kernel<<<1, kNgThreads, 0, s>>>(w, B, T, x, r, p, dinv, sc, lam, tol, max_iter);
  if (!ng_solve(T, B, r, p, dinv, Ap, x, sc, arrivals, status, s, &e)) {
    // systems whose vectors do not fit one CTA's shared memory: three launches per iteration
    const unsigned up_ctas = ng_blocks(B, kNgThreads) < 1024 ? ng_blocks(B, kNgThreads) : 1024;
    for (int it = 0; it < max_iter; ++it) {
      ng_cg_matvec_kernel<<<(unsigned)mv_ctas, 32 * kNgRowWarps, 0, s>>>(T, B, p, Ap, sc, partials);
      ng_cg_update_kernel<<<up_ctas, kNgThreads, 0, s>>>(B, x, r, z, dinv, p, Ap, sc, partials, partials2);
      ng_cg_direction_kernel<<<up_ctas, kNgThreads, 0, s>>>(B, z, p, sc);
    }
  }
  if (e != cudaSuccess) return e;
  ng_split_x_kernel<<<ng_blocks(B, kNgThreads), kNgThreads, 0, s>>>(x, B, sc, x3);
  ng_apply_kernel<<<ng_blocks(P, 32), kNgThreads, 0, s>>>(Gc, B, P, Pp, x3, sc, delta);
  if (stats) ng_stats_kernel<<<1, 1, 0, s>>>(sc, stats);
  return cudaGetLastError();
}

}  // namespace dq

namespace dq {
namespace {
// ||delta||^2 in FP64: per-CTA partials, the last CTA adds them in index order and
// sets the step scale s = min(1, max_norm / (lr ||delta||)) (no limit when max_norm <= 0)
__global__ void ng_norm_kernel(const float* __restrict__ d, int64_t P, double lr, double max_norm,
                               double* partials, unsigned int* counter, double* out) {
  double part = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = (double)d[i];
    part += v * v;
  }
  __shared__ double sh[kNgThreads];
  const double cta = ng_block_sum(part, sh);
  double ss = 0;
  if (ng_finish(cta, partials, counter, &ss) && threadIdx.x == 0) {
    const double nrm = sqrt(ss);
    out[0] = nrm;
    out[1] = (max_norm > 0 && lr * nrm > max_norm) ? max_norm / (lr * nrm) : 1.0;
  }
}

// theta -= lr * s * delta
template <class T>
__global__ void ng_update_kernel(T* __restrict__ theta, const T* __restrict__ d, int64_t P, double lr,
                                 const double* __restrict__ nrm) {
  const double step = lr * nrm[1];
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < P; i += (int64_t)gridDim.x * blockDim.x)
    theta[i] = (T)((double)theta[i] - step * (double)d[i]);
}
}  // namespace

size_t param_update_workspace() { return 1024 * 8 + 256; }

template <class T>
cudaError_t param_update_run(T* theta, const T* delta, int64_t P, double lr, double max_norm, double* stats,
                             unsigned char* ws, cudaStream_t s) {
  double* partials = reinterpret_cast<double*>(ws);
  unsigned int* counter = reinterpret_cast<unsigned int*>(ws + 1024 * 8);
  const unsigned ctas = ng_blocks(P, kNgThreads) < 1024 ? ng_blocks(P, kNgThreads) : 1024;
  cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  if constexpr (sizeof(T) == 4) {
    ng_norm_kernel<<<ctas, kNgThreads, 0, s>>>(delta, P, lr, max_norm, partials, counter, stats);
  } else {
    return cudaErrorInvalidValue;  // FP32 modes only
  }
  ng_update_kernel<T><<<ctas, kNgThreads, 0, s>>>(theta, delta, P, lr, stats);
  return cudaGetLastError();
}
template cudaError_t param_update_run<float>(float*, const float*, int64_t, double, double, double*, unsigned char*,
                                             cudaStream_t);

}  // namespace dq
