// Jet messages of Eq. 17 for constant node channels (layer 0 on spin embeddings, FP32 modes): z_j
// is one of two vectors and has no derivatives, so that of m_i^t[c] = nu_t sum_j w_ij z_j only
// these channels are non-zero:
//   value        sum_j w_ij z_j
//   sender e, x  -w'_ie u_ie,x z_e             (in the slot of e's spin block only)
//   own, x       sum_j w'_ij u_ij,x z_j
//   Laplacian    sum_j (2 w''_ij + 4 w'_ij / d_ij) z_j
// and the electron-nucleus messages on the value, own-coordinate and Laplacian channels.  Every
// other element is written as zero.  The general kernel (forward.cu) forms these with the tables
// and the contraction loops of varying z: 1.76 ms for 152 C4H4 walkers at 256 features, against
// 0.1 ms for the bytes that it writes.  Here a warp owns a receiver and V features per lane, reads
// the filter jets of its edges once, in sender order, and writes a sender's three rows as it goes.
// All messages of 333 C4H4 walkers (four layers, FP32): 7.5 -> 4.1 ms; of 1024 in BF16 mode 22.6 ->
// 11.9; of the two LiH layers of 1024 walkers 0.20 -> 0.12.
// Sums run in the general kernel's order and with its roundings: the same bits (tested; a handle's
// message-kernel mode 1 takes the general kernel here too).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "common.cuh"

namespace dq {
namespace {

constexpr int kMCWarps = 8;

struct MCArgs {
  const float* z0;     // [2][D] node channels of the two spins
  const float* ew;     // [Bc][E][3][D] filter jets w, dw/dd, d2w/dd2
  const float* geo;    // [Bc][E][4] distance and unit vector of every edge
  const float* Y;      // [M][D] nucleus embeddings of the layer
  const int* pair_of;  // [N][N] edge of (i, j), -1 on the diagonal
  void* msg;           // [Bc][N][C][3D], or with msg5 [Bc][N][C][2D] (FwdBuffers)
  void* msg5;          // [Bc][N][5][3D] or nullptr
  int N, n_up, M, C, D, E, n_ee;
};

template <int V>
struct Feat {
  float v[V];
};
template <int V>
__device__ __forceinline__ Feat<V> load_f(const float* p) {
  Feat<V> r;
  if constexpr (V == 4) {
    const float4 x = __ldg(reinterpret_cast<const float4*>(p));
    r.v[0] = x.x, r.v[1] = x.y, r.v[2] = x.z, r.v[3] = x.w;
  } else if constexpr (V == 2) {
    const float2 x = __ldg(reinterpret_cast<const float2*>(p));
    r.v[0] = x.x, r.v[1] = x.y;
  } else {
    r.v[0] = __ldg(p);
  }
  return r;
}
template <int V>
__device__ __forceinline__ void store_f(float* p, const Feat<V>& r) {
  if constexpr (V == 4) *reinterpret_cast<float4*>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
  else if constexpr (V == 2) *reinterpret_cast<float2*>(p) = make_float2(r.v[0], r.v[1]);
  else *p = r.v[0];
}
template <int V>
__device__ __forceinline__ void store_f(__nv_bfloat16* p, const Feat<V>& r) {
  if constexpr (V == 1) {
    *p = __float2bfloat16_rn(r.v[0]);
  } else {
    __nv_bfloat162 h[V / 2];
#pragma unroll
    for (int k = 0; k < V / 2; ++k) h[k] = __floats2bfloat162_rn(r.v[2 * k], r.v[2 * k + 1]);
    if constexpr (V == 4) *reinterpret_cast<uint2*>(p) = *reinterpret_cast<const uint2*>(h);
    else *reinterpret_cast<__nv_bfloat162*>(p) = h[0];
  }
}
template <int V>
__device__ __forceinline__ Feat<V> scaled(const Feat<V>& r, float s) {
  Feat<V> o;
#pragma unroll
  for (int k = 0; k < V; ++k) o.v[k] = r.v[k] * s;
  return o;
}

template <int V, class TO>
__global__ void __launch_bounds__(kMCWarps * 32) messages_const_kernel(const __grid_constant__ MCArgs a) {
  __shared__ float4 s_u[kMCWarps][kMaxElec];  // u_ij and 1 / d_ij of the warp's receiver
  __shared__ int s_p[kMCWarps][kMaxElec];     // its edges
  const int N = a.N, C = a.C, D = a.D, M = a.M, n_up = a.n_up, n_ee = a.n_ee;
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int64_t b = blockIdx.x;
  const int f = blockIdx.y * 32 * V + lane * V;
  const float* ew = a.ew + b * (int64_t)a.E * 3 * D + f;
  const float* geo = a.geo + b * (int64_t)a.E * 4;
  const int mp = (a.msg5 ? 2 : 3) * D;
  TO* msg = static_cast<TO*>(a.msg) + b * (int64_t)N * C * mp + f;
  TO* msg5 = a.msg5 ? static_cast<TO*>(a.msg5) + b * (int64_t)N * 15 * D + f : nullptr;
  const Feat<V> zu = load_f<V>(a.z0 + f), zd = load_f<V>(a.z0 + D + f);
  const Feat<V> zero = {};
  const float nuM = 1.f / (float)M;
  for (int i = warp; i < N; i += kMCWarps) {
    for (int j = lane; j < N; j += 32) {
      const int p = a.pair_of[i * N + j];
      float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j != i) {
        const float4 g = *reinterpret_cast<const float4*>(geo + (int64_t)p * 4);
        const float sg = i < j ? 1.f : -1.f;
        u = make_float4(sg * g.y, sg * g.z, sg * g.w, 1.f / g.x);
      }
      s_u[warp][j] = u;
      s_p[warp][j] = p;
    }
    __syncwarp();
    const bool up = i < n_up;
    const int n_same = up ? n_up : N - n_up, n_opp = N - n_same;
    const float nu_same = 1.f / (float)(n_same - 1 > 1 ? n_same - 1 : 1), nu_opp = 1.f / (float)(n_opp > 1 ? n_opp : 1);
    TO* mi = msg + (int64_t)i * C * mp;
    // the row of the receiver's value (slot 0), own-coordinate (1, 2, 3) or Laplacian (4) channel
    auto special = [&](int slot) {
      const int c = slot == 0 ? 0 : slot == 4 ? C - 1 : 3 * i + slot;
      return msg5 ? msg5 + ((int64_t)i * 5 + slot) * 3 * D : mi + (int64_t)c * mp;
    };
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {  // spin-up, then spin-down senders
      const int j0 = h == 0 ? 0 : n_up, j1 = h == 0 ? n_up : N;
      const bool same = up == (h == 0);
      const float nu = same ? nu_same : nu_opp;
      const int slot = same ? 0 : D, other = same ? D : 0;
      const Feat<V> z = h == 0 ? zu : zd;
      Feat<V> val = {}, own[3] = {}, lap = {};
#pragma unroll 4
      for (int j = j0; j < j1; ++j) {
        if (j == i) continue;
        const float* w = ew + (int64_t)s_p[warp][j] * 3 * D;
        const Feat<V> w0 = load_f<V>(w), w1 = load_f<V>(w + D), w2 = load_f<V>(w + 2 * D);
        const float4 u = s_u[warp][j];
        const float ux[3] = {u.x, u.y, u.z};
        TO* o = mi + (int64_t)(1 + 3 * j) * mp;
#pragma unroll
        for (int k = 0; k < V; ++k) {
          val.v[k] += w0.v[k] * z.v[k];
          const float t = __fmul_rn(__fmaf_rn(4.f * w1.v[k], u.w, 2.f * w2.v[k]), z.v[k]);
          lap.v[k] = __fadd_rn(lap.v[k], t);
        }
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          Feat<V> m;
#pragma unroll
          for (int k = 0; k < V; ++k) {
            const float wu = w1.v[k] * ux[x];
            own[x].v[k] += wu * z.v[k];
            m.v[k] = __fmul_rn(-(wu * z.v[k]), nu);
          }
          store_f<V>(o + (int64_t)x * mp + slot, m);
          store_f<V>(o + (int64_t)x * mp + other, zero);
          if (msg5 == nullptr) store_f<V>(o + (int64_t)x * mp + 2 * D, zero);
        }
      }
      store_f<V>(special(0) + slot, scaled<V>(val, nu));
#pragma unroll
      for (int x = 0; x < 3; ++x) store_f<V>(special(1 + x) + slot, scaled<V>(own[x], nu));
      store_f<V>(special(4) + slot, scaled<V>(lap, nu));
    }
    Feat<V> nv = {}, nx[3] = {}, nl = {};
#pragma unroll 2
    for (int I = 0; I < M; ++I) {
      const int e = n_ee + i * M + I;
      const float* w = ew + (int64_t)e * 3 * D;
      const float4 g = *reinterpret_cast<const float4*>(geo + (int64_t)e * 4);
      const Feat<V> w0 = load_f<V>(w), w1 = load_f<V>(w + D), w2 = load_f<V>(w + 2 * D), y = load_f<V>(a.Y + (int64_t)I * D + f);
#pragma unroll
      for (int k = 0; k < V; ++k) {
        nv.v[k] += w0.v[k] * y.v[k];
        nx[0].v[k] += w1.v[k] * g.y * y.v[k];
        nx[1].v[k] += w1.v[k] * g.z * y.v[k];
        nx[2].v[k] += w1.v[k] * g.w * y.v[k];
        nl.v[k] += (w2.v[k] + 2.f * w1.v[k] / g.x) * y.v[k];
      }
    }
    store_f<V>(special(0) + 2 * D, scaled<V>(nv, nuM));
#pragma unroll
    for (int x = 0; x < 3; ++x) store_f<V>(special(1 + x) + 2 * D, scaled<V>(nx[x], nuM));
    store_f<V>(special(4) + 2 * D, scaled<V>(nl, nuM));
    __syncwarp();
  }
}

template <int V>
cudaError_t launch_mc(const MCArgs& a, int64_t Bc, bool bf16_out, cudaStream_t s) {
  const dim3 grid((unsigned)Bc, (unsigned)(a.D / (32 * V)));
  if (bf16_out) messages_const_kernel<V, __nv_bfloat16><<<grid, kMCWarps * 32, 0, s>>>(a);
  else messages_const_kernel<V, float><<<grid, kMCWarps * 32, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_messages_const(const dq_handle_s& h, const FwdDims& d, const float* params, int l, const float* z0,
                                  const float* ew, const float* geo, void* msg, void* msg5, bool bf16_out,
                                  cudaStream_t s) {
  if (d.Bc <= 0) return cudaSuccess;
  // the nucleus embeddings may start anywhere in the parameter vector: vectors of features only
  // where they are aligned
  const float* Y = params + h.off.layer[l].Y;
  const MCArgs a{z0, ew, geo, Y, h.d_pair_of, msg, msg5, d.N, d.n_up, d.M, d.C, d.D, h.edges.n_all, h.edges.n_ee};
  if (d.D % 128 == 0 && (uintptr_t)Y % 16 == 0) return launch_mc<4>(a, d.Bc, bf16_out, s);
  if (d.D % 64 == 0 && (uintptr_t)Y % 8 == 0) return launch_mc<2>(a, d.Bc, bf16_out, s);
  if (d.D % 32 == 0) return launch_mc<1>(a, d.Bc, bf16_out, s);
  return cudaErrorInvalidValue;
}

}  // namespace dq
