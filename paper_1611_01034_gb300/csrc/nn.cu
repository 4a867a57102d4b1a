// Learned gauge-covariant preconditioner layer (an addition to the method:
// the paper has no learned parts).  Two linear parallel-transport
// convolutions N = L2 o L1 (1 -> 8 -> 1 spinor channels):
//
//     y_o(x) = sum_i sum_d W[o][i][d] (T_d psi_i)(x),   d = self, +-T, +-Z, +-Y, +-X,
//     (T_{+mu} psi)(x) = U_mu(x) psi(x + mu),  (T_{-mu} psi)(x) = U_mu(x - mu)^dagger psi(x - mu),
//
// W[o][i][d] a complex 4 x 4 spin matrix acting trivially on colour, the
// fermion boundary factor on hops across T.  The preconditioner applies
// z = B(v) + N(v - D B(v)).
//
// All kernels are bound by FP32 arithmetic (issue 55 to 72 %, FP32 pipe 50 to
// 67 %).  A transport acts on colour and position, a weight on spin, so they
// commute and every transport is done on the single-channel side: L1 and the
// adjoint of L2 (1 -> 8) transport the input once for all 8 outputs, L2 (8 -> 1)
// sums its channels at the neighbour before transporting, and the gradients use
// <g, T_d h> = <T_d^+ g, h>.  16 samples on 16^4: L1 1.19 -> 0.79 ms, L2 1.14 ->
// 0.74 ms, gradients 2.53 + 1.79 -> 0.98 + 0.98 ms, inference and gradient
// together 10.7 -> 6.0 ms.
#include <cuda_fp16.h>

#include "tm_kernels.h"
#include "tm_lane.cuh"

namespace tmamg {

namespace {

constexpr int kNdir = 9;
constexpr int kC = kNnHidden;

// hidden channels: [rhs][8][component 12][V] complex, FP32 or FP16 (re, im)
template <typename Th>
struct Cx2;
template <>
struct Cx2<float> {
  using V = float2;
  static __device__ __forceinline__ cx<float> get(float2 v) { return {v.x, v.y}; }
  static __device__ __forceinline__ float2 put(cx<float> z) { return make_float2(z.r, z.i); }
};
template <>
struct Cx2<__half> {
  using V = __half2;
  static __device__ __forceinline__ cx<float> get(__half2 v) {
    const float2 f = __half22float2(v);
    return {f.x, f.y};
  }
  static __device__ __forceinline__ __half2 put(cx<float> z) { return __floats2half2_rn(z.r, z.i); }
};

// site, link site and boundary factor of direction d at site s
struct Nb {
  int s, link;
  float sg;
};
__device__ __forceinline__ Nb neighbour(const Lat& g, float bc, int s, const int (&cs)[4], int d) {
  if (d == 0) return {s, s, 1.f};
  const int mu = (d - 1) >> 1;
  const bool fwd = ((d - 1) & 1) == 0;
  const int cm = mu == 0 ? cs[0] : mu == 1 ? cs[1] : mu == 2 ? cs[2] : cs[3];
  const int Lm = mu == 0 ? g.L[0] : mu == 1 ? g.L[1] : mu == 2 ? g.L[2] : g.L[3];
  const int sm = mu == 0 ? g.st[0] : mu == 1 ? g.st[1] : mu == 2 ? g.st[2] : g.st[3];
  const bool edge = fwd ? cm + 1 == Lm : cm == 0;
  const int nb = fwd ? (edge ? s - (Lm - 1) * sm : s + sm) : (edge ? s + (Lm - 1) * sm : s - sm);
  return {nb, fwd ? s : nb, mu == 0 && edge ? bc : 1.f};
}

// phi = T_d p for the neighbour's spinor p
__device__ __forceinline__ void transport(const float* __restrict__ gauge, const Lat& g, const Nb& n, int d,
                                          const cx<float> (&p)[12], cx<float> (&phi)[12]) {
  if (d == 0) {
#pragma unroll
    for (int k = 0; k < 12; ++k) phi[k] = p[k];
    return;
  }
  Link<float> U;
  ld_link(gauge, g.V, (d - 1) >> 1, n.link, U);
#pragma unroll
  for (int sp = 0; sp < 4; ++sp) {
    const cx<float> x[3] = {n.sg * p[3 * sp], n.sg * p[3 * sp + 1], n.sg * p[3 * sp + 2]};
    cx<float> y[3];
    if ((d - 1) & 1)
      su3_dag_mul(U, x, y);
    else
      su3_mul(U, x, y);
    phi[3 * sp] = y[0];
    phi[3 * sp + 1] = y[1];
    phi[3 * sp + 2] = y[2];
  }
}

// One channel to eight (L1, and the adjoint of L2 with its weights): thread =
// (site, colour), the colour fixed per warp, all 32 output spinor components of
// its colour in registers, two output channels as the lanes of packed FP32.  The
// three warps of a site group read the same neighbours (L1).
constexpr int kExpandSites = 64;
template <typename Th>
__global__ void __launch_bounds__(3 * kExpandSites, 2) k_expand(const float* __restrict__ in,
                                                             typename Cx2<Th>::V* __restrict__ out,
                                                             const float* __restrict__ gauge,
                                                             const float2* __restrict__ W, Lat g, float bc) {
  __shared__ float4 Ws[kC / 2 * kNdir * 16];  // [o / 2][d][s][t]: (re, re, im, im) of the two channels
  for (int e = threadIdx.x; e < kC / 2 * kNdir * 16; e += blockDim.x) {
    const int o = e / (kNdir * 16) * 2, k = e % (kNdir * 16);
    const float2 a = W[o * kNdir * 16 + k], b = W[(o + 1) * kNdir * 16 + k];
    Ws[e] = make_float4(a.x, b.x, a.y, b.y);
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, c = warp % 3, r = blockIdx.y;
  const int s = blockIdx.x * kExpandSites + (warp / 3) * 32 + (threadIdx.x & 31);
  if (s >= g.V) return;
  const float* f = in + (long)r * NR_SPINOR * g.V;
  int cs[4];
  site_coords(g, s, cs);
  cx<f2> acc[kC / 2 * 4];
#pragma unroll
  for (int k = 0; k < kC / 2 * 4; ++k) acc[k] = czero<f2>();
#pragma unroll 1
  for (int d = 0; d < kNdir; ++d) {
    const Nb n = neighbour(g, bc, s, cs, d);
    cx<float> p[12], phi[4];
    ld_cx<float, 12>(f, g.V, n.s, p);
    if (d == 0) {
#pragma unroll
      for (int t = 0; t < 4; ++t) phi[t] = c == 0 ? p[3 * t] : c == 1 ? p[3 * t + 1] : p[3 * t + 2];
    } else {
      // row c of U, or of U^dagger
      Link<float> U;
      ld_link(gauge, g.V, (d - 1) >> 1, n.link, U);
      cx<float> u[3];
      if ((d - 1) & 1) {
#pragma unroll
        for (int k = 0; k < 3; ++k) u[k] = conj(c == 0 ? U.u[k][0] : c == 1 ? U.u[k][1] : U.u[k][2]);
      } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) u[k] = c == 0 ? U.u[0][k] : c == 1 ? U.u[1][k] : U.u[2][k];
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) u[k] = n.sg * u[k];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        phi[t] = u[0] * p[3 * t];
        cfma(phi[t], u[1], p[3 * t + 1]);
        cfma(phi[t], u[2], p[3 * t + 2]);
      }
    }
    f2 pr[4], pi[4], pn[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      pr[t] = bcast<f2>(phi[t].r);
      pi[t] = bcast<f2>(phi[t].i);
      pn[t] = bcast<f2>(-phi[t].i);
    }
#pragma unroll
    for (int o = 0; o < kC / 2; ++o)
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(Ws + ((o * kNdir + d) * 4 + sp) * 4 + t);
          cx<f2>& y = acc[o * 4 + sp];
          y.r = lfma(f2{w.x}, pr[t], y.r);
          y.r = lfma(f2{w.y}, pn[t], y.r);
          y.i = lfma(f2{w.x}, pi[t], y.i);
          y.i = lfma(f2{w.y}, pr[t], y.i);
        }
  }
  typename Cx2<Th>::V* q = out + (long)r * kC * 12 * g.V + s;
#pragma unroll
  for (int o = 0; o < kC / 2; ++o)
#pragma unroll
    for (int sp = 0; sp < 4; ++sp) {
      const float2 re = f2_unpack(acc[o * 4 + sp].r), im = f2_unpack(acc[o * 4 + sp].i);
      q[(long)(2 * o * 12 + 3 * sp + c) * g.V] = Cx2<Th>::put(cx<float>{re.x, im.x});
      q[(long)((2 * o + 1) * 12 + 3 * sp + c) * g.V] = Cx2<Th>::put(cx<float>{re.y, im.y});
    }
}

// Eight channels to one (L2): thread = site; per direction the channels are
// summed over their weights at the neighbour, then transported once.
template <typename Th>
__global__ void __launch_bounds__(128, 4) k_reduce(const typename Cx2<Th>::V* __restrict__ in, float* __restrict__ out,
                                                const float* __restrict__ gauge, const float2* __restrict__ W, Lat g,
                                                float bc, int accumulate) {
  __shared__ __align__(16) float2 Ws[kC * kNdir * 16];  // [i][d][s][t]
  for (int e = threadIdx.x; e < kC * kNdir * 16; e += blockDim.x) Ws[e] = W[e];
  __syncthreads();
  const int s = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y;
  if (s >= g.V) return;
  const typename Cx2<Th>::V* f = in + (long)r * kC * 12 * g.V;
  int cs[4];
  site_coords(g, s, cs);
  cx<float> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = cx<float>{0.f, 0.f};
#pragma unroll 1
  for (int d = 0; d < kNdir; ++d) {
    const Nb n = neighbour(g, bc, s, cs, d);
    cx<float> v[12], phi[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = cx<float>{0.f, 0.f};
#pragma unroll 2
    for (int i = 0; i < kC; ++i) {
      cx<float> h[12];
#pragma unroll
      for (int k = 0; k < 12; ++k) h[k] = Cx2<Th>::get(f[(long)(i * 12 + k) * g.V + n.s]);
#pragma unroll
      for (int sp = 0; sp < 4; ++sp) {
        const float4* w = reinterpret_cast<const float4*>(Ws + ((i * kNdir + d) * 4 + sp) * 4);
        const float4 w0 = w[0], w1 = w[1];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          cfma(v[3 * sp + c], cx<float>{w0.x, w0.y}, h[c]);
          cfma(v[3 * sp + c], cx<float>{w0.z, w0.w}, h[3 + c]);
          cfma(v[3 * sp + c], cx<float>{w1.x, w1.y}, h[6 + c]);
          cfma(v[3 * sp + c], cx<float>{w1.z, w1.w}, h[9 + c]);
        }
      }
    }
    transport(gauge, g, n, d, v, phi);
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = acc[k] + phi[k];
  }
  float* o = out + (long)r * NR_SPINOR * g.V;
  if (accumulate) {
    cx<float> q[12];
    ld_cx<float, 12>(o, g.V, s, q);
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = acc[k] + q[k];
  }
  st_cx<float, 12>(o, g.V, s, acc);
}

// Weight gradients, a contraction over sites and colours of the eight-channel
// side h with the transported one-channel side A_d = T_d a:
//   FIRST (W1):  G[o][d][s][t] = sum h_o[s] conj(A_d[t])              (h = g_h, a = r)
//   else  (W2):  G[i][d][s][t] = sum A_opp(d)[s] conj(h_i[t])         (a = g_y; T_d^+ = T_opp(d))
// Persistent CTAs stage tiles of 32 sites in shared memory (one transport per
// thread: 9 directions x 32 sites) and keep the 32 x 36 complex sums in
// registers: 2 groups of 144 threads, each 4 x 2 outputs and half of the sites.
// Every 24 terms are added to a running FP32 pair, so the length of the plain
// FP32 sums does not grow with the lattice.
__device__ __forceinline__ void add_two_sum(float& h, float& l, float x) {
  const float s = __fadd_rn(h, x), b = __fsub_rn(s, h);
  l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, b)), __fsub_rn(x, b)));
  h = s;
}
constexpr int kGTile = 32, kGThreads = 288, kGRows = 4 * kC, kGCols = 4 * kNdir;
// site strides (complex numbers, 2 mod 16): staging stores of neighbouring sites fall on distinct banks
constexpr int kGHs = 3 * kGRows + 2, kGAs = 3 * kGCols + 6;
template <bool FIRST>
__global__ void __launch_bounds__(kGThreads, 2) k_wgrad(const float2* __restrict__ hid, const float* __restrict__ one,
                                                        const float* __restrict__ gauge, Lat g, float bc, int nrhs,
                                                        double2* __restrict__ partial) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<float>* Hs = reinterpret_cast<cx<float>*>(smem_raw);  // [site 32][kGHs]: [colour 3][kGRows]
  cx<float>* As = Hs + kGTile * kGHs;                       // [site 32][kGAs]: [colour 3][kGCols]
  const int tid = threadIdx.x, grp = tid / 144, tg = tid % 144;
  const int row0 = (tg / 18) * 4, col0 = (tg % 18) * 2;  // one channel's spins, two of a direction's
  cx<float> hi[4][2], lo[4][2];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) hi[a][b] = lo[a][b] = cx<float>{0.f, 0.f};
  const int tpr = (g.V + kGTile - 1) / kGTile;
  const int dl = tid / 32, sl = tid & 31;  // this thread's direction and site when staging
  for (long tile = blockIdx.x; tile < (long)tpr * nrhs; tile += gridDim.x) {
    const int r = (int)(tile / tpr), s = (int)(tile % tpr) * kGTile + sl;
    __syncthreads();
    {
      cx<float> phi[12];
      if (s < g.V) {
        int cs[4];
        site_coords(g, s, cs);
        const Nb n = neighbour(g, bc, s, cs, dl);
        cx<float> p[12];
        ld_cx<float, 12>(one + (long)r * NR_SPINOR * g.V, g.V, n.s, p);
        transport(gauge, g, n, dl, p, phi);
      } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) phi[k] = cx<float>{0.f, 0.f};
      }
#pragma unroll
      for (int k = 0; k < 12; ++k) As[sl * kGAs + (k % 3) * kGCols + dl * 4 + k / 3] = phi[k];
    }
    if (dl < kC) {  // channel dl
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        const float2 v = s < g.V ? hid[((long)r * kC * 12 + dl * 12 + k) * g.V + s] : make_float2(0.f, 0.f);
        Hs[sl * kGHs + (k % 3) * kGRows + dl * 4 + k / 3] = cx<float>{v.x, v.y};
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int s0 = grp * 16; s0 < grp * 16 + 16; s0 += 8) {
      cx<float> acc[4][2];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) acc[a][b] = cx<float>{0.f, 0.f};
#pragma unroll 6
      for (int k = 0; k < 24; ++k) {
        const int st = s0 + k / 3, c = k % 3;
        const float4* hp = reinterpret_cast<const float4*>(Hs + st * kGHs + c * kGRows + row0);
        const float4 a0 = *reinterpret_cast<const float4*>(As + st * kGAs + c * kGCols + col0);
        const float4 h0 = hp[0], h1 = hp[1];
        const cx<float> hv[4] = {{h0.x, h0.y}, {h0.z, h0.w}, {h1.x, h1.y}, {h1.z, h1.w}};
        const cx<float> av[2] = {{a0.x, a0.y}, {a0.z, a0.w}};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            if (FIRST)
              cfmac(acc[a][b], av[b], hv[a]);
            else
              cfmac(acc[a][b], hv[a], av[b]);
          }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          add_two_sum(hi[a][b].r, lo[a][b].r, acc[a][b].r);
          add_two_sum(hi[a][b].i, lo[a][b].i, acc[a][b].i);
        }
    }
  }
  // the two groups' sums, then one partial per CTA
  __syncthreads();
  double2* red = reinterpret_cast<double2*>(smem_raw);  // [kGRows * kGCols]
  if (grp == 1) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b)
        red[tg * 8 + a * 2 + b] = make_double2((double)hi[a][b].r + lo[a][b].r, (double)hi[a][b].i + lo[a][b].i);
  }
  __syncthreads();
  if (grp == 1) return;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const double2 u = red[tg * 8 + a * 2 + b];
      const double2 v = make_double2((double)hi[a][b].r + lo[a][b].r + u.x, (double)hi[a][b].i + lo[a][b].i + u.y);
      const int ch = row0 / 4, dc = col0 / 4, t = (col0 & 3) + b;
      const int d = FIRST || dc == 0 ? dc : (((dc - 1) & 1) ? dc - 1 : dc + 1);
      const int e = (ch * kNdir + d) * 16 + (FIRST ? a * 4 + t : t * 4 + a);
      partial[(long)e * gridDim.x + blockIdx.x] = v;
    }
}

// out[e] = sum_cta partial[e][cta]
__global__ void k_wgrad_reduce(const double2* __restrict__ partial, int ncta, double2* __restrict__ out) {
  __shared__ double red[2 * 128];
  const int e = blockIdx.x;
  double a = 0, b = 0;
  for (int c = threadIdx.x; c < ncta; c += blockDim.x) {
    const double2 v = partial[(long)e * ncta + c];
    a += v.x;
    b += v.y;
  }
  red[threadIdx.x] = a;
  red[128 + threadIdx.x] = b;
  __syncthreads();
  for (int w = 64; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      red[threadIdx.x] += red[threadIdx.x + w];
      red[128 + threadIdx.x] += red[128 + threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) out[e] = make_double2(red[0], red[128]);
}

constexpr int kGCtas = 2 * kSms;

template <bool FIRST>
void run_wgrad(const float* hid, const float* one, const float* gauge, const Lat& g, double bc, int nrhs,
               double2* partial, double2* out, cudaStream_t st) {
  const size_t smem = (size_t)kGTile * (kGHs + kGAs) * sizeof(cx<float>);
  static_assert(kGRows * kGCols * sizeof(double2) <= (size_t)kGTile * (kGHs + kGAs) * sizeof(cx<float>),
                "the second group's sums reuse the tiles");
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_wgrad<FIRST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr = true;
  }
  const long tiles = (long)((g.V + kGTile - 1) / kGTile) * nrhs;
  const int ncta = (int)(tiles < kGCtas ? tiles : kGCtas);
  k_wgrad<FIRST><<<ncta, kGThreads, smem, st>>>(reinterpret_cast<const float2*>(hid), one, gauge, g, (float)bc, nrhs,
                                                partial);
  k_wgrad_reduce<<<kC * kNdir * 16, 128, 0, st>>>(partial, ncta, out);
}

template <typename Th>
void run_expand(const float* in, void* out, const float* gauge, const float2* W, const Lat& g, double bc, int nrhs,
                cudaStream_t st) {
  dim3 grid((unsigned)((g.V + kExpandSites - 1) / kExpandSites), nrhs);
  k_expand<Th><<<grid, 3 * kExpandSites, 0, st>>>(in, static_cast<typename Cx2<Th>::V*>(out), gauge, W, g, (float)bc);
}

template <typename Th>
void run_reduce(const void* in, float* out, const float* gauge, const float2* W, const Lat& g, double bc, int nrhs,
                bool acc, cudaStream_t st) {
  dim3 grid((unsigned)((g.V + 127) / 128), nrhs);
  k_reduce<Th><<<grid, 128, 0, st>>>(static_cast<const typename Cx2<Th>::V*>(in), out, gauge, W, g, (float)bc,
                                     acc ? 1 : 0);
}

}  // namespace

long nn_wgrad_partial_doubles2() { return (long)kGCtas * kC * kNdir * 16; }

void nn_layer1(const float* r, void* hid, bool half, const float* gauge, const float2* W1, const Lat& g, double bc,
               int nrhs, cudaStream_t st) {
  if (half)
    run_expand<__half>(r, hid, gauge, W1, g, bc, nrhs, st);
  else
    run_expand<float>(r, hid, gauge, W1, g, bc, nrhs, st);
}

void nn_layer2(const void* hid, bool half, float* y, bool accumulate, const float* gauge, const float2* W2,
               const Lat& g, double bc, int nrhs, cudaStream_t st) {
  if (half)
    run_reduce<__half>(hid, y, gauge, W2, g, bc, nrhs, accumulate, st);
  else
    run_reduce<float>(hid, y, gauge, W2, g, bc, nrhs, accumulate, st);
}

void nn_layer2_adjoint(const float* gy, float* gh, const float* gauge, const float2* W2adj, const Lat& g, double bc,
                       int nrhs, cudaStream_t st) {
  run_expand<float>(gy, gh, gauge, W2adj, g, bc, nrhs, st);
}

void nn_grad_w2(const float* hid, const float* gy, const float* gauge, const Lat& g, double bc, int nrhs,
                double2* partial, double2* out, cudaStream_t st) {
  run_wgrad<false>(hid, gy, gauge, g, bc, nrhs, partial, out, st);
}

void nn_grad_w1(const float* r, const float* gh, const float* gauge, const Lat& g, double bc, int nrhs,
                double2* partial, double2* out, cudaStream_t st) {
  run_wgrad<true>(gh, r, gauge, g, bc, nrhs, partial, out, st);
}

}  // namespace tmamg
