// D(mu) on FP32 input with an FP64-accurate result from pairs of FP32 numbers.
//
// The outer FGMRES applies D(mu) to the preconditioned vectors z_k = B(v_k),
// which the FP32 K-cycle produces; the Arnoldi relation D Z = V H needs that
// product to FP64 accuracy (an FP32 product would put a floor of ~1e-7 under
// the residual).  GB300 runs FP64 at 1/64 of its FP32 rate, so here every real
// is carried as an unevaluated sum h + l of two FP32 numbers (Dekker's
// "double-length" arithmetic, Numer. Math. 18 (1971) 224, with Knuth's
// two-sum): products a.h*b.h are made exact with an FMA, the cross terms and
// the rounding errors gather in l.  Links (all 18 reals, no third-row
// reconstruction) and clover blocks are stored as such pairs; the input is
// FP32 and therefore exact.  The relative error is about 2^-46 (a few 1e-14)
// times the cancellation of the sum, the output is FP64.
//
// Operator as in dirac.cu (Sec. 1: D(mu) = D_W + i mu Gamma5):
//   (D psi)(x) = A(x) psi(x) + i mu gamma5 psi(x)
//       - 1/2 sum_mu [ (1 - gamma_mu) U_mu(x) psi(x+mu) + (1 + gamma_mu) U_mu(x-mu)^+ psi(x-mu) ]
#include <type_traits>

#include "tm_kernels.h"
#include "tm_lane.cuh"
#include "tm_pair.cuh"

namespace tmamg {

namespace {

// i^q x, q at run time (exact; branch-free selects)
__device__ __forceinline__ f2 times_ph(f2 x, int q) {
  const float2 v = f2_unpack(x);
  const bool sw = q & 1;
  const float sr = (q == 1 || q == 2) ? -1.f : 1.f, si = q >= 2 ? -1.f : 1.f;
  return f2_pack(sr * (sw ? v.y : v.x), si * (sw ? v.x : v.y));
}
__device__ __forceinline__ pk2 times_ph(pk2 x, int q) { return {times_ph(x.h, q), times_ph(x.l, q)}; }
// x + y as a pair (exact for FP32 x, y)
__device__ __forceinline__ pk2 pair_sum(f2 x, f2 y) { return two_sum2(x, y); }
__device__ __forceinline__ pk2 pair_sum(pk2 x, pk2 y) {
  const pk2 s = two_sum2(x.h, y.h);
  return {s.h, s.l + (x.l + y.l)};
}

__device__ __forceinline__ int gphase_rt(int mu, int r) {
  return mu == 0 ? 2 : mu == 1 ? (r == 0 ? 3 : 1) : mu == 2 ? (r == 0 ? 2 : 0) : 3;
}

// acc += sign (1 -+ gamma_mu) U^(+) p for hop direction mu (runtime) and
// orientation fwd (U = U_mu(x), psi(x + mu), projector 1 - gamma) or backward
// (U^dagger of U_mu(x - mu), psi(x - mu), projector 1 + gamma); link site sl.
// One copy of the code serves all eight hops, so the kernel's loop over them
// stays in the instruction cache.
template <typename PT>  // input spinor components: exact FP32 (f2) or pairs (pk2)
__device__ __forceinline__ void hop_df_rt(const PT (&p)[12], const float4* __restrict__ gdf, long V, long sl, int mu,
                                          bool fwd, float sign, pk2 (&acc)[12]) {
  const bool sw = mu >= 2;  // A_mu's row r holds its entry in column r (T, Z) or 1 - r (Y, X)
  const f2 sg = f2_pack(sign, sign);
  pk2 h[2][3];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    // (1 - gamma): h = up - A dn; (1 + gamma): h = up + A dn  (exact as pairs for FP32 input)
    const int q = (gphase_rt(mu, r) + (fwd ? 2 : 0)) & 3;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const PT dn = (sw != (r == 1)) ? p[9 + k] : p[6 + k];  // spin 2 + perm(r)
      const pk2 t = pair_sum(p[3 * r + k], times_ph(dn, q));
      h[r][k] = pk2{sg * t.h, sg * t.l};
    }
  }
  pk2 w[2][3];
  const float4* lk = gdf + (long)mu * 9 * V + sl;  // entry e at lk + e V: (re.h, im.h, re.l, im.l)
  const float cj = fwd ? 1.f : -1.f;               // backward hops take conj(U[b][a])
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int a = 0; a < 3; ++a) w[r][a] = pk2{f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const pk2 hi[2] = {times_i(h[0][b]), times_i(h[1][b])};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float4 u = __ldg(lk + (long)(fwd ? 3 * a + b : 3 * b + a) * V);
      const pn2 ur = bc_pair(u.x, u.z), ui = bc_pair(cj * u.y, cj * u.w);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        fma_px(w[r][a], ur, h[r][b]);
        fma_px(w[r][a], ui, hi[r]);
      }
    }
  }
  // lower components: -+ A^dagger w, (A^dagger w)[perm r] = conj(phase r) w[r]
  const int q0 = (4 - gphase_rt(mu, 0) + (fwd ? 2 : 0)) & 3, q1 = (4 - gphase_rt(mu, 1) + (fwd ? 2 : 0)) & 3;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    add_to(acc[k], w[0][k]);
    add_to(acc[3 + k], w[1][k]);
    const pk2 l0 = times_ph(w[0][k], q0), l1 = times_ph(w[1][k], q1);
    add_to(acc[6 + k], sw ? l1 : l0);
    add_to(acc[9 + k], sw ? l0 : l1);
  }
}

struct DfArgs {
  const float4* gdf;
  const float4* cdf4;
  const void* in;     // FP32 (exact in pairs) or FP64 (split into pairs) spinors
  const double* sub;  // if set: out = sub - D in
  double* out;
  Lat g;
  dfl mu, mu_odd;  // twisted mass on even and on odd sites
  float bc;
  int nrhs;
};

// chunks k0 .. k0 + N / 2 - 1 of a site: exact FP32 components, or pairs split from FP64
template <int N>
__device__ __forceinline__ void ld_in(const float* in, long V, long s, int k0, f2 (&p)[N]) {
  const float4* q = reinterpret_cast<const float4*>(in) + (long)k0 * V + s;
#pragma unroll
  for (int k = 0; k < N / 2; ++k) {
    const float4 v = __ldg(q + k * V);
    p[2 * k] = f2_pack(v.x, v.y);
    p[2 * k + 1] = f2_pack(v.z, v.w);
  }
}
__device__ __forceinline__ pk2 pk_of(double re, double im) {
  const dfl a = d2pair(re), b = d2pair(im);
  return {f2_pack(a.h, b.h), f2_pack(a.l, b.l)};
}
template <int N>
__device__ __forceinline__ void ld_in(const double* in, long V, long s, int k0, pk2 (&p)[N]) {
  const double2* q = reinterpret_cast<const double2*>(in) + 2 * ((long)k0 * V + s);
#pragma unroll
  for (int k = 0; k < N / 2; ++k) {
    const double2 v0 = __ldg(q + 2 * k * V), v1 = __ldg(q + 2 * k * V + 1);
    p[2 * k] = pk_of(v0.x, v0.y);
    p[2 * k + 1] = pk_of(v1.x, v1.y);
  }
}
__device__ __forceinline__ double2 pk2d(pk2 a) {
  const float2 h = f2_unpack(a.h), l = f2_unpack(a.l);
  return make_double2(pair2d(dfl{h.x, l.x}), pair2d(dfl{h.y, l.y}));
}

// Bound by FP32 issue and instruction fetch, not by memory (0.67 TB/s).  The
// real and imaginary parts of a pair go through every step of the double-length
// arithmetic alike, so they are the two lanes of packed FP32: half the
// instructions and half the code of the scalar form (2.05 G -> 1.36 G warp
// instructions for 6 right-hand sides at 48 x 24^3).  The two chiralities of the
// clover term run through one copy of their code as well.  Three CTAs per SM
// (168 registers): 2.84 -> 1.95 ms there; four 2.10 ms, two 2.50 ms.
template <typename IN>
__global__ void __launch_bounds__(128, 3) k_dslash_df(DfArgs a) {
  using PT = typename std::conditional<std::is_same<IN, float>::value, f2, pk2>::type;
  const int rhs = a.nrhs == 1 ? 0 : (int)(blockIdx.x % a.nrhs);
  const int s = (a.nrhs == 1 ? blockIdx.x : blockIdx.x / a.nrhs) * blockDim.x + threadIdx.x;
  if (s >= a.g.V) return;
  const long V = a.g.V;
  const long off = (long)rhs * NR_SPINOR * V;
  const IN* in = static_cast<const IN*>(a.in) + off;
  int c[4];
  site_coords(a.g, s, c);
  pk2 acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = pk2{f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)};
  // the eight hops through one copy of the hop code (direction and orientation at run time)
#pragma unroll 1
  for (int hop = 0; hop < 8; ++hop) {
    const int mu = hop >> 1;
    const bool fwd = (hop & 1) == 0;
    const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
    const int Lm = mu == 0 ? a.g.L[0] : mu == 1 ? a.g.L[1] : mu == 2 ? a.g.L[2] : a.g.L[3];
    const int stm = mu == 0 ? a.g.st[0] : mu == 1 ? a.g.st[1] : mu == 2 ? a.g.st[2] : a.g.st[3];
    const int sn = fwd ? (cm + 1 < Lm ? s + stm : s - (Lm - 1) * stm) : (cm > 0 ? s - stm : s + (Lm - 1) * stm);
    const float sign = (mu == 0 && cm == (fwd ? Lm - 1 : 0)) ? a.bc : 1.f;
    PT p[12];
    ld_in(in, V, sn, 0, p);
    hop_df_rt(p, a.gdf, V, fwd ? s : sn, mu, fwd, sign, acc);
  }
  // y = A p + i mu gamma5 p - acc / 2, one chirality (gamma5 = -1, then +1) per turn
  const dfl mus = ((c[0] + c[1] + c[2] + c[3]) & 1) ? a.mu_odd : a.mu;
  const f2 mhalf = f2_pack(-0.5f, -0.5f);
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    PT p[6], ip[6];
    ld_in(in, V, s, 3 * h, p);
    pk2 y[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      ip[i] = times_i(p[i]);
      y[i] = pk2{mhalf * acc[i].h, mhalf * acc[i].l};
    }
    // clover chunk k of a chirality: float4 (r[2k].h, r[2k+1].h, r[2k].l, r[2k+1].l)
    const float4* c4 = a.cdf4 + (long)18 * h * V + s;
    // diagonal reals (chunks 0..2)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float4 d = __ldg(c4 + k * V);
      fma_px(y[2 * k], bc_pair(d.x, d.z), p[2 * k]);
      fma_px(y[2 * k + 1], bc_pair(d.y, d.w), p[2 * k + 1]);
    }
    // upper triangle (0,1),(0,2),...,(4,5): complex entry q = chunk 3 + q
    int q = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int j = i + 1; j < 6; ++j) {
        const float4 u = __ldg(c4 + (3 + q) * V);
        ++q;
        const pn2 ur = bc_pair(u.x, u.z), ui = bc_pair(u.y, u.w), un = bc_pair(-u.y, -u.w);
        fma_px(y[i], ur, p[j]);
        fma_px(y[i], ui, ip[j]);
        fma_px(y[j], ur, p[i]);
        fma_px(y[j], un, ip[i]);
      }
    const pn2 m = bc_pair(h == 0 ? -mus.h : mus.h, h == 0 ? -mus.l : mus.l);
#pragma unroll
    for (int i = 0; i < 6; ++i) fma_px(y[i], m, ip[i]);
    // FP64 output: h + l (or sub - (h + l))
    double2* o = reinterpret_cast<double2*>(a.out + off);
    const double2* sb = a.sub ? reinterpret_cast<const double2*>(a.sub + off) : nullptr;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const long i0 = 2 * ((long)(3 * h + k) * V + s);  // complex numbers 6 h + 2 k, 6 h + 2 k + 1
      double2 v0 = pk2d(y[2 * k]), v1 = pk2d(y[2 * k + 1]);
      if (sb) {
        const double2 b0 = sb[i0], b1 = sb[i0 + 1];
        v0 = make_double2(b0.x - v0.x, b0.y - v0.y);
        v1 = make_double2(b1.x - v1.x, b1.y - v1.y);
      }
      o[i0] = v0;
      o[i0 + 1] = v1;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) acc[i] = acc[6 + i];  // the other chirality next
  }
}

__device__ __forceinline__ float2 split(double x) {
  const float hi = __double2float_rn(x);
  return make_float2(hi, __double2float_rn(x - (double)hi));
}

// natural gauge [V][4][3][3] complex128 -> [4][9][V] float4 pairs
__global__ void k_pack_gauge_df(const double* __restrict__ nat, float4* __restrict__ gdf, int V) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  const int mu = blockIdx.y;
  if (s >= V) return;
  const double2* p = reinterpret_cast<const double2*>(nat) + ((long)s * 4 + mu) * 9;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const double2 v = p[e];
    const float2 re = split(v.x), im = split(v.y);
    gdf[((long)mu * 9 + e) * V + s] = make_float4(re.x, im.x, re.y, im.y);
  }
}

// packed FP64 clover [18 chunks][V] (4 reals each) -> [36][V] float4 pairs
__global__ void k_clover_df(const double* __restrict__ c64, float4* __restrict__ c4, int V) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= V) return;
  double r[72];
  ld_re<double, 72>(c64, V, s, r);
#pragma unroll
  for (int j = 0; j < 36; ++j) {
    const float2 a = split(r[2 * j]), b = split(r[2 * j + 1]);
    c4[(long)j * V + s] = make_float4(a.x, b.x, a.y, b.y);
  }
}

}  // namespace

void launch_pack_gauge_df(const double* nat, void* gdf, const Lat& g, cudaStream_t st) {
  dim3 grid((g.V + 127) / 128, 4);
  k_pack_gauge_df<<<grid, 128, 0, st>>>(nat, static_cast<float4*>(gdf), g.V);
}

void launch_clover_df(const double* c64, void* cdf, const Lat& g, cudaStream_t st) {
  k_clover_df<<<(g.V + 127) / 128, 128, 0, st>>>(c64, static_cast<float4*>(cdf), g.V);
}

DfArgs df_args(const void* gdf, const void* cdf, const void* in, const double* sub, double* out, const Lat& g,
               double mu, double bc_t, int nrhs, double rho) {
  const double muo = mu + rho;
  const float mh = (float)mu, moh = (float)muo;
  return DfArgs{static_cast<const float4*>(gdf), static_cast<const float4*>(cdf), in, sub, out, g,
                dfl{mh, (float)(mu - (double)mh)}, dfl{moh, (float)(muo - (double)moh)}, (float)bc_t, nrhs};
}

void launch_dslash_df(const void* gdf, const void* cdf, const float* in, double* out, const Lat& g, double mu,
                      double bc_t, int nrhs, cudaStream_t st, double rho) {
  dim3 grid((unsigned)((g.V + 127) / 128) * (unsigned)nrhs);
  k_dslash_df<float><<<grid, 128, 0, st>>>(df_args(gdf, cdf, in, nullptr, out, g, mu, bc_t, nrhs, rho));
}

void launch_residual_df(const void* gdf, const void* cdf, const double* x, const double* b, double* r, const Lat& g,
                        double mu, double bc_t, int nrhs, cudaStream_t st, double rho) {
  dim3 grid((unsigned)((g.V + 127) / 128) * (unsigned)nrhs);
  k_dslash_df<double><<<grid, 128, 0, st>>>(df_args(gdf, cdf, x, b, r, g, mu, bc_t, nrhs, rho));
}

}  // namespace tmamg
