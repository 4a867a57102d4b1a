// Arnoldi steps of the outer FGMRES in FP32-pair arithmetic.
//
// The fine-level Krylov basis is FP64, and one Arnoldi step with classical
// Gram-Schmidt and one reorthogonalisation (CGS2) costs about 32 (k + 1)
// FP64 multiply-adds per complex element against k + 1 basis vectors.  On
// GB300 the FP64 rate (two FMA per clock per SM) makes that the limit, not
// the memory traffic.  These kernels keep the FP64 vectors in memory, split
// every loaded value into a pair h + l of FP32 numbers with integer
// operations (tm_pair.cuh), and do the products and sums in pair arithmetic
// (about 47 significant bits); results written back are FP64.  Each vector
// update is fused with the reduction that follows it in CGS2, so one step
// reads the basis three times instead of four:
//   d1 = V^H w                       (launch_pdot_b)
//   w -= V d1;  d2 = V^H w           (launch_pcaxpy_dot_b)
//   w -= V d2;  n = |w|^2            (launch_pcaxpy_norm_b)
// Partial sums per CTA are converted to FP64 and reduced in a fixed order,
// so every result is deterministic.
//
// With one complex number per packed FP32 operation (real and imaginary part as
// its lanes), the next element's loads in flight and a reduce-scatter for the
// CTAs' FP64 sums, latency and issue slots are the limit in turn (dot: issue 61 %,
// DRAM 66 % at k = 4).  Us at 32 x 16^3, six right-hand sides (151 MB per vector of
// the batch), for k = 1, 2, 3, 4 basis vectors, scalar form -> this one:
//   dot            184 218 260 299 -> 100 113 124 143
//   update + dot   290 334 391 449 -> 155 181 213 242
//   update + norm  197 236 274 310 -> 140 163 184 208
// From 5 vectors on the 8-wide kernels, with the loads of one element only in flight (k_pdot_partial_b<8> spills 52
// bytes), and from 9 on updates without a reduction fused in; for k = 5, 8, 9, 16, 17, 25:
//   dot            514 669 880 1288 1505 2145 -> 247 312 454 610 745 1040
//   update + dot   798 1062 - - - -           -> 558 692 - - - -
//   update         - - 354 579 614 869        -> - - 375 571 625 874
//   update + norm  346 449 483 725 761 1041   -> 268 345 406 621 681 958
#include "tm_kernels.h"
#include "tm_pair.cuh"

namespace tmamg {

namespace {

constexpr int kPairThreads = 256;
constexpr int kChunk = 8;  // basis vectors handled per CTA in registers

int pair_grid(long ncx) { return dot_grid_for(ncx); }

__device__ __forceinline__ double2 ld_raw(const double* __restrict__ p, long i) {
  return reinterpret_cast<const double2*>(p)[i];
}
__device__ __forceinline__ pk2 to_pair(double2 v) { return cx2pair(v.x, v.y); }
__device__ __forceinline__ void st_pair(double* __restrict__ p, long i, pk2 a) {
  const float2 h = f2_unpack(a.h), l = f2_unpack(a.l);
  reinterpret_cast<double2*>(p)[i] = make_double2(pair2d(dfl{h.x, l.x}), pair2d(dfl{h.y, l.y}));
}
__device__ __forceinline__ pk2 pzero() { return {f2_pack(0.f, 0.f), f2_pack(0.f, 0.f)}; }
__device__ __forceinline__ f2 swap(f2 a) {
  const float2 v = f2_unpack(a);
  return f2_pack(v.y, v.x);
}
__device__ __forceinline__ pk2 swap(pk2 a) { return {swap(a.h), swap(a.l)}; }

// conj(x) y summed with the lanes of x as they are loaded: a = (xr yr, xi yi), b = (xr yi, xi yr)
struct DotAcc {
  pk2 a, b;
};
// its real and imaginary part in FP64
__device__ __forceinline__ double dot_re(const DotAcc& d) {
  const float2 h = f2_unpack(d.a.h), l = f2_unpack(d.a.l);
  dfl s{h.x, l.x};
  add_to(s, dfl{h.y, l.y});
  return pair2d(s);
}
__device__ __forceinline__ double dot_im(const DotAcc& d) {
  const float2 h = f2_unpack(d.b.h), l = f2_unpack(d.b.l);
  dfl s{h.x, l.x};
  add_to(s, dfl{-h.y, -l.y});
  return pair2d(s);
}
// a complex coefficient: its parts broadcast to both lanes
struct Coef {
  pn2 r, i;
};
__device__ __forceinline__ Coef coef(double re, double im) {
  const dfl a = d2pair(re), b = d2pair(im);
  return {bc_pair(a.h, a.l), bc_pair(b.h, b.l)};
}
// CTA's sums of d into the partials of right-hand side r, vectors j0 .. k
template <int KC>
__device__ __forceinline__ void put_partials(const DotAcc (&d)[KC], int r, int j0, int k, double* __restrict__ part) {
  __shared__ double red[kPairThreads / 32 * 2 * KC], fin[2 * KC];
  double v[2 * KC];
#pragma unroll
  for (int jj = 0; jj < KC; ++jj) {
    v[2 * jj] = dot_re(d[jj]);
    v[2 * jj + 1] = dot_im(d[jj]);
  }
  block_reduce_n<double, 2 * KC>(v, red, fin);
  if (threadIdx.x < 2 * KC) {
    const int jj = threadIdx.x >> 1;
    if (j0 + jj < k)
      part[(((long)r * k + j0 + jj) * gridDim.x + blockIdx.x) * 2 + (threadIdx.x & 1)] = fin[threadIdx.x];
  }
}

// stage 1 of d_j = sum_i conj(X_j[i]) y[i] for j in the CTA's chunk of KC
// (KC = 4 for short bases: fewer registers, more warps in flight)
template <int KC>
__global__ void __launch_bounds__(kPairThreads, 2) k_pdot_partial_b(const double* __restrict__ X, long xstr, long ldx,
                                                                 int k, const double* __restrict__ y, long ystr,
                                                                 long ncx, double* __restrict__ part,
                                                                 const int* __restrict__ active) {
  const int r = blockIdx.z;
  if (active && !active[r]) return;
  const int j0 = blockIdx.y * KC;
  DotAcc d[KC];
#pragma unroll
  for (int m = 0; m < KC; ++m) d[m] = DotAcc{pzero(), pzero()};
  const double* yr = y + r * ystr;
  const double* Xr = X + r * xstr + j0 * ldx;
  const long step = (long)gridDim.x * blockDim.x;
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  double2 yn = make_double2(0, 0), xn[KC];
  auto fetch = [&]() {
    yn = ld_raw(yr, i);
#pragma unroll
    for (int jj = 0; jj < KC; ++jj)
      if (j0 + jj < k) xn[jj] = ld_raw(Xr + jj * ldx, i);
  };
  constexpr bool kAhead = KC <= 4;  // the next element's loads in flight; with 8 vectors it costs a CTA per SM
  if (kAhead && i < ncx) fetch();
  while (i < ncx) {
    if (!kAhead) fetch();  // still all loads before the first conversion, which branches
    const double2 y0 = yn;
    double2 x0[KC];
#pragma unroll
    for (int jj = 0; jj < KC; ++jj) x0[jj] = xn[jj];
    i += step;
    if (kAhead && i < ncx) fetch();
    const pk2 yv = to_pair(y0);
    const pn2 ya = lane_pair(yv), yb = lane_pair(swap(yv));
#pragma unroll
    for (int jj = 0; jj < KC; ++jj)
      if (j0 + jj < k) {
        const pk2 x = to_pair(x0[jj]);
        fma_px(d[jj].a, ya, x);
        fma_px(d[jj].b, yb, x);
      }
  }
  put_partials<KC>(d, r, j0, k, part);
}

// y -= sum_j c_j X_j over all k vectors; MODE 1 (k <= KC) also forms the
// partial sums of d_j = X_j^H y with the updated y, MODE 2 those of |y|^2
template <int MODE, int KC = kChunk>
__global__ void __launch_bounds__(kPairThreads, MODE == 1 ? (KC <= 4 ? 2 : 1) : 3) k_pcaxpy_b(const double* __restrict__ X, long xstr, long ldx, int k,
                                                           const double* __restrict__ c, long cstr,
                                                           double* __restrict__ y, long ystr, long ncx,
                                                           double* __restrict__ part, const int* __restrict__ active) {
  extern __shared__ __align__(16) unsigned char praw[];
  Coef* cs = reinterpret_cast<Coef*>(praw);  // -c_j, [k]
  const int r = blockIdx.y;
  if (active && !active[r]) return;
  const double* cr = c + r * cstr;
  for (int j = threadIdx.x; j < k; j += blockDim.x) cs[j] = coef(-cr[2 * j], -cr[2 * j + 1]);
  __syncthreads();
  double* yr = y + r * ystr;
  const double* Xr = X + r * xstr;
  DotAcc d[MODE == 1 ? KC : 1];
#pragma unroll
  for (int m = 0; m < (MODE == 1 ? KC : 1); ++m) d[m] = DotAcc{pzero(), pzero()};
  // loads of the next element (its first NB vectors) in flight while one is worked on, and all before
  // the first conversion, which branches; with 8 vectors kept that would cost a CTA per SM
  constexpr int NB = MODE == 1 ? KC : 4;
  constexpr bool kAhead = NB <= 4;
  const long step = (long)gridDim.x * blockDim.x;
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  double2 yn = make_double2(0, 0), xn[NB];
#pragma unroll
  for (int j = 0; j < NB; ++j) xn[j] = make_double2(0, 0);
  auto fetch = [&](long e) {
    yn = ld_raw(yr, e);
#pragma unroll
    for (int j = 0; j < NB; ++j)
      if (j < k) xn[j] = ld_raw(Xr + j * ldx, e);
  };
  if (kAhead && i < ncx) fetch(i);
  for (; i < ncx; i += step) {
    if (!kAhead) fetch(i);
    const double2 y0 = yn;
    double2 x0[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) x0[j] = xn[j];
    if (kAhead && i + step < ncx) fetch(i + step);
    pk2 ti = pzero();  // acc: sum of Re c x, ti: of Im c x
    pk2 acc;
    if constexpr (MODE == 1) {
      pk2 xs[KC];
#pragma unroll
      for (int j = 0; j < KC; ++j) xs[j] = pzero();
      acc = to_pair(y0);
#pragma unroll
      for (int j = 0; j < KC; ++j) {
        if (j < k) {
          xs[j] = to_pair(x0[j]);
          fma_px(acc, cs[j].r, xs[j]);
          fma_px(ti, cs[j].i, xs[j]);
        }
      }
      add_to(acc, times_i(ti));
      const pn2 ya = lane_pair(acc), yb = lane_pair(swap(acc));
#pragma unroll
      for (int j = 0; j < KC; ++j)
        if (j < k) {
          fma_px(d[j].a, ya, xs[j]);
          fma_px(d[j].b, yb, xs[j]);
        }
    } else {
      acc = to_pair(y0);
      for (int j0 = 0; j0 < k; j0 += NB) {
        if (j0 > 0) {
#pragma unroll
          for (int j = 0; j < NB; ++j)
            if (j0 + j < k) x0[j] = ld_raw(Xr + (j0 + j) * ldx, i);
        }
#pragma unroll
        for (int j = 0; j < NB; ++j)
          if (j0 + j < k) {
            const pk2 x = to_pair(x0[j]);
            fma_px(acc, cs[j0 + j].r, x);
            fma_px(ti, cs[j0 + j].i, x);
          }
      }
      add_to(acc, times_i(ti));
      if constexpr (MODE == 2) fma_px(d[0].a, lane_pair(acc), acc);
    }
    st_pair(yr, i, acc);
  }
  if constexpr (MODE == 1) {
    put_partials<KC>(d, r, 0, k, part);
  } else if constexpr (MODE == 2) {
    __shared__ double red[kPairThreads / 32], fin[1];
    const double v[1] = {dot_re(d[0])};
    block_reduce_n<double, 1>(v, red, fin);
    if (threadIdx.x == 0) part[(long)r * gridDim.x + blockIdx.x] = fin[0];
  }
}

// out[r * ostr + 2 j + {0,1}] = sum over the G partials of (r, j), fixed order
__global__ void k_preduce_b(const double* __restrict__ part, int G, int k, double* __restrict__ out, long ostr,
                            const int* __restrict__ active) {
  __shared__ double red[32 * 2];
  const int j = blockIdx.x, r = blockIdx.y;
  if (active && !active[r]) return;
  double d[2] = {0, 0};
  const double* p = part + ((long)r * k + j) * G * 2;
  for (int b = threadIdx.x; b < G; b += blockDim.x) {
    d[0] += p[2 * b];
    d[1] += p[2 * b + 1];
  }
  block_allreduce<double, 2>(d, red);
  if (threadIdx.x == 0) {
    out[r * ostr + 2 * j] = d[0];
    out[r * ostr + 2 * j + 1] = d[1];
  }
}

__global__ void k_preduce_norm_b(const double* __restrict__ part, int G, double* __restrict__ out,
                                 const int* __restrict__ active) {
  __shared__ double red[32];
  const int r = blockIdx.x;
  if (active && !active[r]) return;
  double d[1] = {0};
  for (int b = threadIdx.x; b < G; b += blockDim.x) d[0] += part[(long)r * G + b];
  block_allreduce<double, 1>(d, red);
  if (threadIdx.x == 0) out[r] = d[0];
}

// x += sum_j c_j Z_j, Z FP32 (exact in a pair), x FP64; active[r] = terms of rhs r (0: skip)
__global__ void __launch_bounds__(kPairThreads) k_plincomb_b(const float* __restrict__ Z, long zstr, long ldz, int k,
                                                             const double* __restrict__ c, long cstr,
                                                             double* __restrict__ x, long xstr, long ncx,
                                                             const int* __restrict__ active) {
  extern __shared__ __align__(16) unsigned char praw[];
  Coef* cs = reinterpret_cast<Coef*>(praw);
  const int r = blockIdx.y;
  if (active && !active[r]) return;
  const int kr = active ? min(k, active[r]) : k;
  const double* cr = c + r * cstr;
  for (int j = threadIdx.x; j < kr; j += blockDim.x) cs[j] = coef(cr[2 * j], cr[2 * j + 1]);
  __syncthreads();
  double* xr = x + r * xstr;
  const float* Zr = Z + r * zstr;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < ncx; i += (long)gridDim.x * blockDim.x) {
    pk2 acc = to_pair(ld_raw(xr, i)), ti = pzero();
#pragma unroll 4
    for (int j = 0; j < kr; ++j) {
      const float2 v = reinterpret_cast<const float2*>(Zr + j * ldz)[i];
      const f2 z = f2_pack(v.x, v.y);
      fma_px(acc, cs[j].r, z);
      fma_px(ti, cs[j].i, z);
    }
    add_to(acc, times_i(ti));
    st_pair(xr, i, acc);
  }
}

size_t pair_smem(int k) { return (size_t)k * sizeof(Coef); }
constexpr int kShort = 4;  // bases of at most 4 vectors take the 4-wide kernels

}  // namespace

void launch_pdot_b(const double* X, long xstr, long ldx, int k, const double* y, long ystr, long ncx, double* out,
                   long ostr, double* scratch, int nrhs, const int* active, cudaStream_t st) {
  const int G = pair_grid(ncx);
  if (k <= kShort)
    k_pdot_partial_b<kShort><<<dim3(G, 1, nrhs), kPairThreads, 0, st>>>(X, xstr, ldx, k, y, ystr, ncx, scratch,
                                                                        active);
  else
    k_pdot_partial_b<kChunk><<<dim3(G, (k + kChunk - 1) / kChunk, nrhs), kPairThreads, 0, st>>>(
        X, xstr, ldx, k, y, ystr, ncx, scratch, active);
  k_preduce_b<<<dim3(k, nrhs), 256, 0, st>>>(scratch, G, k, out, ostr, active);
}

int launch_pcaxpy_dot_b(const double* X, long xstr, long ldx, int k, const double* c, long cstr, double* y, long ystr,
                        long ncx, double* out, long ostr, double* scratch, int nrhs, const int* active,
                        cudaStream_t st) {
  const int G = pair_grid(ncx);
  if (k <= kShort) {
    k_pcaxpy_b<1, kShort><<<dim3(G, nrhs), kPairThreads, pair_smem(k), st>>>(X, xstr, ldx, k, c, cstr, y, ystr, ncx,
                                                                             scratch, active);
    k_preduce_b<<<dim3(k, nrhs), 256, 0, st>>>(scratch, G, k, out, ostr, active);
    return 2;
  }
  if (k <= kChunk) {
    k_pcaxpy_b<1><<<dim3(G, nrhs), kPairThreads, pair_smem(k), st>>>(X, xstr, ldx, k, c, cstr, y, ystr, ncx, scratch,
                                                                     active);
    k_preduce_b<<<dim3(k, nrhs), 256, 0, st>>>(scratch, G, k, out, ostr, active);
    return 2;
  }
  k_pcaxpy_b<0><<<dim3(G, nrhs), kPairThreads, pair_smem(k), st>>>(X, xstr, ldx, k, c, cstr, y, ystr, ncx, nullptr,
                                                                   active);
  launch_pdot_b(X, xstr, ldx, k, y, ystr, ncx, out, ostr, scratch, nrhs, active, st);
  return 3;
}

void launch_pcaxpy_norm_b(const double* X, long xstr, long ldx, int k, const double* c, long cstr, double* y,
                          long ystr, long ncx, double* nrm, double* scratch, int nrhs, const int* active,
                          cudaStream_t st) {
  const int G = pair_grid(ncx);
  k_pcaxpy_b<2><<<dim3(G, nrhs), kPairThreads, pair_smem(k), st>>>(X, xstr, ldx, k, c, cstr, y, ystr, ncx, scratch,
                                                                   active);
  k_preduce_norm_b<<<nrhs, 256, 0, st>>>(scratch, G, nrm, active);
}

void launch_plincomb_b(const float* Z, long zstr, long ldz, int k, const double* c, long cstr, double* x, long xstr,
                       long ncx, int nrhs, const int* active, cudaStream_t st) {
  k_plincomb_b<<<dim3(pair_grid(ncx), nrhs), kPairThreads, pair_smem(k), st>>>(Z, zstr, ldz, k, c, cstr,
                                                                                          x, xstr, ncx, active);
}

}  // namespace tmamg
