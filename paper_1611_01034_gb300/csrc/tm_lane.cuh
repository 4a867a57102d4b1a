// Two right-hand sides per thread as the two lanes of packed FP32 arithmetic
// (add / sub / mul / fma .rn.f32x2, sm_100 and later).
//
// The rate of the FP32 pipe is the same packed or not (measured: 72 against
// 75 TFLOP/s on independent chains); what packing halves is the instructions,
// and the operator entries (links, clover, D_oo^-1) are loaded, converted and
// rebuilt once for both lanes.  Kernels written over a lane type R run with
// R = float or double (one right-hand side) and R = f2 (two); operator
// entries stay scalars and are broadcast where they are used.
#pragma once
#include <type_traits>

#include "tm_internal.cuh"

namespace tmamg {

struct f2 {
  unsigned long long v;
};

__device__ __forceinline__ f2 f2_pack(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(f2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ f2 operator+(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator-(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator*(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 lfma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ float lfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double lfma(double a, double b, double c) { return fma(a, b, c); }

// lane type R: its scalar, its lane count, a broadcast
template <class R>
struct LaneOf {
  using T = R;
  static constexpr int n = 1;
};
template <>
struct LaneOf<f2> {
  using T = float;
  static constexpr int n = 2;
};
template <class R>
__device__ __forceinline__ R bcast(typename LaneOf<R>::T s) {
  if constexpr (LaneOf<R>::n == 2)
    return f2_pack(s, s);
  else
    return s;
}
template <class R>
__device__ __forceinline__ cx<R> czero() {
  return cx<R>{bcast<R>(0), bcast<R>(0)};
}

// a + i^p w, p known at compile time after inlining
template <class R>
__device__ __forceinline__ cx<R> add_ph(cx<R> a, cx<R> w, int p) {
  switch (p & 3) {
    case 0: return {a.r + w.r, a.i + w.i};
    case 1: return {a.r - w.i, a.i + w.r};
    case 2: return {a.r - w.r, a.i - w.i};
    default: return {a.r + w.i, a.i - w.r};
  }
}
// acc += u x, acc += conj(u) x for a scalar u
template <class R, class T>
__device__ __forceinline__ void lcfma(cx<R>& acc, cx<T> u, cx<R> x) {
  const R ur = bcast<R>(u.r), ui = bcast<R>(u.i), un = bcast<R>(-u.i);
  acc.r = lfma(ur, x.r, acc.r);
  acc.r = lfma(un, x.i, acc.r);
  acc.i = lfma(ur, x.i, acc.i);
  acc.i = lfma(ui, x.r, acc.i);
}
template <class R, class T>
__device__ __forceinline__ void lcfmac(cx<R>& acc, cx<T> u, cx<R> x) {
  const R ur = bcast<R>(u.r), ui = bcast<R>(u.i), un = bcast<R>(-u.i);
  acc.r = lfma(ur, x.r, acc.r);
  acc.r = lfma(ui, x.i, acc.r);
  acc.i = lfma(ur, x.i, acc.i);
  acc.i = lfma(un, x.r, acc.i);
}
// y = u x (first term of a sum)
template <class R, class T>
__device__ __forceinline__ cx<R> lcmul(cx<T> u, cx<R> x) {
  const R ur = bcast<R>(u.r), ui = bcast<R>(u.i), un = bcast<R>(-u.i);
  return {lfma(un, x.i, ur * x.r), lfma(ui, x.r, ur * x.i)};
}
template <class R, class T>
__device__ __forceinline__ cx<R> lcmulc(cx<T> u, cx<R> x) {
  const R ur = bcast<R>(u.r), ui = bcast<R>(u.i), un = bcast<R>(-u.i);
  return {lfma(ui, x.i, ur * x.r), lfma(un, x.r, ur * x.i)};
}

// NC complex numbers of site s of one (R = T) or two fields in the chunked layout
template <class R, int NC, class T>
__device__ __forceinline__ void ld_lanes(const T* __restrict__ p0, const T* __restrict__ p1, long V, long s,
                                         cx<R> (&z)[NC]) {
  if constexpr (LaneOf<R>::n == 1) {
    ld_cx<T, NC>(p0, V, s, z);
  } else {
    const float4* a = reinterpret_cast<const float4*>(p0);
    const float4* b = reinterpret_cast<const float4*>(p1);
#pragma unroll
    for (int k = 0; k < NC / 2; ++k) {
      const float4 u = __ldg(a + k * V + s), v = __ldg(b + k * V + s);
      z[2 * k] = cx<R>{f2_pack(u.x, v.x), f2_pack(u.y, v.y)};
      z[2 * k + 1] = cx<R>{f2_pack(u.z, v.z), f2_pack(u.w, v.w)};
    }
  }
}
// the same through ordinary loads: a field that this thread has written earlier in the kernel
template <class R, int NC, class T>
__device__ __forceinline__ void ld_lanes_rw(const T* p0, const T* p1, long V, long s, cx<R> (&z)[NC]) {
  using V4 = typename std::conditional<sizeof(T) == 8, double4_16a, float4>::type;
  const V4* a = reinterpret_cast<const V4*>(p0);
  const V4* b = reinterpret_cast<const V4*>(p1);
#pragma unroll
  for (int k = 0; k < NC / 2; ++k) {
    const V4 u = a[k * V + s];
    if constexpr (LaneOf<R>::n == 1) {
      z[2 * k] = cx<R>{u.x, u.y};
      z[2 * k + 1] = cx<R>{u.z, u.w};
    } else {
      const V4 v = b[k * V + s];
      z[2 * k] = cx<R>{f2_pack(u.x, v.x), f2_pack(u.y, v.y)};
      z[2 * k + 1] = cx<R>{f2_pack(u.z, v.z), f2_pack(u.w, v.w)};
    }
  }
}
template <class R, int NC, class T>
__device__ __forceinline__ void st_lanes(T* __restrict__ p0, T* __restrict__ p1, long V, long s,
                                         const cx<R> (&z)[NC]) {
  if constexpr (LaneOf<R>::n == 1) {
    st_cx<T, NC>(p0, V, s, z);
  } else {
    float4* a = reinterpret_cast<float4*>(p0);
    float4* b = reinterpret_cast<float4*>(p1);
#pragma unroll
    for (int k = 0; k < NC / 2; ++k) {
      const float2 xr = f2_unpack(z[2 * k].r), xi = f2_unpack(z[2 * k].i);
      const float2 yr = f2_unpack(z[2 * k + 1].r), yi = f2_unpack(z[2 * k + 1].i);
      a[k * V + s] = make_float4(xr.x, xi.x, yr.x, yi.x);
      b[k * V + s] = make_float4(xr.y, xi.y, yr.y, yi.y);
    }
  }
}
// one complex number in shared memory as a single access
template <class R>
__device__ __forceinline__ cx<R> ld_shared(const cx<R>* p) {
  if constexpr (sizeof(cx<R>) == 16) {
    const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(p);
    cx<R> z;
    memcpy(&z, &u, 16);
    return z;
  } else {
    return *p;
  }
}
template <class R>
__device__ __forceinline__ void st_shared(cx<R>* p, cx<R> z) {
  if constexpr (sizeof(cx<R>) == 16) {
    ulonglong2 u;
    memcpy(&u, &z, 16);
    *reinterpret_cast<ulonglong2*>(p) = u;
  } else {
    *p = z;
  }
}

// acc += (1 -+ gamma_MU) U^(+) p (without the -1/2): FWD (1 - gamma) U p, p = psi(x + MU);
// otherwise (1 + gamma) U^dagger p, p = psi(x - MU).  p(k) returns component k, each read once.
template <class R, class T, int MU, bool FWD, class P>
__device__ __forceinline__ void hop_lanes(P p, const Link<T>& U, cx<R> (&acc)[12]) {
  cx<R> h[2][3], w[2][3];
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k)
      h[r][k] = add_ph(p(3 * r + k), p(3 * (2 + gperm(MU, r)) + k), gphase(MU, r) + (FWD ? 2 : 0));
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const cx<T> u = FWD ? U.u[a][b] : U.u[b][a];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (b == 0)
          w[r][a] = FWD ? lcmul(u, h[r][b]) : lcmulc(u, h[r][b]);
        else if (FWD)
          lcfma(w[r][a], u, h[r][b]);
        else
          lcfmac(w[r][a], u, h[r][b]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int lo = 3 * (2 + gperm(MU, r)) + k;
      acc[3 * r + k] = acc[3 * r + k] + w[r][k];
      acc[lo] = add_ph(acc[lo], w[r][k], conjph(gphase(MU, r)) + (FWD ? 2 : 0));
    }
}

// y[h] += (M + i sg mu) x for one chirality: M Hermitian 6x6 packed as 36 reals; the large
// diagonal last, so that the sums before it round at a smaller size
template <class R, class T>
__device__ __forceinline__ void herm6_lanes(const T (&m)[36], T sgmu, const cx<R>* x, cx<R>* y) {
  const R mp = bcast<R>(sgmu), mn = bcast<R>(-sgmu);
  int k = 6;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
#pragma unroll
    for (int j = i + 1; j < 6; ++j) {
      const R ur = bcast<R>(m[k]), ui = bcast<R>(m[k + 1]), un = bcast<R>(-m[k + 1]);
      k += 2;
      y[i].r = lfma(ur, x[j].r, y[i].r);
      y[i].i = lfma(ur, x[j].i, y[i].i);
      y[j].r = lfma(ur, x[i].r, y[j].r);
      y[j].i = lfma(ur, x[i].i, y[j].i);
      y[i].r = lfma(un, x[j].i, y[i].r);
      y[i].i = lfma(ui, x[j].r, y[i].i);
      y[j].r = lfma(ui, x[i].i, y[j].r);
      y[j].i = lfma(un, x[i].r, y[j].i);
    }
  }
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const R d = bcast<R>(m[i]);
    y[i].r = lfma(d, x[i].r, y[i].r);
    y[i].i = lfma(d, x[i].i, y[i].i);
    y[i].r = lfma(mn, x[i].i, y[i].r);
    y[i].i = lfma(mp, x[i].r, y[i].i);
  }
}

}  // namespace tmamg
