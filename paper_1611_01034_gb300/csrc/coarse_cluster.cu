// The whole coarsest odd-even GMRES solve (Sec. 3) in one launch, where launches and
// the host's decisions, not the arithmetic, take the time.
//
// One cluster of eight CTAs per right-hand side.  A CTA owns an eighth of the
// even and of the odd coarse sites and their slices of every vector; slices that
// neighbours read (the basis vector in work, D_oo^-1 D_oe v, the iterate) go
// through global memory (L2), inner products through distributed shared memory,
// and the steps are separated by the hardware cluster barrier.  The Hessenberg
// columns, Givens rotations and the stopping decisions are FP64 as on the host
// path, computed by every CTA from the same sums in the same order, so all of
// them decide alike.  The method is that of the host-driven solve: CGS2, restart,
// true residual per cycle, tolerance relative to the reduced right-hand side.
//
// One right-hand side on a larger system runs the same code on the whole chip: a
// cooperative launch of one CTA per SM, the inner products' partial sums in global
// memory, the steps separated by a counter that every CTA adds to and polls (with a
// limit: a CTA that runs into it stops waiting, leaves its loops and reports the
// timeout).
//
// Host-driven, an Arnoldi step takes eight launches and a decision on the host.  Here it
// takes four barriers, and what bounds it is latency: of the barriers, of L2, and of FP64,
// whose pipe a warp instruction holds for about 64 cycles however many of its lanes count.
// So FP64 work is spread over lanes and warps (sums of eight lanes each, the rotations
// kept as one matrix instead of applied one after another, the norm from the second
// projection's sums by Pythagoras) and put beside other work: the Hessenberg column is
// turned while one warp takes the norm, the next rotation is made while the others write
// the basis vector.  FP32, 24 steps from zero, us per step of the whole call with its launch,
// reduced right-hand side, odd sites and wait (at 0.3 MB 11.5 of the 13.6 are the step itself):
//
//   MB            0.3   2.4   5.3   7.2   7.4   29    59    85   118   231   340
//   host-driven    54    57    63    63    63    69    69    75   120   150   215
//   cluster       13.6  19.3  23.9  27.4  29.0  80     -     -     -     -     -
//   whole chip    19.8  22.9  25.4  27.4  26.0  28.0  32.8  35.4  50    74    92
#include <cooperative_groups.h>
#include <cuda.h>

#include "tm_kernels.h"

namespace tmamg {

namespace {

namespace cg = cooperative_groups;

constexpr int kCl = 8;            // CTAs per cluster
constexpr int kClThreads = 512;
// bytes read per step up to which eight SMs are faster than the chip with its dearer barriers
constexpr long kClMaxBytes = 6L << 20;
constexpr size_t kClSmem = 200 * 1024;
constexpr int kGridCtas = kSms;         // of the whole-chip form, one per SM
constexpr unsigned kGridPolls = 1u << 22;   // of one barrier before a CTA gives up, unless the caller sets it

struct ClLayout {  // shared memory, in bytes from its start
  size_t H, Q, g, y, hc, rc, part, dots, cf, w, bh, xs, pt, ac, nbr, site, vs, total;
  int vsm;  // the own slices of the basis are held in shared memory too
};

__host__ __device__ inline ClLayout cl_layout(int m, int nown, int n, size_t cxb) {
  ClLayout L;
  size_t o = 0;
  auto take = [&](size_t b) {
    const size_t at = o;
    o += (b + 15) / 16 * 16;
    return at;
  };
  L.H = take((size_t)(m + 1) * m * 16);
  L.g = take((size_t)(m + 1) * 16);
  L.Q = take((size_t)(m + 1) * (m + 1) * 16);
  L.hc = take((size_t)(m + 1) * 16);
  L.rc = take((size_t)(m + 1) * 16);
  L.y = take((size_t)m * 16);
  L.part = take((size_t)3 * 2 * (m + 1) * 8);  // this CTA's partial sums: two projections, norm
  L.dots = take((size_t)2 * 2 * (m + 1) * 8);  // summed projections of the two passes
  L.cf = take((size_t)(m + 1) * cxb);          // the same in T
  L.w = take((size_t)nown * n * cxb);
  L.bh = take((size_t)nown * n * cxb);
  L.xs = take((size_t)nown * 9 * n * cxb);
  L.pt = take((size_t)nown * 9 * n * cxb);
  L.ac = take((size_t)nown * n * cxb);
  L.nbr = take((size_t)2 * nown * 8 * sizeof(int));
  L.site = take((size_t)2 * nown * sizeof(int));
  const size_t vb = ((size_t)(m + 1) * nown * n * cxb + 15) / 16 * 16;
  L.vsm = o + vb <= kClSmem;
  L.vs = take(L.vsm ? vb : 0);
  L.total = o;
  return L;
}

template <typename T>
struct ClArgs {
  const T* Dc;
  const T* Dinv;
  OEGeom oe;
  const T* b;   // [rhs][Vc][n]
  T* x;         // [rhs][Vc][n]
  T* V;         // [rhs][m + 1][nc]
  T* u;         // [rhs][nc] odd work vector
  T* xe;        // [rhs][nc] even iterate
  T mu_c;
  double tol;
  int m, maxit;
  int* out;     // [rhs][2]: steps, 1 if something was not finite
  int once;     // one cycle, no true residual: exactly m steps unless the estimate reaches tol
  // whole-chip form
  double* gpart;       // [3][CTAs][2 (m + 1)] partial sums
  unsigned* count;     // barrier counter, zero at the start
  int* err;            // ERRF_TIMEOUT
  unsigned polls;      // of one barrier before a CTA gives up
};

// complex number written by another SM earlier in the kernel: from L2
__device__ __forceinline__ cx<float> ld_l2(const cx<float>* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return {v.x, v.y};
}
__device__ __forceinline__ cx<double> ld_l2(const cx<double>* p) {
  const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return {v.x, v.y};
}

// rotation of (a, b) to (rho, 0), b >= 0, by a whole warp: lane 0's rsqrt is of |a|^2, the others' of
// |a|^2 + b^2
__device__ __forceinline__ void warp_givens(cx<double> a, double b, double& c, cx<double>& s, cx<double>& rho) {
  const double a2 = a.r * a.r + a.i * a.i, n2 = a2 + b * b;
  const double r = rsqrt((threadIdx.x & 31) == 0 ? a2 : n2);
  const double ra = __shfl_sync(0xffffffffu, r, 0), rn = __shfl_sync(0xffffffffu, r, 1);
  if (b == 0) {
    c = 1;
    s = cx<double>{0, 0};
    rho = a;
  } else if (a2 == 0) {
    c = 0;
    s = cx<double>{1, 0};
    rho = cx<double>{b, 0};
  } else {
    const cx<double> ph{a.r * ra, a.i * ra};
    c = (a2 * ra) * rn;
    s = (b * rn) * ph;
    rho = (n2 * rn) * ph;
  }
}

// sum over col of B[col n] v[col], sixteen loads in flight
template <typename T>
__device__ __forceinline__ cx<T> row_dot(const cx<T>* B, const cx<T>* v, int n) {
  cx<T> acc{0, 0};
  int c = 0;
  for (; c + 16 <= n; c += 16) {
    cx<T> t[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) t[i] = B[(long)(c + i) * n];
#pragma unroll
    for (int i = 0; i < 16; ++i) cfma(acc, t[i], v[c + i]);
  }
#pragma unroll 8
  for (; c < n; ++c) cfma(acc, B[(long)c * n], v[c]);
  return acc;
}

template <typename T, bool GRID>
__device__ __forceinline__ void coarse_gmres(const ClArgs<T>& a) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int parts = GRID ? (int)gridDim.x : kCl;
  const int rank = GRID ? blockIdx.x : blockIdx.x % kCl, rhs = GRID ? 0 : blockIdx.x / kCl, tid = threadIdx.x;
  __shared__ int dead;  // this CTA gave up waiting
  if (tid == 0) dead = 0;
  unsigned epoch = 0;
  auto barrier = [&]() {
    if constexpr (GRID) {
      ++epoch;
      __syncthreads();
      if (tid == 0 && !dead) {
        __threadfence();
        atomicAdd(a.count, 1u);
        const unsigned target = epoch * gridDim.x;
        unsigned polls = 0, seen;
        do {
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.count) : "memory");
        } while (seen < target && ++polls < a.polls);
        if (seen < target) {
          dead = 1;
          atomicOr(a.err, ERRF_TIMEOUT);
        }
        __threadfence();
      }
      __syncthreads();
    } else {
      cg::this_cluster().sync();
    }
  };
  const int n = 2 * a.oe.nv, nh = a.oe.nhalf, m = a.m;
  const int q = (nh + parts - 1) / parts, k0 = min(rank * q, nh), nown = min(q, nh - k0);  // own compact sites
  const long nc = (long)nh * n;
  const ClLayout L = cl_layout(m, q, n, sizeof(cx<T>));
  cx<double>* H = reinterpret_cast<cx<double>*>(sm + L.H);
  cx<double>* g = reinterpret_cast<cx<double>*>(sm + L.g);
  double* Q = reinterpret_cast<double*>(sm + L.Q);    // product of the rotations, row stride 2 (m + 1)
  double* hc = reinterpret_cast<double*>(sm + L.hc);  // a Hessenberg column
  double* rc = reinterpret_cast<double*>(sm + L.rc);  // Q times it
  cx<double>* y = reinterpret_cast<cx<double>*>(sm + L.y);
  double* part = reinterpret_cast<double*>(sm + L.part);
  double* dots = reinterpret_cast<double*>(sm + L.dots);
  cx<T>* w = reinterpret_cast<cx<T>*>(sm + L.w);
  cx<T>* bh = reinterpret_cast<cx<T>*>(sm + L.bh);
  cx<T>* xs = reinterpret_cast<cx<T>*>(sm + L.xs);
  cx<T>* pt = reinterpret_cast<cx<T>*>(sm + L.pt);
  cx<T>* ac = reinterpret_cast<cx<T>*>(sm + L.ac);
  int* nbr = reinterpret_cast<int*>(sm + L.nbr);  // [parity][own site][8] compact neighbours
  int* site = reinterpret_cast<int*>(sm + L.site);  // [parity][own site] coarse sites
  cx<T>* cf = reinterpret_cast<cx<T>*>(sm + L.cf);
  __shared__ double red[kClThreads / 32];
  __shared__ int flag;
  const int pstr = 2 * (m + 1);
  const cx<T>* Dc = reinterpret_cast<const cx<T>*>(a.Dc);
  const cx<T>* Di = reinterpret_cast<const cx<T>*>(a.Dinv);
  const cx<T>* b = reinterpret_cast<const cx<T>*>(a.b) + (long)rhs * a.oe.gc.V * n;
  cx<T>* x = reinterpret_cast<cx<T>*>(a.x) + (long)rhs * a.oe.gc.V * n;
  cx<T>* V = reinterpret_cast<cx<T>*>(a.V) + (long)rhs * (m + 1) * nc;
  cx<T>* u = reinterpret_cast<cx<T>*>(a.u) + rhs * nc;
  cx<T>* xe = reinterpret_cast<cx<T>*>(a.xe) + rhs * nc;
  const int own = nown * n;           // own complex numbers of a compact vector
  const long o0 = (long)k0 * n;       // their offset
  // own slices of the basis: in shared memory where they fit, else the global ones
  cx<T>* Vo = L.vsm ? reinterpret_cast<cx<T>*>(sm + L.vs) : V + o0;
  const long vst = L.vsm ? own : nc;
  for (int e = tid; e < 2 * nown; e += kClThreads)
    site[e] = e < nown ? a.oe.even_site[k0 + e] : a.oe.odd_site[k0 + e - nown];
  __syncthreads();
  auto site_of = [&](int odd, int k) { return site[odd * nown + k]; };

  for (int e = tid; e < 2 * nown * 8; e += kClThreads) {
    const int odd = e / (nown * 8), k = (e / 8) % nown, t = e % 8;
    const int s = site_of(odd, k);
    int c[4];
    site_coords(a.oe.gc, s, c);
    const int mu = t >> 1;
    nbr[e] = a.oe.cidx[(t & 1) ? nb_bwd(a.oe.gc, s, c, mu) : nb_fwd(a.oe.gc, s, c, mu)];
  }
  __syncthreads();

  // out = sum of the 8 hops (and, with self, the self block times v's own slice) of src at the own
  // sites of one parity
  auto blocks = [&](int odd, const cx<T>* src, const cx<T>* self, cx<T>* out) {
    for (int e = tid; e < nown * 9 * n; e += kClThreads) {
      const int k = e / (9 * n), t = (e / n) % 9, col = e % n;
      cx<T> v{0, 0};
      if (t > 0)
        v = ld_l2(src + (long)nbr[(odd * nown + k) * 8 + t - 1] * n + col);
      else if (self)
        v = ld_l2(self + (long)(k0 + k) * n + col);
      xs[e] = v;
    }
    __syncthreads();
    for (int e = tid; e < nown * 9 * n; e += kClThreads) {
      const int k = e / (9 * n), t = (e / n) % 9, row = e % n;
      if (t > 0 || self) pt[e] = row_dot(Dc + ((long)site_of(odd, k) * 9 + t) * n * n + row, xs + (e - row), n);
    }
    __syncthreads();
    for (int e = tid; e < own; e += kClThreads) {
      const int k = e / n, row = e % n;
      cx<T> hop = pt[(k * 9 + 1) * n + row];
#pragma unroll
      for (int t = 2; t < 9; ++t) hop = hop + pt[(k * 9 + t) * n + row];
      if (self) {
        cx<T> d = pt[k * 9 * n + row];
        const cx<T> v = xs[k * 9 * n + row];
        const T sg = row < n / 2 ? -a.mu_c : a.mu_c;  // i mu_c Gamma5_c
        d.r -= sg * v.i;
        d.i += sg * v.r;
        out[e] = d - hop;
      } else {
        out[e] = hop;
      }
    }
    __syncthreads();
  };
  // out[own odd site] = D_oo^-1 ac
  auto dinv = [&](cx<T>* out, bool full) {
    for (int e = tid; e < own; e += kClThreads) {
      const int k = e / n, row = e % n;
      const cx<T> acc = row_dot(Di + (long)(k0 + k) * n * n + row, ac + k * n, n);
      if (full)
        out[(long)site_of(1, k) * n + row] = acc;
      else
        out[(long)(k0 + k) * n + row] = acc;
    }
  };
  // w = S v for the even vector v in global memory (every slice visible)
  auto schur = [&](const cx<T>* v) {
    blocks(1, v, nullptr, ac);
    dinv(u, false);
    barrier();
    blocks(0, u, v, w);
  };
  // sum over the CTAs of cnt partial sums at part + at, into to (every thread may read them after)
  // and, in T, into tt
  auto gather = [&](int at, int cnt, double* to, T* tt) {
    if constexpr (GRID) {
      double* gp = a.gpart + (long)(at / pstr) * parts * pstr;  // [CTA][2 (m + 1)]
      __syncthreads();
      for (int e = tid; e < cnt; e += kClThreads) gp[(long)rank * pstr + e] = part[at + e];
      barrier();
    } else {
      barrier();
    }
    // eight lanes per sum, each a fixed eighth of the CTAs (a warp's FP64 instruction holds its
    // scheduler's pipe for 64 cycles however many lanes are active, so they are counted)
    const int sub = tid & 7;
    for (int e0 = 0; e0 < cnt; e0 += kClThreads / 8) {
      if (e0 + ((tid & ~31) >> 3) >= cnt) break;
      const int e = e0 + (tid >> 3);
      double s = 0;
      if (e < cnt) {
        if constexpr (GRID) {
          const double* gp = a.gpart + (long)(at / pstr) * parts * pstr;
#pragma unroll 16
          for (int c = sub; c < parts; c += 8) s += __ldcg(gp + (long)c * pstr + e);
        } else {
          s = cg::this_cluster().map_shared_rank(part, sub)[at + e];
        }
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (e < cnt && sub == 0) {
        to[e] = s;
        if (tt) tt[e] = (T)s;
      }
    }
    __syncthreads();
  };
  // V_0..k^H w summed over the CTAs into to (and into cf in T), with |w|^2 behind them
  auto project = [&](int k, int pass, double* to) {
    const int warp = tid >> 5, lane = tid & 31;
    for (int j = warp; j <= k + pass; j += kClThreads / 32) {
      const cx<T>* Vj = j <= k ? Vo + j * vst : w;
      cx<T> d{0, 0};
      for (int i = lane; i < own; i += 32) cfmac(d, Vj[i], w[i]);
      // the lower lanes sum the real parts, the upper ones the imaginary parts
      const bool hi = lane & 16;
      double t = hi ? d.i : d.r;
      t += __shfl_xor_sync(0xffffffffu, hi ? d.r : d.i, 16);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if ((lane & 15) == 0) part[pass * pstr + 2 * j + hi] = t;
    }
    gather(pass * pstr, 2 * (k + 1) + pass, to, reinterpret_cast<T*>(cf));
  };
  // w -= V_0..k cf
  auto subtract = [&](int k) {
    for (int i = tid; i < own; i += kClThreads) {
      cx<T> acc = w[i];
#pragma unroll 4
      for (int j = 0; j <= k; ++j) cfma(acc, -cf[j], Vo[j * vst + i]);
      w[i] = acc;
    }
  };
  __shared__ double nrm2, nrm;  // |w|^2, |w|
  __shared__ T inv;             // 1 / |w|, 0 for w = 0
  __shared__ int st;            // of the norm: 0 usable, 1 not finite, 2 to be summed anew
  auto norm_of = [&](const cx<T>* v) {  // leaves nrm, inv and st
    T s = 0;
    for (int i = tid; i < own; i += kClThreads) s += norm2(v[i]);
    double d = s;
    if ((tid & ~31) < own) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    }
    if ((tid & 31) == 0) red[tid >> 5] = d;
    __syncthreads();
    if (tid < 32) {
      double t = tid < kClThreads / 32 ? red[tid] : 0.0;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (tid == 0) part[2 * pstr] = t;
    }
    gather(2 * pstr, 1, &nrm2, nullptr);
    if (tid == 0) {
      const double r = rsqrt(nrm2);
      nrm = nrm2 > 0 ? nrm2 * r : nrm2;
      inv = nrm2 > 0 ? (T)r : T(0);
      st = isfinite(nrm2) ? 0 : 1;
    }
    __syncthreads();
  };
  // own slice of v_j = v / |v| for element i
  auto put = [&](int j, int i, cx<T> v) {
    v = inv * v;
    V[j * nc + o0 + i] = v;
    if (L.vsm) Vo[j * vst + i] = v;
  };

  // reduced right-hand side b_e - D_eo D_oo^-1 b_o, iterate 0
  for (int e = tid; e < own; e += kClThreads) {
    ac[e] = b[(long)site_of(1, e / n) * n + e % n];
    xe[o0 + e] = cx<T>{0, 0};
  }
  __syncthreads();
  dinv(u, false);
  barrier();
  blocks(0, u, nullptr, ac);
  for (int e = tid; e < own; e += kClThreads) bh[e] = b[(long)site_of(0, e / n) * n + e % n] - ac[e];
  __syncthreads();
  norm_of(bh);
  const double bnorm = nrm;
  double beta = bnorm;
  int iters = 0, bad = st;
  for (int e = tid; e < own; e += kClThreads) w[e] = bh[e];
  __syncthreads();
  while (!bad && !dead && bnorm > 0 && beta > a.tol * bnorm && iters < a.maxit) {
    for (int i = tid; i < own; i += kClThreads) put(0, i, w[i]);
    if (tid == 0) {
      g[0] = cx<double>{beta, 0.0};
      Q[0] = 1;
      Q[1] = 0;
    }
    barrier();
    int k = 0;
    for (;; ++k) {
      schur(V + k * nc);
      project(k, 0, dots);
      subtract(k);
      __syncthreads();
      project(k, 1, dots + pstr);
      // |w|^2 after the second pass is the one before it less that of the projections; where little of
      // it is left (a basis that spans nearly everything) it is summed anew
      const double* d2 = dots + pstr;
      if (tid < 32) {
        T s = 0;
        for (int j = tid; j <= k; j += 32) s += norm2(cf[j]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (tid == 0) {
          const double ww = d2[2 * (k + 1)], h2 = ww - s;
          const double r = rsqrt(h2);
          nrm = h2 > 0 ? h2 * r : 0.0;
          inv = h2 > 0 ? (T)r : T(0);
          st = !isfinite(ww) ? 1 : (h2 >= 0.25 * ww ? 0 : 2);
        }
      } else {
        // meanwhile the others: the Hessenberg column, turned by the rotations so far
        for (int j = tid - 32; j < 2 * (k + 1); j += kClThreads - 32) hc[j] = dots[j] + d2[j];
        asm volatile("bar.sync 1, %0;" ::"n"(kClThreads - 32) : "memory");
        const int sub = tid & 7;  // eight lanes per row and component
        for (int e0 = 0; e0 < 2 * (k + 1); e0 += (kClThreads - 32) / 8) {
          const int e = e0 + ((tid - 32) >> 3), row = e >> 1;
          if (e0 + (((tid - 32) & ~31) >> 3) >= 2 * (k + 1)) break;
          double s = 0;
          if (row <= k)
            for (int i = sub; i <= k; i += 8) {
              const double qr = Q[row * pstr + 2 * i], qi = Q[row * pstr + 2 * i + 1];
              s += qr * hc[2 * i + (e & 1)];
              s += ((e & 1) ? qi : -qi) * hc[2 * i + 1 - (e & 1)];
            }
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (row <= k && sub == 0) rc[e] = s;
        }
      }
      __syncthreads();
      const int again = st;
      if (again) {
        subtract(k);
        __syncthreads();
        norm_of(w);
      }
      if (st || dead) {
        bad = 1;
        break;
      }
      // the last warp makes the next rotation while the others write v_k+1
      if (tid >= kClThreads - 32) {
        const int lane = tid & 31;
        double c;
        cx<double> s, rho;
        warp_givens(cx<double>{rc[2 * k], rc[2 * k + 1]}, nrm, c, s, rho);
        for (int j = lane; j < k; j += 32) H[j * m + k] = cx<double>{rc[2 * j], rc[2 * j + 1]};
        cx<double>* q0 = reinterpret_cast<cx<double>*>(Q + k * pstr);
        cx<double>* q1 = reinterpret_cast<cx<double>*>(Q + (k + 1) * pstr);
        for (int i = lane; i <= k; i += 32) {
          const cx<double> v = q0[i];
          q0[i] = c * v;
          q1[i] = -cmulc(s, v);
        }
        for (int j = lane; j <= k; j += 32) reinterpret_cast<cx<double>*>(Q + j * pstr)[k + 1] = j == k ? s : cx<double>{0, 0};
        if (lane == 0) {
          q1[k + 1] = cx<double>{c, 0};
          H[k * m + k] = rho;
          const cx<double> g1 = -cmulc(s, g[k]);
          g[k + 1] = g1;
          g[k] = c * g[k];
          const double lim = a.tol * bnorm;
          flag = nrm == 0 || g1.r * g1.r + g1.i * g1.i <= lim * lim || iters + 1 >= a.maxit || k + 1 >= m;
        }
      }
      if (again) {
        for (int i = tid; i < own; i += kClThreads) put(k + 1, i, w[i]);
      } else {
        for (int i = tid; i < own; i += kClThreads) {
          cx<T> acc = w[i];
#pragma unroll 4
          for (int j = 0; j <= k; ++j) cfma(acc, -cf[j], Vo[j * vst + i]);
          put(k + 1, i, acc);
        }
      }
      ++iters;
      barrier();
      if (flag) break;
    }
    if (bad) break;
    ++k;  // steps of this cycle
    // back substitution, column by column: lane l holds rows l and l + 32
    if (tid < 32) {
      cx<double> acc[2], dc[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int i = tid + 32 * r;
        acc[r] = dc[r] = cx<double>{0, 0};
        if (i < k) {
          acc[r] = g[i];
          const cx<double> d = H[i * m + i];
          const double dn = d.r * d.r + d.i * d.i, rd = dn > 0 ? 1.0 / dn : 0.0;
          dc[r] = cx<double>{d.r * rd, -d.i * rd};  // 1 / H_ii, 0 for H_ii = 0
        }
      }
      for (int i = k - 1; i >= 0; --i) {
        const cx<double> yo = (i < 32 ? acc[0] : acc[1]) * (i < 32 ? dc[0] : dc[1]);
        const cx<double> yi{__shfl_sync(0xffffffffu, yo.r, i & 31), __shfl_sync(0xffffffffu, yo.i, i & 31)};
        if (tid == 0) y[i] = yi;
        if (tid < i) acc[0] = acc[0] - H[tid * m + i] * yi;
        if (i > 32 && tid + 32 < i) acc[1] = acc[1] - H[(tid + 32) * m + i] * yi;
      }
    }
    __syncthreads();
    if (tid < k) cf[tid] = cx<T>{(T)y[tid].r, (T)y[tid].i};
    __syncthreads();
    for (int i = tid; i < own; i += kClThreads) {
      cx<T> acc = xe[o0 + i];
#pragma unroll 4
      for (int j = 0; j < k; ++j) cfma(acc, cf[j], Vo[j * vst + i]);
      xe[o0 + i] = acc;
    }
    barrier();
    if (a.once) break;
    // true residual of the reduced system
    schur(xe);
    for (int e = tid; e < own; e += kClThreads) w[e] = bh[e] - w[e];
    __syncthreads();
    norm_of(w);
    beta = nrm;
    bad = st;
  }
  if (a.once && (bad || dead))  // the caller has no other sign of it
    for (int i = tid; i < own; i += kClThreads) xe[o0 + i] = cx<T>{(T)NAN, (T)NAN};
  barrier();
  // x_e, then x_o = D_oo^-1 (b_o - D_oe x_e); NaN from a CTA that gave up, whose neighbours' x_e may be old
  blocks(1, xe, nullptr, ac);
  for (int e = tid; e < own; e += kClThreads) {
    const int k = e / n, row = e % n;
    x[(long)site_of(0, k) * n + row] = dead ? cx<T>{(T)NAN, (T)NAN} : xe[o0 + e];
    ac[e] = b[(long)site_of(1, k) * n + row] - ac[e];
  }
  __syncthreads();
  dinv(x, true);
  if (rank == 0 && tid == 0) {
    a.out[2 * rhs] = iters;
    a.out[2 * rhs + 1] = bad;
  }
  if constexpr (!GRID) barrier();  // no CTA leaves while another may read its partial sums
}

template <typename T>
__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(kClThreads) k_coarse_gmres(ClArgs<T> a) {
  coarse_gmres<T, false>(a);
}
template <typename T>
__global__ void __launch_bounds__(kClThreads, 1) k_coarse_gmres_grid(ClArgs<T> a) {
  coarse_gmres<T, true>(a);
}

}  // namespace

namespace {
long step_bytes(const OEGeom& oe, size_t real_bytes) {
  // 17 of the 18 blocks of a site pair and the odd inverse
  const long n = 2 * oe.nv;
  return (long)oe.nhalf * 18 * n * n * 2 * (long)real_bytes;
}
}  // namespace

namespace {
template <typename F>
F driver_call(const char* name, unsigned version) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult found;
  if (cudaGetDriverEntryPointByVersion(name, &p, version, cudaEnableDefault, &found) != cudaSuccess ||
      found != cudaDriverEntryPointSuccess) {
    cudaGetLastError();
    p = nullptr;
  }
  return reinterpret_cast<F>(p);
}

// SMs that work on this stream may run on (a green context has a part of the device's), and how
// many of them are certain to share a cluster; false if the driver does not say (about 1 us)
bool stream_sms(cudaStream_t st, int* sms, int* together) {
  static const auto get_ctx =
      driver_call<CUresult (*)(CUstream, CUcontext*, CUgreenCtx*)>("cuStreamGetCtx", 12050);
  static const auto ctx_res =
      driver_call<CUresult (*)(CUcontext, CUdevResource*, CUdevResourceType)>("cuCtxGetDevResource", 12040);
  static const auto green_res =
      driver_call<CUresult (*)(CUgreenCtx, CUdevResource*, CUdevResourceType)>("cuGreenCtxGetDevResource", 12040);
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  CUdevResource r{};
  if (!get_ctx || !ctx_res || !green_res) return false;
  // in a thread's first call with the default stream no context is current yet: cudaFree(0) makes it so
  if (get_ctx(st, &ctx, &green) != CUDA_SUCCESS &&
      (cudaFree(nullptr) != cudaSuccess || get_ctx(st, &ctx, &green) != CUDA_SUCCESS))
    return false;
  if ((green ? green_res(green, &r, CU_DEV_RESOURCE_TYPE_SM) : ctx_res(ctx, &r, CU_DEV_RESOURCE_TYPE_SM)) != CUDA_SUCCESS)
    return false;
  *sms = (int)r.sm.smCount;
  *together = (int)r.sm.smCoscheduledAlignment;
  return true;
}
}  // namespace

bool coarse_cluster_fits(const OEGeom& oe, int restart, int nrhs, size_t real_bytes, cudaStream_t st) {
  const int q = (oe.nhalf + kCl - 1) / kCl;
  if (restart > kCoarseOneLaunchSteps || step_bytes(oe, real_bytes) > kClMaxBytes || nrhs * kCl > kSms ||
      cl_layout(restart, q, 2 * oe.nv, 2 * real_bytes).total > kClSmem)
    return false;
  int sms = 0, together = 0;
  return stream_sms(st, &sms, &together) && together >= kCl;  // a cluster's CTAs take an SM each
}

bool coarse_grid_fits(const OEGeom& oe, int restart, size_t real_bytes, cudaStream_t st) {
  int sms = 0, together = 0;
  if (!stream_sms(st, &sms, &together) || sms < kGridCtas) return false;  // all CTAs have to be resident
  const int q = (oe.nhalf + kGridCtas - 1) / kGridCtas;
  return restart <= kCoarseOneLaunchSteps && cl_layout(restart, q, 2 * oe.nv, 2 * real_bytes).total <= kClSmem;
}
long coarse_grid_scratch_doubles(int restart) { return 3L * kGridCtas * 2 * (restart + 1) + 1; }

template <typename T>
void launch_coarse_gmres(const T* Dc, const T* Dinv, const T* b, T* x, T* V, T* u, T* xe, int* out, const OEGeom& oe,
                         double mu_c, double tol, int restart, int maxit, int nrhs, cudaStream_t st) {
  const int q = (oe.nhalf + kCl - 1) / kCl;
  const size_t smem = cl_layout(restart, q, 2 * oe.nv, 2 * sizeof(T)).total;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_coarse_gmres<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmem);
    attr = true;
  }
  ClArgs<T> a{Dc, Dinv, oe, b, x, V, u, xe, (T)mu_c, tol, restart, maxit, out, 0, nullptr, nullptr, nullptr, 0};
  k_coarse_gmres<T><<<kCl * nrhs, kClThreads, smem, st>>>(a);
}

template <typename T>
void launch_coarse_gmres_grid(const T* Dc, const T* Dinv, const T* b, T* x, T* V, T* u, T* xe, int* out,
                              double* scratch, int* err, const OEGeom& oe, double mu_c, double tol, int restart,
                              int maxit, bool once, cudaStream_t st, unsigned polls) {
  const int q = (oe.nhalf + kGridCtas - 1) / kGridCtas, ctas = (oe.nhalf + q - 1) / q;
  const size_t smem = cl_layout(restart, q, 2 * oe.nv, 2 * sizeof(T)).total;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_coarse_gmres_grid<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmem);
    attr = true;
  }
  unsigned* count = reinterpret_cast<unsigned*>(scratch);
  cudaMemsetAsync(count, 0, sizeof(double), st);
  ClArgs<T> a{Dc, Dinv, oe, b, x, V, u, xe, (T)mu_c, tol, restart, maxit, out, once ? 1 : 0, scratch + 1, count, err,
              polls ? polls : kGridPolls};
  void* args[] = {&a};
  cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_coarse_gmres_grid<T>), dim3(ctas), dim3(kClThreads), args,
                              smem, st);
}
#define TM_INST(T)                                                                                                    \
  template void launch_coarse_gmres<T>(const T*, const T*, const T*, T*, T*, T*, T*, int*, const OEGeom&, double,     \
                                       double, int, int, int, cudaStream_t);                                          \
  template void launch_coarse_gmres_grid<T>(const T*, const T*, const T*, T*, T*, T*, T*, int*, double*, int*,        \
                                            const OEGeom&, double, double, int, int, bool, cudaStream_t, unsigned);
TM_INST(double)
TM_INST(float)
#undef TM_INST

}  // namespace tmamg
