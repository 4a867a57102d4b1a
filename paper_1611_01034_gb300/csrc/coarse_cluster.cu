// The whole coarsest odd-even GMRES solve (Sec. 3) in one launch, for coarse
// systems so small that launches and the host's decisions, not the arithmetic,
// take the time.
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
// An Arnoldi step took eight launches and a host decision (about 55 us); here it
// takes five cluster barriers.
#include <cooperative_groups.h>

#include "tm_kernels.h"

namespace tmamg {

namespace {

namespace cg = cooperative_groups;

constexpr int kCl = 8;            // CTAs per cluster
constexpr int kClThreads = 512;
constexpr int kClMaxRestart = 48;  // Hessenberg matrix in shared memory
constexpr long kClMaxBytes = 6L << 20;  // coarse operator read per step through eight SMs

struct ClLayout {  // shared memory, in bytes from its start
  size_t H, g, cs, sn, y, part, dots, w, bh, xs, pt, ac, nbr, total;
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
  L.cs = take((size_t)m * 8);
  L.sn = take((size_t)m * 16);
  L.y = take((size_t)m * 16);
  L.part = take((size_t)3 * 2 * (m + 1) * 8);  // this CTA's partial sums: two projections, norm
  L.dots = take((size_t)2 * 2 * (m + 1) * 8);  // summed projections of the two passes
  L.w = take((size_t)nown * n * cxb);
  L.bh = take((size_t)nown * n * cxb);
  L.xs = take((size_t)nown * 9 * n * cxb);
  L.pt = take((size_t)nown * 9 * n * cxb);
  L.ac = take((size_t)nown * n * cxb);
  L.nbr = take((size_t)2 * nown * 8 * sizeof(int));
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

__device__ __forceinline__ void cl_givens(cx<double> a, double b, double& c, cx<double>& s, cx<double>& rho) {
  const double aa = sqrt(a.r * a.r + a.i * a.i);
  if (b == 0) {
    c = 1;
    s = cx<double>{0, 0};
    rho = a;
  } else if (aa == 0) {
    c = 0;
    s = cx<double>{1, 0};
    rho = cx<double>{b, 0};
  } else {
    const double nu = hypot(aa, b);
    c = aa / nu;
    const cx<double> ph{a.r / aa, a.i / aa};
    s = (b / nu) * ph;
    rho = nu * ph;
  }
}

template <typename T>
__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(kClThreads) k_coarse_gmres(ClArgs<T> a) {
  extern __shared__ __align__(16) unsigned char sm[];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = blockIdx.x % kCl, rhs = blockIdx.x / kCl, tid = threadIdx.x;
  const int n = 2 * a.oe.nv, nh = a.oe.nhalf, m = a.m;
  const int q = (nh + kCl - 1) / kCl, k0 = min(rank * q, nh), nown = min(q, nh - k0);  // own compact sites
  const long nc = (long)nh * n;
  const ClLayout L = cl_layout(m, q, n, sizeof(cx<T>));
  cx<double>* H = reinterpret_cast<cx<double>*>(sm + L.H);
  cx<double>* g = reinterpret_cast<cx<double>*>(sm + L.g);
  double* cs = reinterpret_cast<double*>(sm + L.cs);
  cx<double>* sn = reinterpret_cast<cx<double>*>(sm + L.sn);
  cx<double>* y = reinterpret_cast<cx<double>*>(sm + L.y);
  double* part = reinterpret_cast<double*>(sm + L.part);
  double* dots = reinterpret_cast<double*>(sm + L.dots);
  cx<T>* w = reinterpret_cast<cx<T>*>(sm + L.w);
  cx<T>* bh = reinterpret_cast<cx<T>*>(sm + L.bh);
  cx<T>* xs = reinterpret_cast<cx<T>*>(sm + L.xs);
  cx<T>* pt = reinterpret_cast<cx<T>*>(sm + L.pt);
  cx<T>* ac = reinterpret_cast<cx<T>*>(sm + L.ac);
  int* nbr = reinterpret_cast<int*>(sm + L.nbr);  // [parity][own site][8] compact neighbours
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
  auto site_of = [&](int odd, int k) { return odd ? a.oe.odd_site[k0 + k] : a.oe.even_site[k0 + k]; };

  for (int e = tid; e < 2 * nown * 8; e += kClThreads) {
    const int odd = e / (nown * 8), k = (e / 8) % nown, t = e % 8;
    const int s = site_of(odd, k);
    int c[4];
    site_coords(a.oe.gc, s, c);
    const int mu = t >> 1;
    nbr[e] = a.oe.cidx[(t & 1) ? nb_bwd(a.oe.gc, s, c, mu) : nb_fwd(a.oe.gc, s, c, mu)];
  }
  __syncthreads();

  // ac = sum of the 8 hops (and, with self, the self block times v's own slice) of src at the own
  // sites of one parity
  auto blocks = [&](int odd, const cx<T>* src, const cx<T>* self) {
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
      cx<T> acc{0, 0};
      if (t > 0 || self) {
        const cx<T>* B = Dc + ((long)site_of(odd, k) * 9 + t) * n * n + row;
        const cx<T>* v = xs + (e - row);
#pragma unroll 8
        for (int col = 0; col < n; ++col) cfma(acc, B[(long)col * n], v[col]);
      }
      pt[e] = acc;
    }
    __syncthreads();
    for (int e = tid; e < own; e += kClThreads) {
      const int k = e / n, row = e % n;
      cx<T> hop = pt[(k * 9 + 1) * n + row];
      for (int t = 2; t < 9; ++t) hop = hop + pt[(k * 9 + t) * n + row];
      if (self) {
        cx<T> d = pt[k * 9 * n + row];
        const cx<T> v = xs[k * 9 * n + row];
        const T sg = row < n / 2 ? -a.mu_c : a.mu_c;  // i mu_c Gamma5_c
        d.r -= sg * v.i;
        d.i += sg * v.r;
        ac[e] = d - hop;
      } else {
        ac[e] = hop;
      }
    }
    __syncthreads();
  };
  // out[own odd site] = D_oo^-1 ac
  auto dinv = [&](cx<T>* out, bool full) {
    for (int e = tid; e < own; e += kClThreads) {
      const int k = e / n, row = e % n;
      const cx<T>* M = Di + (long)(k0 + k) * n * n + row;
      cx<T> acc{0, 0};
#pragma unroll 8
      for (int col = 0; col < n; ++col) cfma(acc, M[(long)col * n], ac[k * n + col]);
      if (full)
        out[(long)site_of(1, k) * n + row] = acc;
      else
        out[(long)(k0 + k) * n + row] = acc;
    }
  };
  // w = S v for the even vector v in global memory (every slice visible)
  auto schur = [&](const cx<T>* v) {
    blocks(1, v, nullptr);
    dinv(u, false);
    cluster.sync();
    blocks(0, u, v);
    for (int e = tid; e < own; e += kClThreads) w[e] = ac[e];
    __syncthreads();
  };
  // sum over the cluster of cnt partial sums at part + at, into to (every thread may read them after)
  auto gather = [&](int at, int cnt, double* to) {
    cluster.sync();
    for (int e = tid; e < cnt; e += kClThreads) {
      double v[kCl], s = 0;
#pragma unroll
      for (int c = 0; c < kCl; ++c) v[c] = cluster.map_shared_rank(part, c)[at + e];
#pragma unroll
      for (int c = 0; c < kCl; ++c) s += v[c];
      to[e] = s;
    }
    __syncthreads();
  };
  // w -= V_0..k (V^H w), the projections left in to
  auto project = [&](int k, int pass, double* to) {
    const int warp = tid >> 5, lane = tid & 31;
    for (int j = warp; j <= k; j += kClThreads / 32) {
      const cx<T>* Vj = V + j * nc + o0;
      cx<T> d{0, 0};
      for (int i = lane; i < own; i += 32) cfmac(d, Vj[i], w[i]);
      double dr = d.r, di = d.i;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        dr += __shfl_xor_sync(0xffffffffu, dr, o);
        di += __shfl_xor_sync(0xffffffffu, di, o);
      }
      if (lane == 0) {
        part[pass * pstr + 2 * j] = dr;
        part[pass * pstr + 2 * j + 1] = di;
      }
    }
    gather(pass * pstr, 2 * (k + 1), to);
    for (int i = tid; i < own; i += kClThreads) {
      cx<T> acc = w[i];
      for (int j = 0; j <= k; ++j) {
        const cx<T> c{(T)to[2 * j], (T)to[2 * j + 1]};
        cfma(acc, -c, V[j * nc + o0 + i]);
      }
      w[i] = acc;
    }
    __syncthreads();
  };
  __shared__ double nrm2;
  auto norm2_w = [&](const cx<T>* v) {
    T s = 0;
    for (int i = tid; i < own; i += kClThreads) s += norm2(v[i]);
    double d = s;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if ((tid & 31) == 0) red[tid >> 5] = d;
    __syncthreads();
    if (tid == 0) {
      double t = 0;
      for (int k = 0; k < kClThreads / 32; ++k) t += red[k];
      part[2 * pstr] = t;
    }
    gather(2 * pstr, 1, &nrm2);
    return nrm2;
  };
  // own slice of v_j = src / |src|, visible to the cluster
  auto put_basis = [&](int j, const cx<T>* src, double nrm) {
    const T inv = nrm > 0 ? (T)(1.0 / nrm) : T(0);
    for (int i = tid; i < own; i += kClThreads) V[j * nc + o0 + i] = inv * src[i];
    cluster.sync();
  };

  // reduced right-hand side b_e - D_eo D_oo^-1 b_o, iterate 0
  for (int e = tid; e < own; e += kClThreads) {
    ac[e] = b[(long)site_of(1, e / n) * n + e % n];
    xe[o0 + e] = cx<T>{0, 0};
  }
  __syncthreads();
  dinv(u, false);
  cluster.sync();
  blocks(0, u, nullptr);
  for (int e = tid; e < own; e += kClThreads) bh[e] = b[(long)site_of(0, e / n) * n + e % n] - ac[e];
  __syncthreads();
  const double bnorm = sqrt(norm2_w(bh));
  double beta = bnorm;
  int iters = 0, bad = isfinite(bnorm) ? 0 : 1;
  for (int e = tid; e < own; e += kClThreads) w[e] = bh[e];
  __syncthreads();
  while (!bad && bnorm > 0 && beta > a.tol * bnorm && iters < a.maxit) {
    put_basis(0, w, beta);
    if (tid == 0)
      for (int j = 0; j <= m; ++j) g[j] = cx<double>{j == 0 ? beta : 0.0, 0.0};
    int k = 0;
    for (;; ++k) {
      schur(V + k * nc);
      project(k, 0, dots);
      project(k, 1, dots + pstr);
      const double hn = sqrt(norm2_w(w));
      if (!isfinite(hn)) {
        bad = 1;
        break;
      }
      if (tid == 0) {
        const double* d1 = dots;
        const double* d2 = dots + pstr;
        cx<double> c0{d1[0] + d2[0], d1[1] + d2[1]};
        for (int j = 0; j < k; ++j) {
          const cx<double> c1{d1[2 * j + 2] + d2[2 * j + 2], d1[2 * j + 3] + d2[2 * j + 3]};
          H[j * m + k] = cs[j] * c0 + sn[j] * c1;
          c0 = cs[j] * c1 - cmulc(sn[j], c0);
        }
        double c;
        cx<double> s, rho;
        cl_givens(c0, hn, c, s, rho);
        cs[k] = c;
        sn[k] = s;
        H[k * m + k] = rho;
        g[k + 1] = -cmulc(s, g[k]);
        g[k] = c * g[k];
        const double res = sqrt(g[k + 1].r * g[k + 1].r + g[k + 1].i * g[k + 1].i);
        flag = hn == 0 || res <= a.tol * bnorm || iters + 1 >= a.maxit || k + 1 >= m;
      }
      ++iters;
      __syncthreads();
      if (flag) break;
      put_basis(k + 1, w, hn);
    }
    if (bad) break;
    ++k;  // steps of this cycle
    if (tid == 0) {
      for (int i = k - 1; i >= 0; --i) {
        cx<double> acc = g[i];
        for (int j = i + 1; j < k; ++j) acc = acc - H[i * m + j] * y[j];
        const cx<double> d = H[i * m + i];
        const double dn = d.r * d.r + d.i * d.i;
        y[i] = dn > 0 ? cx<double>{(acc.r * d.r + acc.i * d.i) / dn, (acc.i * d.r - acc.r * d.i) / dn}
                      : cx<double>{0, 0};
      }
    }
    __syncthreads();
    for (int i = tid; i < own; i += kClThreads) {
      cx<T> acc = xe[o0 + i];
      for (int j = 0; j < k; ++j) cfma(acc, cx<T>{(T)y[j].r, (T)y[j].i}, V[j * nc + o0 + i]);
      xe[o0 + i] = acc;
    }
    cluster.sync();
    // true residual of the reduced system
    schur(xe);
    for (int e = tid; e < own; e += kClThreads) w[e] = bh[e] - w[e];
    __syncthreads();
    beta = sqrt(norm2_w(w));
    if (!isfinite(beta)) bad = 1;
  }
  cluster.sync();
  // x_e, then x_o = D_oo^-1 (b_o - D_oe x_e)
  blocks(1, xe, nullptr);
  for (int e = tid; e < own; e += kClThreads) {
    const int k = e / n, row = e % n;
    x[(long)site_of(0, k) * n + row] = xe[o0 + e];
    ac[e] = b[(long)site_of(1, k) * n + row] - ac[e];
  }
  __syncthreads();
  dinv(x, true);
  if (rank == 0 && tid == 0) {
    a.out[2 * rhs] = iters;
    a.out[2 * rhs + 1] = bad;
  }
  cluster.sync();  // no CTA leaves while another may read its partial sums
}

}  // namespace

bool coarse_cluster_fits(const OEGeom& oe, int restart, int nrhs, size_t real_bytes) {
  const int n = 2 * oe.nv, q = (oe.nhalf + kCl - 1) / kCl;
  // 17 of the 18 blocks of a site pair and the odd inverse, per step, through the cluster's SMs
  const long bytes = (long)oe.nhalf * 18 * n * n * 2 * (long)real_bytes;
  return restart <= kClMaxRestart && bytes <= kClMaxBytes && nrhs * kCl <= 152 &&
         cl_layout(restart, q, n, 2 * real_bytes).total <= 200 * 1024;
}

template <typename T>
void launch_coarse_gmres(const T* Dc, const T* Dinv, const T* b, T* x, T* V, T* u, T* xe, int* out, const OEGeom& oe,
                         double mu_c, double tol, int restart, int maxit, int nrhs, cudaStream_t st) {
  const int q = (oe.nhalf + kCl - 1) / kCl;
  const size_t smem = cl_layout(restart, q, 2 * oe.nv, 2 * sizeof(T)).total;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_coarse_gmres<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    attr = true;
  }
  ClArgs<T> a{Dc, Dinv, oe, b, x, V, u, xe, (T)mu_c, tol, restart, maxit, out};
  k_coarse_gmres<T><<<kCl * nrhs, kClThreads, smem, st>>>(a);
}
template void launch_coarse_gmres<double>(const double*, const double*, const double*, double*, double*, double*,
                                          double*, int*, const OEGeom&, double, double, int, int, int, cudaStream_t);
template void launch_coarse_gmres<float>(const float*, const float*, const float*, float*, float*, float*, float*,
                                         int*, const OEGeom&, double, double, int, int, int, cudaStream_t);

}  // namespace tmamg
