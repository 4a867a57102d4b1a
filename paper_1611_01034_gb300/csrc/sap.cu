// SAP smoother M of eq. (1): red/black multiplicative Schwarz with
// block-local minimal-residual solves (Sec. 1 of the paper: the smoother is
// the Schwarz Alternating Procedure and damps the UV modes).
//
// One launch processes every block of one colour.  One CTA owns one block,
// one thread one site.  The CTA
//   1. forms r = b - D x on its block with the full operator (neighbours in
//      the other colour are read from global memory; blocks of one colour are
//      never adjacent, so no CTA reads sites another CTA writes);
//   2. keeps r in shared memory and runs n_MR steps of
//        q = D_B r;  alpha = <q, r> / <q, q>;  e += alpha r;  r -= alpha q
//      with the Dirichlet block operator D_B (hops leaving the block are
//      dropped), the two inner products reduced by warp shuffles;
//   3. adds e to x.
// Block colour = parity of the sum of block coordinates; every dimension has
// an even number (>= 2) of blocks, so no block touches itself or a block of
// its own colour.
#include <algorithm>
#include <type_traits>

#include "tm_kernels.h"
#include "tm_lane.cuh"
#include "tm_stencil.cuh"

namespace tmamg {

template <typename T>
struct SapArgs {
  const T* gauge;
  const T* clover;
  const T* b;
  T* x;
  SapGeom sg;
  T mu;
  T bc;
  int n_mr;
  int colour;
  int nrhs;
  T rho;  // odd sites carry mu + rho
};

template <typename T, int MU>
__device__ __forceinline__ void block_hops(const cx<T>* __restrict__ rs, int BS, int l, const int lc[4],
                                           const int lst[4], const T* __restrict__ gauge, const Lat& g, int s,
                                           const int c[4], const int blk[4], cx<T> (&acc)[12]) {
  if (lc[MU] < blk[MU] - 1) {
    cx<T> p[12];
    const int ln = l + lst[MU];
#pragma unroll
    for (int k = 0; k < 12; ++k) p[k] = rs[k * BS + ln];
    hop_fwd_p<T, MU>(p, gauge, g.V, s, T(1), acc);
  }
  if (lc[MU] > 0) {
    cx<T> p[12];
    const int ln = l - lst[MU];
#pragma unroll
    for (int k = 0; k < 12; ++k) p[k] = rs[k * BS + ln];
    hop_bwd_p<T, MU>(p, gauge, g.V, nb_bwd(g, s, c, MU), T(1), acc);
  }
}

// FP32: two CTAs per SM (128 registers); FP64 would spill heavily at that bound.
// MT: most threads of a CTA, one per site; blocks of more than 256 sites (1024 at
// most) take the 64 registers that are left for them and spill the rest.
template <typename T, int MT>
__global__ void __launch_bounds__(MT, sizeof(T) == 4 && MT == 256 ? 2 : 1) k_sap(SapArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SapGeom& sg = a.sg;
  const Lat& g = sg.g;
  const int BS = sg.bsites;
  cx<T>* rs = reinterpret_cast<cx<T>*>(smem_raw);  // [12][BS]
  T* red = reinterpret_cast<T*>(rs + 12 * BS);     // [32 * 3]
  // consecutive CTAs take the same block for consecutive right-hand sides, so
  // the block's links and clover are read from DRAM once and then from L2
  const int rhs = blockIdx.x % a.nrhs;
  const long off = (long)rhs * NR_SPINOR * g.V;
  T* x = a.x + off;

  // the (blockIdx.x / nrhs)-th block of this colour
  int k = blockIdx.x / a.nrhs;
  const int nbxh = sg.nb[3] / 2;
  int bc4[4];
  const int bxh = k % nbxh;
  k /= nbxh;
  bc4[2] = k % sg.nb[2];
  k /= sg.nb[2];
  bc4[1] = k % sg.nb[1];
  bc4[0] = k / sg.nb[1];
  bc4[3] = 2 * bxh + ((bc4[0] + bc4[1] + bc4[2] + a.colour) & 1);

  const int l = threadIdx.x;
  const bool act = l < BS;
  int lc[4], c[4], lst[4];
  lst[3] = 1;
  lst[2] = sg.blk[3];
  lst[1] = sg.blk[3] * sg.blk[2];
  lst[0] = lst[1] * sg.blk[1];
  int s = 0;
  {
    int q = act ? l : 0;
    lc[3] = q % sg.blk[3];
    q /= sg.blk[3];
    lc[2] = q % sg.blk[2];
    q /= sg.blk[2];
    lc[1] = q % sg.blk[1];
    lc[0] = q / sg.blk[1];
#pragma unroll
    for (int d = 0; d < 4; ++d) c[d] = bc4[d] * sg.blk[d] + lc[d];
    s = ((c[0] * g.L[1] + c[1]) * g.L[2] + c[2]) * g.L[3] + c[3];
  }

  cx<T> r[12], e[12];
  const T half = T(0.5);
  const T mus = ((c[0] + c[1] + c[2] + c[3]) & 1) ? a.mu + a.rho : a.mu;
  if (act) {
    cx<T> acc[12], p[12];
    all_hops_global<T>(x, a.gauge, g, s, c, a.bc, acc);
    ld_cx<T, 12>(x, g.V, s, p);
    site_diag<T>(a.clover, g.V, s, mus, p, r);
#pragma unroll
    for (int i = 0; i < 12; ++i) r[i] = half * acc[i] - r[i];  // -D x
    if (a.b) {
      cx<T> bb[12];
      ld_cx<T, 12>(a.b + off, g.V, s, bb);
#pragma unroll
      for (int i = 0; i < 12; ++i) r[i] = r[i] + bb[i];
    }
#pragma unroll
    for (int i = 0; i < 12; ++i) rs[i * BS + l] = r[i];
  }
#pragma unroll
  for (int i = 0; i < 12; ++i) e[i] = cx<T>{0, 0};

  for (int it = 0; it < a.n_mr; ++it) {
    __syncthreads();
    cx<T> q[12];
    T dots[3] = {0, 0, 0};
    if (act) {
      cx<T> acc[12];
#pragma unroll
      for (int i = 0; i < 12; ++i) acc[i] = cx<T>{0, 0};
      block_hops<T, 0>(rs, BS, l, lc, lst, a.gauge, g, s, c, sg.blk, acc);
      block_hops<T, 1>(rs, BS, l, lc, lst, a.gauge, g, s, c, sg.blk, acc);
      block_hops<T, 2>(rs, BS, l, lc, lst, a.gauge, g, s, c, sg.blk, acc);
      block_hops<T, 3>(rs, BS, l, lc, lst, a.gauge, g, s, c, sg.blk, acc);
      site_diag<T>(a.clover, g.V, s, mus, r, q);
#pragma unroll
      for (int i = 0; i < 12; ++i) {
        q[i] = q[i] - half * acc[i];
        dots[0] = fma(q[i].r, r[i].r, fma(q[i].i, r[i].i, dots[0]));   // Re <q, r>
        dots[1] = fma(q[i].r, r[i].i, fma(-q[i].i, r[i].r, dots[1]));  // Im <q, r>
        dots[2] = fma(q[i].r, q[i].r, fma(q[i].i, q[i].i, dots[2]));   // <q, q>
      }
    }
    block_allreduce<T, 3>(dots, red);
    const cx<T> alpha = dots[2] > T(0) ? cx<T>{dots[0] / dots[2], dots[1] / dots[2]} : cx<T>{0, 0};
    if (act) {
#pragma unroll
      for (int i = 0; i < 12; ++i) {
        cfma(e[i], alpha, r[i]);
        cfma(r[i], -alpha, q[i]);
      }
    }
    __syncthreads();
    if (act) {
#pragma unroll
      for (int i = 0; i < 12; ++i) rs[i * BS + l] = r[i];
    }
  }
  __syncthreads();
  if (act) {
    cx<T> p[12];
    ld_cx<T, 12>(x, g.V, s, p);
#pragma unroll
    for (int i = 0; i < 12; ++i) p[i] = p[i] + e[i];
    st_cx<T, 12>(x, g.V, s, p);
  }
}

namespace {

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// sums of 3 values over the CTA; red holds 3 values per warp, read by the next call only after a barrier
template <class R>
__device__ __forceinline__ void lanes_allreduce3(R (&v)[3], R* red) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if constexpr (LaneOf<R>::n == 2)
        v[k] = v[k] + f2{__shfl_xor_sync(0xffffffffu, v[k].v, o)};
      else
        v[k] = v[k] + __shfl_xor_sync(0xffffffffu, v[k], o);
    }
  }
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int k = 0; k < 3; ++k) red[(threadIdx.x >> 5) * 3 + k] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    R s = red[k];
    for (int w = 1; w < (int)blockDim.x >> 5; ++w) s = s + red[w * 3 + k];
    v[k] = s;
  }
}

// <q, r> / <q, q> from the three sums, 0 where <q, q> is not positive
__device__ __forceinline__ float mr_ratio(float n, float d) { return d > 0.f ? n / d : 0.f; }
__device__ __forceinline__ double mr_ratio(double n, double d) { return d > 0.0 ? n / d : 0.0; }
__device__ __forceinline__ f2 mr_ratio(f2 n, f2 d) {
  const float2 a = f2_unpack(n), b = f2_unpack(d);
  return f2_pack(mr_ratio(a.x, b.x), mr_ratio(a.y, b.y));
}

}  // namespace

// The same for 4^4 blocks in FP32, with everything that the MR steps read on the
// chip: the block's links in shared memory (48 KB), the site's clover blocks and e,
// which only their own thread reads, in tensor memory (96 columns per warp), r in
// shared memory.  The general kernel reads links and clover from L1 and L2 in every
// step and waits for them: four sweeps, one right-hand side, 32 x 16^3, 342 -> 291
// us; 8^4 218 -> 169 us; three sweeps of 7 at 24^2 x 16^2 1.63 -> 1.37 ms.  Measured
// and left out: two right-hand sides per thread as packed lanes, as in the odd-even
// form (4 right-hand sides 878 -> 900 us: eight warps per SM wait longer); e alone
// moved to shared memory (320 us).
namespace {

// N words per thread to and from tensor memory (the loads wait; tmem_wait_st for the stores)
__device__ __forceinline__ void tmem_st8(unsigned ta, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(ta), "f"(v[0]), "f"(v[1]),
               "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_st4w(unsigned ta, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(ta), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3])
               : "memory");
}
__device__ __forceinline__ void tmem_ld8(unsigned ta, float* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "r"(ta)
               : "memory");
}
__device__ __forceinline__ void tmem_ld4w(unsigned ta, float* v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "r"(ta)
               : "memory");
}
// after this the loaded registers may be read: they pass through it
template <int N>
__device__ __forceinline__ void tmem_loaded(float (&v)[N]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < N; ++k) asm volatile("" : "+f"(v[k])::"memory");
}

constexpr int kS4 = 256;                 // sites of a block
constexpr unsigned kS4Cols = 256;        // tensor memory columns: (72 clover + 24 e) for two warps per quarter
constexpr size_t kS4Smem = 12 * kS4 * sizeof(float4) + 12 * kS4 * sizeof(cx<float>);

__global__ void __launch_bounds__(kS4, 2) k_sap4(SapArgs<float> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned tmem_base;
  __shared__ float red[8 * 3];
  float4* lk = reinterpret_cast<float4*>(smem_raw);                       // [mu][chunk][site]
  cx<float>* rs = reinterpret_cast<cx<float>*>(lk + 12 * kS4);            // [12][site]
  const SapGeom& sg = a.sg;
  const Lat& g = sg.g;
  const long V = g.V;
  const int l = threadIdx.x, warp = l >> 5;
  const long off = (long)(blockIdx.x % a.nrhs) * NR_SPINOR * V;  // right-hand sides fastest (operator reuse in L2)
  float* x = a.x + off;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(kS4Cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  int k = blockIdx.x / a.nrhs;
  const int nbxh = sg.nb[3] / 2;
  int bc4[4];
  const int bxh = k % nbxh;
  k /= nbxh;
  bc4[2] = k % sg.nb[2];
  k /= sg.nb[2];
  bc4[1] = k % sg.nb[1];
  bc4[0] = k / sg.nb[1];
  bc4[3] = 2 * bxh + ((bc4[0] + bc4[1] + bc4[2] + a.colour) & 1);
  const int lc[4] = {l >> 6, (l >> 4) & 3, (l >> 2) & 3, l & 3};
  constexpr int lst[4] = {64, 16, 4, 1};
  int c[4];
#pragma unroll
  for (int d = 0; d < 4; ++d) c[d] = 4 * bc4[d] + lc[d];
  const int s = ((c[0] * g.L[1] + c[1]) * g.L[2] + c[2]) * g.L[3] + c[3];
  const float mus = ((c[0] + c[1] + c[2] + c[3]) & 1) ? a.mu + a.rho : a.mu;
  auto rows = [&](const float4 (&v)[3], Link<float>& U) {
    const cx<float> z[6] = {{v[0].x, v[0].y}, {v[0].z, v[0].w}, {v[1].x, v[1].y},
                            {v[1].z, v[1].w}, {v[2].x, v[2].y}, {v[2].z, v[2].w}};
    link_from_rows(z, U);
  };
  auto scale = [&](Link<float>& U) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) U.u[i][j] = a.bc * U.u[i][j];
  };
  const float4* gl = reinterpret_cast<const float4*>(a.gauge);

  // r = b - D x: forward hops with the site's own links, which go to shared memory
  cx<float> acc[12];
#pragma unroll
  for (int i = 0; i < 12; ++i) acc[i] = cx<float>{0.f, 0.f};
  auto fwd = [&](auto MUC) {
    constexpr int MU = decltype(MUC)::value;
    cx<float> p[12];
    ld_cx<float, 12>(x, V, nb_fwd(g, s, c, MU), p);
    float4 v[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      v[q] = __ldg(gl + (MU * 3 + q) * V + s);
      lk[(MU * 3 + q) * kS4 + l] = v[q];
    }
    Link<float> U;
    rows(v, U);
    if (MU == 0 && c[0] == g.L[0] - 1) scale(U);
    hop_lanes<float, float, MU, true>([&](int i) { return p[i]; }, U, acc);
  };
  fwd(std::integral_constant<int, 0>{});
  fwd(std::integral_constant<int, 1>{});
  fwd(std::integral_constant<int, 2>{});
  fwd(std::integral_constant<int, 3>{});
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned ta = tmem_base + ((unsigned)(warp & 3) << 21) + (unsigned)(warp >> 2) * 96;  // clover, e at + 72
  auto bwd = [&](auto MUC) {
    constexpr int MU = decltype(MUC)::value;
    const int sb = nb_bwd(g, s, c, MU);
    cx<float> p[12];
    ld_cx<float, 12>(x, V, sb, p);
    float4 v[3];
#pragma unroll
    for (int q = 0; q < 3; ++q)
      v[q] = lc[MU] > 0 ? lk[(MU * 3 + q) * kS4 + l - lst[MU]] : __ldg(gl + (MU * 3 + q) * V + sb);
    Link<float> U;
    rows(v, U);
    if (MU == 0 && c[0] == 0) scale(U);
    hop_lanes<float, float, MU, false>([&](int i) { return p[i]; }, U, acc);
  };
  bwd(std::integral_constant<int, 0>{});
  bwd(std::integral_constant<int, 1>{});
  bwd(std::integral_constant<int, 2>{});
  bwd(std::integral_constant<int, 3>{});
  __syncwarp();  // the tensor-memory accesses are warp-wide
  {
    cx<float> p[12];
    ld_cx<float, 12>(x, V, s, p);
#pragma unroll
    for (int i = 0; i < 12; ++i) acc[i] = -0.5f * acc[i];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float m[36];
      ld_re<float, 36>(a.clover + (long)h * 36 * V, V, s, m);
#pragma unroll
      for (int q = 0; q < 4; ++q) tmem_st8(ta + 36 * h + 8 * q, m + 8 * q);
      tmem_st4w(ta + 36 * h + 32, m + 32);
      herm6_lanes<float, float>(m, h == 0 ? -mus : mus, p + 6 * h, acc + 6 * h);
    }
    const float z[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 3; ++q) tmem_st8(ta + 72 + 8 * q, z);
    if (a.b) {
      ld_cx<float, 12>(a.b + off, V, s, p);
#pragma unroll
      for (int i = 0; i < 12; ++i) acc[i] = p[i] - acc[i];
    } else {
#pragma unroll
      for (int i = 0; i < 12; ++i) acc[i] = -acc[i];
    }
#pragma unroll
    for (int i = 0; i < 12; ++i) rs[i * kS4 + l] = acc[i];
    tmem_wait_st();
  }
#pragma unroll 1
  for (int it = 0; it < a.n_mr; ++it) {
    __syncthreads();
    cx<float> q[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) q[i] = cx<float>{0.f, 0.f};
    auto hop = [&](auto MUC) {
      constexpr int MU = decltype(MUC)::value;
      if (lc[MU] < 3) {
        const cx<float>* sp = rs + l + lst[MU];
        const float4 v[3] = {lk[(MU * 3) * kS4 + l], lk[(MU * 3 + 1) * kS4 + l], lk[(MU * 3 + 2) * kS4 + l]};
        Link<float> U;
        rows(v, U);
        hop_lanes<float, float, MU, true>([&](int i) { return sp[i * kS4]; }, U, q);
      }
      if (lc[MU] > 0) {
        const int ln = l - lst[MU];
        const cx<float>* sp = rs + ln;
        const float4 v[3] = {lk[(MU * 3) * kS4 + ln], lk[(MU * 3 + 1) * kS4 + ln], lk[(MU * 3 + 2) * kS4 + ln]};
        Link<float> U;
        rows(v, U);
        hop_lanes<float, float, MU, false>([&](int i) { return sp[i * kS4]; }, U, q);
      }
    };
    hop(std::integral_constant<int, 0>{});
    hop(std::integral_constant<int, 1>{});
    hop(std::integral_constant<int, 2>{});
    hop(std::integral_constant<int, 3>{});
    __syncwarp();
    cx<float> r[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      r[i] = rs[i * kS4 + l];
      q[i] = -0.5f * q[i];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float m[36];
#pragma unroll
      for (int w = 0; w < 4; ++w) tmem_ld8(ta + 36 * h + 8 * w, m + 8 * w);
      tmem_ld4w(ta + 36 * h + 32, m + 32);
      tmem_loaded(m);
      herm6_lanes<float, float>(m, h == 0 ? -mus : mus, r + 6 * h, q + 6 * h);
    }
    float dots[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      dots[0] = fmaf(q[i].r, r[i].r, fmaf(q[i].i, r[i].i, dots[0]));   // Re <q, r>
      dots[1] = fmaf(q[i].r, r[i].i, fmaf(-q[i].i, r[i].r, dots[1]));  // Im <q, r>
      dots[2] = fmaf(q[i].r, q[i].r, fmaf(q[i].i, q[i].i, dots[2]));   // <q, q>
    }
    lanes_allreduce3<float>(dots, red);  // its barrier: every neighbour's r has been read
    const cx<float> al{mr_ratio(dots[0], dots[2]), mr_ratio(dots[1], dots[2])};
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      float e[8];
      tmem_ld8(ta + 72 + 8 * w, e);
      tmem_loaded(e);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        cx<float> z{e[2 * i], e[2 * i + 1]};
        cfma(z, al, r[4 * w + i]);
        e[2 * i] = z.r;
        e[2 * i + 1] = z.i;
      }
      tmem_st8(ta + 72 + 8 * w, e);
    }
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      cfma(r[i], -al, q[i]);
      rs[i * kS4 + l] = r[i];
    }
    tmem_wait_st();
  }
  {
    cx<float> p[12];
    ld_cx<float, 12>(x, V, s, p);
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      float e[8];
      tmem_ld8(ta + 72 + 8 * w, e);
      tmem_loaded(e);
#pragma unroll
      for (int i = 0; i < 4; ++i) p[4 * w + i] = p[4 * w + i] + cx<float>{e[2 * i], e[2 * i + 1]};
    }
    st_cx<float, 12>(x, V, s, p);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kS4Cols) : "memory");
}

}  // namespace

template <typename T>
void launch_sap_colour(const T* gauge, const T* clover, const T* b, T* x, const SapGeom& sg, double mu,
                       double bc_t, int n_mr, int colour, int nrhs, cudaStream_t st, double rho) {
  const int threads = (sg.bsites + 31) / 32 * 32;
  const size_t smem = 12 * sg.bsites * sizeof(cx<T>) + 32 * 3 * sizeof(T);
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(k_sap<T, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(k_sap<T, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    attr_set = true;
  }
  const int nblk_colour = sg.nb[0] * sg.nb[1] * sg.nb[2] * sg.nb[3] / 2;
  SapArgs<T> a{gauge, clover, b, x, sg, (T)mu, (T)bc_t, n_mr, colour, nrhs, (T)rho};
  if constexpr (std::is_same<T, float>::value) {
    bool b4 = true;
    for (int d = 0; d < 4; ++d) b4 = b4 && sg.blk[d] == 4;
    if (b4) {
      static bool attr4 = false;
      if (!attr4) {
        cudaFuncSetAttribute(k_sap4, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kS4Smem);
        attr4 = true;
      }
      k_sap4<<<nblk_colour * nrhs, kS4, kS4Smem, st>>>(a);
      return;
    }
  }
  dim3 grid(nblk_colour * nrhs);
  if (threads <= 256)
    k_sap<T, 256><<<grid, threads, smem, st>>>(a);
  else
    k_sap<T, 1024><<<grid, threads, smem, st>>>(a);
}

template void launch_sap_colour<double>(const double*, const double*, const double*, double*, const SapGeom&,
                                        double, double, int, int, int, cudaStream_t, double);
template void launch_sap_colour<float>(const float*, const float*, const float*, float*, const SapGeom&, double,
                                       double, int, int, int, cudaStream_t, double);

// ===========================================================================
// Odd-even block solve (Sec. 3: odd-even preconditioning is used in the
// smoother).  Within a block B (all dims even, origin on an even site, so the
// site parity (t+z+y+x) mod 2 splits it into two halves of BS/2 sites),
//   D_B = [[D_ee, D_eo], [D_oe, D_oo]],
// D_ee, D_oo the site-diagonal A(x) + i mu gamma5, D_eo, D_oe the Dirichlet
// intra-block hops.  The MR steps run on the Schur complement
//   S = D_ee - D_eo D_oo^-1 D_oe  over the even sites,
// with right-hand side r_e - D_eo D_oo^-1 r_o; afterwards
//   e_o = D_oo^-1 (r_o - D_oe e_e).
// D_oo^-1 comes precomputed per odd site (launch_clover_inverse).
//
// One CTA owns one block and one lane type R of right-hand sides (two at once
// as packed FP32, or one); thread j owns the j-th even and the j-th odd site
// (same t, z, y; x = 2 j_x + parity offset), so no lane idles in either
// half-step.  The kernel waits on operator loads (L1 and L2) and issue, not on
// DRAM: two right-hand sides per thread share every operator load, conversion
// and link row and halve the instructions (823 M -> 497 M warp instructions
// per 6-rhs launch at 48 x 24^3).  Their 255 registers leave two CTAs per SM;
// a bound of 168 registers (three CTAs) spills and its shared memory takes the
// L1 from the operator: 1.96 ms against 1.11 ms per launch (one right-hand
// side per thread: 1.24 ms; lattice-ordered operator before: 1.50 ms).
//
// The kernel walks 2 n_MR + 3 half-steps, odd and even alternating, so that the
// hop gather, D_oo^-1 and the site-diagonal term each appear once in the code
// (the instruction cache holds the loop); H = the sum of the intra-block hops,
// D_eo, D_oe = -H/2:
//   step 0 (odd):            od = D_oo^-1 r_o; x_o += od
//   step 1 (even):           rho = r_e + H od / 2
//   step 2k (odd, k >= 1):   od = D_oo^-1 H rho
//   step 2k+1 (even):        q = D_ee rho - H od / 4; MR update of e_e, rho
//   step 2 n_MR + 2 (odd):   x_o += D_oo^-1 H e_e / 2; x_e += e_e
// ===========================================================================
namespace {

// index of a site within its parity class, from block-local coordinates
__device__ __forceinline__ int half_index(const int lc[4], const int blk[4]) {
  return ((lc[0] * blk[1] + lc[1]) * blk[2] + lc[2]) * (blk[3] / 2) + (lc[3] >> 1);
}
// linear index of a block from its block coordinates
__device__ __forceinline__ int block_linear(const SapGeom& sg, const int bc[4]) {
  return ((bc[0] * sg.nb[1] + bc[1]) * sg.nb[2] + bc[2]) * sg.nb[3] + bc[3];
}

template <typename T, int NC, int S>
__device__ __forceinline__ void ld_op(const void* __restrict__ base, long off, long V, long s, cx<T> (&z)[NC]) {
  if constexpr (S == ST_NATIVE)
    ld_cx<T, NC>(static_cast<const T*>(base) + off, V, s, z);
  else
    ld_cx16<T, S, NC>(static_cast<const unsigned short*>(base) + off, V, s, z);
}

}  // namespace

template <typename T>
struct SapOeArgs {
  // links, clover and D_oo^-1 as T in lattice order, or in 16 bits in block
  // order (kernel parameter S): site index block * BS + parity * HB + half_index
  const void* gauge;
  const void* clover;
  const void* dinv;
  const T* b;
  T* x;
  SapGeom sg;
  T mu;
  T bc;
  int n_mr;
  int colour;
  int nrhs;
  T rho;  // odd sites carry mu + rho (D_oo^-1 is built with it)
};

// MT: most threads of a CTA, one per even site.  Blocks of more than 256 sites
// (1024 at most) run one right-hand side at a time and keep e_e, which only its
// own thread reads, out of shared memory, which the two fields that the hops
// gather fill.
template <class R, int S, int MT>
__global__ void __launch_bounds__(MT, MT > 128 ? 1 : sizeof(R) == 4 ? 3 : 2)
    k_sap_oe(SapOeArgs<typename LaneOf<R>::T> a) {
  using T = typename LaneOf<R>::T;
  constexpr bool BLOCKED = S != ST_NATIVE;  // operator in block order
  constexpr bool E_OWN = MT > 128;          // e_e in the thread's own storage
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SapGeom& sg = a.sg;
  const Lat& g = sg.g;
  const int HB = sg.bsites / 2;
  cx<R>* ev = reinterpret_cast<cx<R>*>(smem_raw);  // [12][HB] even-site values (rho, then e_e)
  cx<R>* od = ev + 12 * HB;                         // [12][HB] odd-site values
  cx<R>* ee = od + 12 * HB;                         // [12][HB] e_e
  R* red = reinterpret_cast<R*>(E_OWN ? ee : ee + 12 * HB);  // 3 per warp
  cx<R> e_own[E_OWN ? 12 : 1];
  const int groups = a.nrhs / LaneOf<R>::n;  // right-hand sides fastest over the CTAs (operator reuse in L2)
  const long fs = (long)NR_SPINOR * g.V;
  const long r0 = (long)(blockIdx.x % groups) * LaneOf<R>::n * fs;
  T* x0 = a.x + r0;
  T* x1 = x0 + fs;  // second lane
  const T* b0 = a.b ? a.b + r0 : nullptr;
  const T* b1 = b0 + fs;
  const long Vh = g.V / 2;

  int k = blockIdx.x / groups;
  const int nbxh = sg.nb[3] / 2;
  int bc4[4];
  const int bxh = k % nbxh;
  k /= nbxh;
  bc4[2] = k % sg.nb[2];
  k /= sg.nb[2];
  bc4[1] = k % sg.nb[1];
  bc4[0] = k / sg.nb[1];
  bc4[3] = 2 * bxh + ((bc4[0] + bc4[1] + bc4[2] + a.colour) & 1);
  const int bl = block_linear(sg, bc4);

  const int j = threadIdx.x;
  const bool act = j < HB;
  // block-local coordinates of the j-th even site; the j-th odd site differs in x only
  int lce[4];
  int pr;
  {
    int q = act ? j : 0;
    const int bxh2 = sg.blk[3] / 2;
    const int xh = q % bxh2;
    q /= bxh2;
    lce[2] = q % sg.blk[2];
    q /= sg.blk[2];
    lce[1] = q % sg.blk[1];
    lce[0] = q / sg.blk[1];
    pr = (lce[0] + lce[1] + lce[2]) & 1;
    lce[3] = 2 * xh + pr;
  }
  auto site_of = [&](int parity, int (&lc)[4], int (&c)[4]) {
    lc[0] = lce[0];
    lc[1] = lce[1];
    lc[2] = lce[2];
    lc[3] = lce[3] - pr + (pr ^ parity);
#pragma unroll
    for (int d = 0; d < 4; ++d) c[d] = bc4[d] * sg.blk[d] + lc[d];
    return ((c[0] * g.L[1] + c[1]) * g.L[2] + c[2]) * g.L[3] + c[3];
  };
  // operator index of the j-th site of the given parity
  auto own_op = [&](int parity, int s) { return BLOCKED ? bl * sg.bsites + parity * HB + j : s; };
  auto link = [&](int mu, long so, Link<T>& U) {
    cx<T> z[6];
    ld_op<T, 6, S>(a.gauge, (long)mu * NR_LINK * g.V, g.V, so, z);
    link_from_rows(z, U);
  };
  // y += (A + i m gamma5) p
  auto diag = [&](long so, T m, const cx<R> (&p)[12], cx<R> (&y)[12]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      T mm[36];
      ld_re_s<T, S, 36>(BLOCKED ? static_cast<const void*>(static_cast<const unsigned short*>(a.clover) + (long)h * 36 * g.V)
                                : static_cast<const void*>(static_cast<const T*>(a.clover) + (long)h * 36 * g.V),
                        g.V, so, mm);
      herm6_lanes<R, T>(mm, h == 0 ? -m : m, p + 6 * h, y + 6 * h);
    }
  };

  // r = b - D x on the odd (pass 0, -> od) and the even site (pass 1, -> ev)
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    if (act) {
      const int par = pass ^ 1;
      int lc[4], c[4];
      const int s = site_of(par, lc, c);
      const int so = own_op(par, s);
      cx<R> acc[12];
#pragma unroll
      for (int i = 0; i < 12; ++i) acc[i] = czero<R>();
      auto hops = [&](auto MUC) {
        constexpr int MU = decltype(MUC)::value;
        {
          cx<R> p[12];
          ld_lanes<R, 12, T>(x0, x1, g.V, nb_fwd(g, s, c, MU), p);
          Link<T> U;
          link(MU, so, U);
          if (MU == 0 && c[0] == g.L[0] - 1) {
#pragma unroll
            for (int i = 0; i < 12; ++i) p[i] = cx<R>{bcast<R>(a.bc) * p[i].r, bcast<R>(a.bc) * p[i].i};
          }
          hop_lanes<R, T, MU, true>([&](int i) { return p[i]; }, U, acc);
        }
        {
          cx<R> p[12];
          const int sb = nb_bwd(g, s, c, MU);
          ld_lanes<R, 12, T>(x0, x1, g.V, sb, p);
          int ob = sb;
          if (BLOCKED) {  // the link belongs to the neighbour, in this block or the one before it
            int ln[4] = {lc[0], lc[1], lc[2], lc[3]}, bn[4] = {bc4[0], bc4[1], bc4[2], bc4[3]};
            if (lc[MU] > 0) {
              ln[MU] = lc[MU] - 1;
            } else {
              ln[MU] = sg.blk[MU] - 1;
              bn[MU] = bn[MU] > 0 ? bn[MU] - 1 : sg.nb[MU] - 1;
            }
            ob = block_linear(sg, bn) * sg.bsites + (par ^ 1) * HB + half_index(ln, sg.blk);
          }
          Link<T> U;
          link(MU, ob, U);
          if (MU == 0 && c[0] == 0) {
#pragma unroll
            for (int i = 0; i < 12; ++i) p[i] = cx<R>{bcast<R>(a.bc) * p[i].r, bcast<R>(a.bc) * p[i].i};
          }
          hop_lanes<R, T, MU, false>([&](int i) { return p[i]; }, U, acc);
        }
      };
      hops(std::integral_constant<int, 0>{});
      hops(std::integral_constant<int, 1>{});
      hops(std::integral_constant<int, 2>{});
      hops(std::integral_constant<int, 3>{});
      // acc = -H x / 2 + A x, then b - acc
#pragma unroll
      for (int i = 0; i < 12; ++i) acc[i] = cx<R>{bcast<R>(T(-0.5)) * acc[i].r, bcast<R>(T(-0.5)) * acc[i].i};
      cx<R> p[12];
      ld_lanes<R, 12, T>(x0, x1, g.V, s, p);
      diag(so, par ? a.mu + a.rho : a.mu, p, acc);
      if (b0) {
        ld_lanes<R, 12, T>(b0, b1, g.V, s, p);
#pragma unroll
        for (int i = 0; i < 12; ++i) acc[i] = p[i] - acc[i];
      } else {
#pragma unroll
        for (int i = 0; i < 12; ++i) acc[i] = czero<R>() - acc[i];
      }
      cx<R>* to = par ? od : ev;
#pragma unroll
      for (int i = 0; i < 12; ++i) st_shared(to + i * HB + j, acc[i]);
    }
  }

  const int nsteps = 2 * a.n_mr + 3;
#pragma unroll 1
  for (int st = 0; st < nsteps; ++st) {
    const int parity = (st & 1) ^ 1;  // even steps work on odd sites
    __syncthreads();
    cx<R> acc[12];
    int lc[4], c[4];
    const int s = site_of(parity, lc, c);
    const int so = own_op(parity, s);
    if (act && st > 0) {
      const cx<R>* src = parity ? ev : od;
#pragma unroll
      for (int i = 0; i < 12; ++i) acc[i] = czero<R>();
      auto hops = [&](auto MUC) {
        constexpr int MU = decltype(MUC)::value;
        if (lc[MU] < sg.blk[MU] - 1) {
          int ln[4] = {lc[0], lc[1], lc[2], lc[3]};
          ln[MU] += 1;
          const cx<R>* sp = src + half_index(ln, sg.blk);
          Link<T> U;
          link(MU, so, U);
          hop_lanes<R, T, MU, true>([&](int i) { return ld_shared(sp + i * HB); }, U, acc);
        }
        if (lc[MU] > 0) {
          int ln[4] = {lc[0], lc[1], lc[2], lc[3]};
          ln[MU] -= 1;
          const int jn = half_index(ln, sg.blk);
          const cx<R>* sp = src + jn;
          Link<T> U;
          link(MU, BLOCKED ? bl * sg.bsites + (parity ^ 1) * HB + jn : nb_bwd(g, s, c, MU), U);
          hop_lanes<R, T, MU, false>([&](int i) { return ld_shared(sp + i * HB); }, U, acc);
        }
      };
      hops(std::integral_constant<int, 0>{});
      hops(std::integral_constant<int, 1>{});
      hops(std::integral_constant<int, 2>{});
      hops(std::integral_constant<int, 3>{});
    }
    if (parity) {
      // odd site: D_oo^-1 of r_o (step 0) or of the hops
      if (act) {
        const bool last = st == nsteps - 1;
        if (st == 0) {
#pragma unroll
          for (int i = 0; i < 12; ++i) acc[i] = ld_shared(od + i * HB + j);
        }
        cx<R> y[12];
        const long di = BLOCKED ? bl * HB + j : s >> 1;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int i = 0; i < 6; ++i) {
            cx<T> m[6];
            ld_op<T, 6, S>(a.dinv, (long)(h * 6 + i) * 12 * Vh, Vh, di, m);  // row i of block h
            y[6 * h + i] = lcmul(m[0], acc[6 * h]);
#pragma unroll
            for (int q = 1; q < 6; ++q) lcfma(y[6 * h + i], m[q], acc[6 * h + q]);
          }
        if (!last) {
#pragma unroll
          for (int i = 0; i < 12; ++i) st_shared(od + i * HB + j, y[i]);
        }
        if (st == 0 || last) {
          // every residual of the block has been formed from the old x (barrier above)
          const R w = bcast<R>(st == 0 ? T(1) : T(0.5));
          cx<R> p[12];
          ld_lanes_rw<R, 12, T>(x0, x1, g.V, s, p);
#pragma unroll
          for (int i = 0; i < 12; ++i) p[i] = cx<R>{lfma(w, y[i].r, p[i].r), lfma(w, y[i].i, p[i].i)};
          st_lanes<R, 12, T>(x0, x1, g.V, s, p);
        }
        if (last) {
          int lc2[4], c2[4];
          const int s2 = site_of(0, lc2, c2);
          cx<R> p[12];
          ld_lanes_rw<R, 12, T>(x0, x1, g.V, s2, p);
#pragma unroll
          for (int i = 0; i < 12; ++i) p[i] = p[i] + ld_shared(ev + i * HB + j);
          st_lanes<R, 12, T>(x0, x1, g.V, s2, p);
        }
      }
    } else {
      const bool store_e = (st - 1) / 2 == a.n_mr;  // the next odd step gathers e_e
      cx<R> rho[12];
      if (act) {
#pragma unroll
        for (int i = 0; i < 12; ++i) rho[i] = ld_shared(ev + i * HB + j);
      }
      if (st == 1) {
        if (act) {
          const R hf = bcast<R>(T(0.5));
#pragma unroll
          for (int i = 0; i < 12; ++i) {
            rho[i] = cx<R>{lfma(hf, acc[i].r, rho[i].r), lfma(hf, acc[i].i, rho[i].i)};
            if constexpr (E_OWN)
              e_own[i] = czero<R>();
            else
              st_shared(ee + i * HB + j, czero<R>());
            st_shared(ev + i * HB + j, store_e ? czero<R>() : rho[i]);
          }
        }
      } else {
        R dots[3] = {bcast<R>(T(0)), bcast<R>(T(0)), bcast<R>(T(0))};
        if (act) {
          const R mq = bcast<R>(T(-0.25));
#pragma unroll
          for (int i = 0; i < 12; ++i) acc[i] = cx<R>{mq * acc[i].r, mq * acc[i].i};
          diag(so, a.mu, rho, acc);  // acc = q
          R d1 = bcast<R>(T(0));
#pragma unroll
          for (int i = 0; i < 12; ++i) {
            dots[0] = lfma(acc[i].r, rho[i].r, lfma(acc[i].i, rho[i].i, dots[0]));  // Re <q, rho>
            dots[1] = lfma(acc[i].r, rho[i].i, dots[1]);                           // Im <q, rho> = the difference
            d1 = lfma(acc[i].i, rho[i].r, d1);
            dots[2] = lfma(acc[i].r, acc[i].r, lfma(acc[i].i, acc[i].i, dots[2]));  // <q, q>
          }
          dots[1] = dots[1] - d1;
        }
        lanes_allreduce3<R>(dots, red);
        if (act) {
          const R ar = mr_ratio(dots[0], dots[2]), ai = mr_ratio(dots[1], dots[2]);
          const R nr = bcast<R>(T(0)) - ar, ni = bcast<R>(T(0)) - ai;
#pragma unroll
          for (int i = 0; i < 12; ++i) {
            cx<R> e;
            if constexpr (E_OWN)
              e = e_own[i];
            else
              e = ld_shared(ee + i * HB + j);
            e.r = lfma(ni, rho[i].i, lfma(ar, rho[i].r, e.r));
            e.i = lfma(ai, rho[i].r, lfma(ar, rho[i].i, e.i));
            if constexpr (E_OWN)
              e_own[i] = e;
            else if (!store_e)
              st_shared(ee + i * HB + j, e);
            cx<R> q = rho[i];  // rho - alpha q
            q.r = lfma(ai, acc[i].i, lfma(nr, acc[i].r, q.r));
            q.i = lfma(ni, acc[i].r, lfma(nr, acc[i].i, q.i));
            st_shared(ev + i * HB + j, store_e ? e : q);
          }
        }
      }
    }
  }
}

template <class R, int S, int MT>
void sap_oe_t(const SapOeArgs<typename LaneOf<R>::T>& a, int nblocks, cudaStream_t st) {
  const int HB = a.sg.bsites / 2;
  const int threads = (HB + 31) / 32 * 32;
  const size_t smem = (MT > 128 ? 24 : 36) * (size_t)HB * sizeof(cx<R>) + (threads / 32) * 3 * sizeof(R);
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(k_sap_oe<R, S, MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    attr_set = true;
  }
  k_sap_oe<R, S, MT><<<dim3(nblocks * (a.nrhs / LaneOf<R>::n)), threads, smem, st>>>(a);
}
template <class R, int S>
void sap_oe_s(const SapOeArgs<typename LaneOf<R>::T>& a, int nblocks, cudaStream_t st) {
  if constexpr (LaneOf<R>::n == 1) {
    if (a.sg.bsites > 256) return sap_oe_t<R, S, 512>(a, nblocks, st);
  }
  sap_oe_t<R, S, 128>(a, nblocks, st);
}

// ===========================================================================
// The same block solve for 4^4 blocks, a 16-bit operator and pairs of
// right-hand sides.  k_sap_oe holds 74 KB of shared memory per CTA for such a
// pair and needs 255 registers, so two CTAs share an SM.  Here the sums e_e and
// e_o, which only their own thread reads, live in tensor memory (96 of 128
// allocated columns), shared memory holds just the two fields that the hops
// gather (48 KB), and with the block's shape known at compile time 168
// registers suffice: three CTAs, 12 warps per SM (6-rhs launch at 48 x 24^3:
// 1.11 -> 1.02 ms).  Measured and left out: the block's operator (78 KB) staged
// in shared memory for two or three pairs of one larger CTA (1.25 and 1.61 ms:
// its warps wait in the same phases), four CTAs per SM (128 registers, 1.63 ms).
//
// e_o needs no half-step of its own: with z_k = D_oo^-1 H rho_k, which every MR
// step forms anyway, D_oo^-1 H e_e = sum_k alpha_k z_k, so the last odd half-step
// of k_sap_oe becomes one more running sum:
//   step 0 (odd):           od = D_oo^-1 r_o; e_o = 2 od
//   step 1 (even):          rho = r_e + H od / 2
//   step 2k (odd, k >= 1):  od = z = D_oo^-1 H rho
//   step 2k+1 (even):       q = D_ee rho - H od / 4; e_e += alpha rho, e_o += alpha z,
//                           rho -= alpha q
//   then x_e += e_e, x_o += e_o / 2.
// ===========================================================================
namespace {

constexpr int kB4 = 256, kH4 = 128;           // sites of a 4^4 block, of one parity
constexpr unsigned kTmemCols = 128;  // e_e at column 0, e_o at 48

// four complex pairs (16 words per thread) to and from tensor memory; the caller waits
__device__ __forceinline__ void tmem_st4(unsigned ta, const cx<f2>* z) {
  float2 v[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[2 * k] = f2_unpack(z[k].r);
    v[2 * k + 1] = f2_unpack(z[k].i);
  }
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(ta),
      "f"(v[0].x), "f"(v[0].y), "f"(v[1].x), "f"(v[1].y), "f"(v[2].x), "f"(v[2].y), "f"(v[3].x), "f"(v[3].y),
      "f"(v[4].x), "f"(v[4].y), "f"(v[5].x), "f"(v[5].y), "f"(v[6].x), "f"(v[6].y), "f"(v[7].x), "f"(v[7].y)
      : "memory");
}
__device__ __forceinline__ void tmem_ld4(unsigned ta, cx<f2>* z) {
  float v[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
      : "r"(ta)
      : "memory");
#pragma unroll
  for (int k = 0; k < 4; ++k) z[k] = cx<f2>{f2_pack(v[4 * k], v[4 * k + 1]), f2_pack(v[4 * k + 2], v[4 * k + 3])};
}

// two complex numbers of a 16-bit chunk
template <int S>
__device__ __forceinline__ void unpack_chunk(uint2 v, cx<float>& a, cx<float>& b) {
  const float2 p = unpack16x2<S>(v.x), q = unpack16x2<S>(v.y);
  a = cx<float>{p.x, p.y};
  b = cx<float>{q.x, q.y};
}

template <int S>
__global__ void __launch_bounds__(kH4, 3) k_sap_oe4(SapOeArgs<float> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned tmem_base;
  __shared__ f2 red[4 * 3];
  const SapGeom& sg = a.sg;
  const Lat& g = sg.g;
  const int pairs = a.nrhs / 2;
  const int j = threadIdx.x, warp = j >> 5;
  const long V = g.V, Vh = g.V / 2;

  int bc4[4];
  {
    int k = blockIdx.x / pairs;  // pairs fastest over the CTAs (operator reuse in L2)
    const int nbxh = sg.nb[3] / 2;
    const int bxh = k % nbxh;
    k /= nbxh;
    bc4[2] = k % sg.nb[2];
    k /= sg.nb[2];
    bc4[1] = k % sg.nb[1];
    bc4[0] = k / sg.nb[1];
    bc4[3] = 2 * bxh + ((bc4[0] + bc4[1] + bc4[2] + a.colour) & 1);
  }
  const int bl = block_linear(sg, bc4);
  const uint2* gauge = static_cast<const uint2*>(a.gauge);
  const uint2* clover = static_cast<const uint2*>(a.clover);
  const uint2* dinv = static_cast<const uint2*>(a.dinv);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned ta = tmem_base + ((unsigned)warp << 21);  // a warp reaches its own 32 lanes
  {
    const int grp = blockIdx.x % pairs;
    cx<f2>* ev = reinterpret_cast<cx<f2>*>(smem_raw);  // [12][128] rho
    cx<f2>* od = ev + 12 * kH4;                         // [12][128] u_o and z
    const long fs = (long)NR_SPINOR * V;
    float* x0 = a.x + 2 * grp * fs;
    float* x1 = x0 + fs;
    const float* b0 = a.b ? a.b + 2 * grp * fs : nullptr;
    const float* b1 = a.b ? b0 + fs : nullptr;
    // j = ((t 4 + z) 4 + y) 2 + (x >> 1)
    const int lt = j >> 5, lz = (j >> 3) & 3, ly = (j >> 1) & 3, xh = j & 1;
    const int pr = (lt + lz + ly) & 1;  // x parity of the even site
    const uint2* olink = gauge + (long)bl * kB4;
    const uint2* oclov = clover + (long)bl * kB4;
    const uint2* odinv = dinv + (long)bl * kH4 + j;
    auto link = [&](int mu, int w, Link<float>& U) {  // site w of the block in block order
      cx<float> z[6];
#pragma unroll
      for (int k = 0; k < 3; ++k) unpack_chunk<S>(__ldg(olink + (mu * 3 + k) * V + w), z[2 * k], z[2 * k + 1]);
      link_from_rows(z, U);
    };
    // y += (A + i m gamma5) p, the clover chunk k of the site from ld(k)
    auto diag = [&](auto ld, float m, const cx<f2>(&p)[12], cx<f2>(&y)[12]) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float mm[36];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          cx<float> u, v;
          unpack_chunk<S>(ld(9 * h + k), u, v);
          mm[4 * k] = u.r;
          mm[4 * k + 1] = u.i;
          mm[4 * k + 2] = v.r;
          mm[4 * k + 3] = v.i;
        }
        herm6_lanes<f2, float>(mm, h == 0 ? -m : m, p + 6 * h, y + 6 * h);
      }
    };
    auto site = [&](int par, int (&c)[4]) {
      c[0] = 4 * bc4[0] + lt;
      c[1] = 4 * bc4[1] + lz;
      c[2] = 4 * bc4[2] + ly;
      c[3] = 4 * bc4[3] + 2 * xh + (pr ^ par);
      return ((c[0] * g.L[1] + c[1]) * g.L[2] + c[2]) * g.L[3] + c[3];
    };

    // r = b - D x on the odd (pass 0, -> od) and the even site (pass 1, -> ev)
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      const int par = pass ^ 1;
      int c[4];
      const int s = site(par, c);
      const int lx = 2 * xh + (pr ^ par), own = par * kH4 + j;
      cx<f2> acc[12];
#pragma unroll
      for (int i = 0; i < 12; ++i) acc[i] = czero<f2>();
      auto hops = [&](auto MUC) {
        constexpr int MU = decltype(MUC)::value;
        const int lm = MU == 0 ? lt : MU == 1 ? lz : MU == 2 ? ly : lx;
        const int js = MU == 0 ? 32 : MU == 1 ? 8 : 2;
        {
          cx<f2> p[12];
          ld_lanes<f2, 12, float>(x0, x1, V, nb_fwd(g, s, c, MU), p);
          Link<float> U;
          link(MU, own, U);
          if (MU == 0 && c[0] == g.L[0] - 1) {
#pragma unroll
            for (int i = 0; i < 12; ++i) p[i] = cx<f2>{bcast<f2>(a.bc) * p[i].r, bcast<f2>(a.bc) * p[i].i};
          }
          hop_lanes<f2, float, MU, true>([&](int i) { return p[i]; }, U, acc);
        }
        {
          cx<f2> p[12];
          ld_lanes<f2, 12, float>(x0, x1, V, nb_bwd(g, s, c, MU), p);
          cx<float> z[6];
          if (lm > 0) {
            const int jn = MU < 3 ? j - js : (j & ~1) + ((lx - 1) >> 1);
#pragma unroll
            for (int k = 0; k < 3; ++k)
              unpack_chunk<S>(__ldg(olink + (MU * 3 + k) * V + (par ^ 1) * kH4 + jn), z[2 * k], z[2 * k + 1]);
          } else {  // the link belongs to the block before this one
            int bn[4] = {bc4[0], bc4[1], bc4[2], bc4[3]};
            bn[MU] = bn[MU] > 0 ? bn[MU] - 1 : sg.nb[MU] - 1;
            const int jn = MU < 3 ? j + 3 * js : (j & ~1) + 1;
            const uint2* src = gauge + (long)block_linear(sg, bn) * kB4 + (par ^ 1) * kH4 + jn;
#pragma unroll
            for (int k = 0; k < 3; ++k) unpack_chunk<S>(__ldg(src + (MU * 3 + k) * V), z[2 * k], z[2 * k + 1]);
          }
          Link<float> U;
          link_from_rows(z, U);
          if (MU == 0 && c[0] == 0) {
#pragma unroll
            for (int i = 0; i < 12; ++i) p[i] = cx<f2>{bcast<f2>(a.bc) * p[i].r, bcast<f2>(a.bc) * p[i].i};
          }
          hop_lanes<f2, float, MU, false>([&](int i) { return p[i]; }, U, acc);
        }
      };
      hops(std::integral_constant<int, 0>{});
      hops(std::integral_constant<int, 1>{});
      hops(std::integral_constant<int, 2>{});
      hops(std::integral_constant<int, 3>{});
#pragma unroll
      for (int i = 0; i < 12; ++i) acc[i] = cx<f2>{bcast<f2>(-0.5f) * acc[i].r, bcast<f2>(-0.5f) * acc[i].i};
      cx<f2> p[12];
      ld_lanes<f2, 12, float>(x0, x1, V, s, p);
      diag([&](int k) { return __ldg(oclov + k * V + own); }, par ? a.mu + a.rho : a.mu, p, acc);
      cx<f2>* to = par ? od : ev;
      if (b0) {
        ld_lanes<f2, 12, float>(b0, b1, V, s, p);
#pragma unroll
        for (int i = 0; i < 12; ++i) st_shared(to + i * kH4 + j, p[i] - acc[i]);
      } else {
#pragma unroll
        for (int i = 0; i < 12; ++i) st_shared(to + i * kH4 + j, czero<f2>() - acc[i]);
      }
    }

    const int nsteps = 2 * a.n_mr + 2;
#pragma unroll 1
    for (int st = 0; st < nsteps; ++st) {
      const int parity = (st & 1) ^ 1;  // even steps work on odd sites
      __syncthreads();
      cx<f2> acc[12];
      if (st > 0) {
        const cx<f2>* src = parity ? ev : od;
        const int own = parity * kH4 + j, oth = (parity ^ 1) * kH4;
        const int lx = 2 * xh + (pr ^ parity);
#pragma unroll
        for (int i = 0; i < 12; ++i) acc[i] = czero<f2>();
        auto hops = [&](auto MUC) {
          constexpr int MU = decltype(MUC)::value;
          const int lm = MU == 0 ? lt : MU == 1 ? lz : MU == 2 ? ly : lx;
          const int js = MU == 0 ? 32 : MU == 1 ? 8 : 2;
          if (lm < 3) {
            const cx<f2>* sp = src + (MU < 3 ? j + js : (j & ~1) + ((lx + 1) >> 1));
            Link<float> U;
            link(MU, own, U);
            hop_lanes<f2, float, MU, true>([&](int i) { return ld_shared(sp + i * kH4); }, U, acc);
          }
          if (lm > 0) {
            const int jn = MU < 3 ? j - js : (j & ~1) + ((lx - 1) >> 1);
            const cx<f2>* sp = src + jn;
            Link<float> U;
            link(MU, oth + jn, U);
            hop_lanes<f2, float, MU, false>([&](int i) { return ld_shared(sp + i * kH4); }, U, acc);
          }
        };
        hops(std::integral_constant<int, 0>{});
        hops(std::integral_constant<int, 1>{});
        hops(std::integral_constant<int, 2>{});
        hops(std::integral_constant<int, 3>{});
      }
      __syncwarp();  // the tensor-memory accesses below are warp-wide
      if (parity) {
        if (st == 0) {
#pragma unroll
          for (int i = 0; i < 12; ++i) acc[i] = ld_shared(od + i * kH4 + j);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          cx<f2> y[6];
#pragma unroll
          for (int i = 0; i < 6; ++i) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {  // chunk (6 h + i) 3 + q: entries 2 q, 2 q + 1 of row i
              cx<float> u, v;
              unpack_chunk<S>(__ldg(odinv + ((6 * h + i) * 3 + q) * Vh), u, v);
              if (q == 0)
                y[i] = lcmul(u, acc[6 * h]);
              else
                lcfma(y[i], u, acc[6 * h + 2 * q]);
              lcfma(y[i], v, acc[6 * h + 2 * q + 1]);
            }
          }
#pragma unroll
          for (int i = 0; i < 6; ++i) st_shared(od + (6 * h + i) * kH4 + j, y[i]);
        }
        if (st == 0) {
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            cx<f2> e[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = czero<f2>();
            tmem_st4(ta + 16 * q, e);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const cx<f2> u = ld_shared(od + (4 * q + i) * kH4 + j);
              e[i] = u + u;
            }
            tmem_st4(ta + 48 + 16 * q, e);
          }
          tmem_wait_st();
        }
      } else {
        cx<f2> rho[12];
#pragma unroll
        for (int i = 0; i < 12; ++i) rho[i] = ld_shared(ev + i * kH4 + j);
        if (st == 1) {
          const f2 hf = bcast<f2>(0.5f);
#pragma unroll
          for (int i = 0; i < 12; ++i)
            st_shared(ev + i * kH4 + j, cx<f2>{lfma(hf, acc[i].r, rho[i].r), lfma(hf, acc[i].i, rho[i].i)});
        } else {
          const f2 mq = bcast<f2>(-0.25f);
#pragma unroll
          for (int i = 0; i < 12; ++i) acc[i] = cx<f2>{mq * acc[i].r, mq * acc[i].i};
          diag([&](int k) { return __ldg(oclov + k * V + j); }, a.mu, rho, acc);  // acc = q
          f2 dots[3] = {bcast<f2>(0.f), bcast<f2>(0.f), bcast<f2>(0.f)}, d1 = bcast<f2>(0.f);
#pragma unroll
          for (int i = 0; i < 12; ++i) {
            dots[0] = lfma(acc[i].r, rho[i].r, lfma(acc[i].i, rho[i].i, dots[0]));  // Re <q, rho>
            dots[1] = lfma(acc[i].r, rho[i].i, dots[1]);                           // Im <q, rho> = the difference
            d1 = lfma(acc[i].i, rho[i].r, d1);
            dots[2] = lfma(acc[i].r, acc[i].r, lfma(acc[i].i, acc[i].i, dots[2]));  // <q, q>
          }
          dots[1] = dots[1] - d1;
#pragma unroll
          for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dots[k] = dots[k] + f2{__shfl_xor_sync(0xffffffffu, dots[k].v, o)};
          }
          if ((j & 31) == 0) {
#pragma unroll
            for (int k = 0; k < 3; ++k) red[(j >> 5) * 3 + k] = dots[k];
          }
          __syncthreads();
#pragma unroll
          for (int k = 0; k < 3; ++k) dots[k] = (red[k] + red[3 + k]) + (red[6 + k] + red[9 + k]);
          const f2 ar = mr_ratio(dots[0], dots[2]), ai = mr_ratio(dots[1], dots[2]);
          const f2 nr = bcast<f2>(0.f) - ar, ni = bcast<f2>(0.f) - ai;
#pragma unroll
          for (int i = 0; i < 12; ++i) {
            cx<f2> q = rho[i];  // rho - alpha q
            q.r = lfma(ai, acc[i].i, lfma(nr, acc[i].r, q.r));
            q.i = lfma(ni, acc[i].r, lfma(nr, acc[i].i, q.i));
            st_shared(ev + i * kH4 + j, q);
          }
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            cx<f2> e[4];
            tmem_ld4(ta + 16 * q, e);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const cx<f2> r = rho[4 * q + i];
              e[i].r = lfma(ni, r.i, lfma(ar, r.r, e[i].r));
              e[i].i = lfma(ai, r.r, lfma(ar, r.i, e[i].i));
            }
            tmem_st4(ta + 16 * q, e);
            tmem_ld4(ta + 48 + 16 * q, e);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const cx<f2> z = ld_shared(od + (4 * q + i) * kH4 + j);
              e[i].r = lfma(ni, z.i, lfma(ar, z.r, e[i].r));
              e[i].i = lfma(ai, z.r, lfma(ar, z.i, e[i].i));
            }
            tmem_st4(ta + 48 + 16 * q, e);
          }
          tmem_wait_st();
        }
      }
    }
    // x_e += e_e, x_o += e_o / 2
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      int c[4];
      const int s = site(par, c);
      const f2 w = bcast<f2>(par ? 0.5f : 1.f);
      cx<f2> p[12];
      ld_lanes<f2, 12, float>(x0, x1, V, s, p);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        cx<f2> e[4];
        tmem_ld4(ta + 48 * par + 16 * q, e);
#pragma unroll
        for (int i = 0; i < 4; ++i) p[4 * q + i] = cx<f2>{lfma(w, e[i].r, p[4 * q + i].r), lfma(w, e[i].i, p[4 * q + i].i)};
      }
      st_lanes<f2, 12, float>(x0, x1, V, s, p);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
}

template <int S>
void sap_oe4_s(const SapOeArgs<float>& a, int nblocks, cudaStream_t st) {
  constexpr size_t smem = 24 * kH4 * sizeof(cx<f2>);
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(k_sap_oe4<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr_set = true;
  }
  k_sap_oe4<S><<<dim3(nblocks * (a.nrhs / 2)), kH4, smem, st>>>(a);
}

}  // namespace

namespace {
// time of `warps` warps, up to four per SM at once in each of N slots: whole waves of N and the rest, in
// units of one slot alone
template <int N>
double wave_time(long warps, const double (&t)[N]) {
  const long c = std::max(1L, (warps + 4 * kSms - 1) / (4 * kSms));
  return (double)(c / N) * t[N - 1] + (c % N ? t[c % N - 1] : 0.0);
}
}  // namespace

// Whole pairs two to a thread and an odd one out in a launch of its own, or all alone: by the waves that each
// takes.  An SM holds three slots of four warps of k_sap_oe on one right-hand side and of k_sap_oe4 (168
// registers), two of k_sap_oe on pairs (255); the times of one, two and three slots are relative to one slot of
// right-hand sides alone.  A lone FP32 right-hand side whose blocks in flight hold more than 64 MB of operator
// reads it from DRAM in every half-step (twice the time; others on the same block share it in L2).  Us of 3
// sweeps, alone against pairs (and one), 4^4 blocks:
//                 FP32 operator                               16-bit
//   rhs           2          3          4          6          2          3          4          6
//   16^3 x 8   306  381   395  676   396  394   499  535   271  356   331  615   332  366   423  505
//   16^4       431  420   556  778   877  599  1112 1013   332  369   429  639   645  523   833  715
//   32 x 16^3  953  734  1154 1308  1512 1300  2096 1857   655  534   847  906  1129 1027  1557 1412
//   24^3 x 16 1343 1337  1808 2448  2292 2008  3300 2844   897  800  1305 1293  1699 1483  2480 2122
// and 2^4 blocks at 16^3 x 8: 2 right-hand sides 642 426, 3 732 745 (FP32), 615 429, 738 743.  Over 722 such pairs
// of times (blocks of 16 to 256 sites, 8^4 to 48 x 24^3, 2 to 12 right-hand sides) the form taken is at most
// 1.08 times slower than the other.
extern "C" int tmamg_sap_oe_paired(const int* nb, const int* blk, int nrhs, int s16) {
  constexpr double alone[3] = {1, 1.3, 1.65}, pairs[2] = {1.3, 1.75}, pairs4[3] = {1.35, 1.93, 2.64};
  const long blocks = (long)nb[0] * nb[1] * nb[2] * nb[3] / 2;  // of one colour
  const int bsites = blk[0] * blk[1] * blk[2] * blk[3];
  const long wpb = (bsites / 2 + 31) / 32, w = blocks * wpb;  // warps per block, per right-hand side
  const bool b4 = s16 != ST_NATIVE && blk[0] == 4 && blk[1] == 4 && blk[2] == 4 && blk[3] == 4;
  double paired = b4 ? wave_time(w * (nrhs / 2), pairs4) : wave_time(w * (nrhs / 2), pairs);
  if (nrhs & 1) {
    const long in_flight = std::min(blocks, 12 * kSms / wpb) * bsites * (s16 == ST_NATIVE ? 768 : 384);
    paired += wave_time(w, alone) * (in_flight > 64e6 ? 2 : 1) + 0.4;
  }
  // blocks of more than 256 sites have no form for pairs
  return nrhs < 2 || bsites > 256 || wave_time(w * nrhs, alone) <= paired ? 0 : nrhs & ~1;
}

template <typename T>
void launch_sap_oe_colour(const void* gauge, const void* clover, const void* dinv, const T* b, T* x,
                          const SapGeom& sg, double mu, double bc_t, int n_mr, int colour, int nrhs, cudaStream_t st,
                          double rho, int s16) {
  const int nblk_colour = sg.nb[0] * sg.nb[1] * sg.nb[2] * sg.nb[3] / 2;
  SapOeArgs<T> a{gauge, clover, dinv, b, x, sg, (T)mu, (T)bc_t, n_mr, colour, nrhs, (T)rho};
  if constexpr (std::is_same<T, float>::value) {
    a.nrhs = tmamg_sap_oe_paired(sg.nb, sg.blk, nrhs, s16);
    if (a.nrhs) {
      bool b4 = s16 != ST_NATIVE;  // k_sap_oe4 has the block shape and 16-bit storage built in
      for (int d = 0; d < 4; ++d) b4 = b4 && sg.blk[d] == 4;
      if (b4 && s16 == ST_F16)
        sap_oe4_s<ST_F16>(a, nblk_colour, st);
      else if (b4)
        sap_oe4_s<ST_BF16>(a, nblk_colour, st);
      else if (s16 == ST_F16)
        sap_oe_s<f2, ST_F16>(a, nblk_colour, st);
      else if (s16 == ST_BF16)
        sap_oe_s<f2, ST_BF16>(a, nblk_colour, st);
      else
        sap_oe_s<f2, ST_NATIVE>(a, nblk_colour, st);
    }
    const long off = (long)a.nrhs * NR_SPINOR * sg.g.V;
    a.nrhs = nrhs - a.nrhs;
    if (!a.nrhs) return;
    a.x += off;
    if (a.b) a.b += off;
    if (s16 == ST_F16) return sap_oe_s<T, ST_F16>(a, nblk_colour, st);
    if (s16 == ST_BF16) return sap_oe_s<T, ST_BF16>(a, nblk_colour, st);
  }
  sap_oe_s<T, ST_NATIVE>(a, nblk_colour, st);
}

template void launch_sap_oe_colour<double>(const void*, const void*, const void*, const double*, double*,
                                           const SapGeom&, double, double, int, int, int, cudaStream_t, double, int);
template void launch_sap_oe_colour<float>(const void*, const void*, const void*, const float*, float*,
                                          const SapGeom&, double, double, int, int, int, cudaStream_t, double, int);

// 16-bit copy in block order of a chunked FP32 field, a chunk plane of n sites per
// blockIdx.y: all V sites, or the V / 2 odd ones by their index s >> 1
template <int KIND>
__global__ void k_to16_blocks(const float4* __restrict__ in, uint2* __restrict__ out, SapGeom sg, int n) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int HB = sg.bsites / 2;
  const bool half = n != sg.g.V;
  int c[4], lc[4], bc[4];
  site_coords(sg.g, half ? 2 * s : s, c);
  if (half) c[3] = (c[3] & ~1) | (((c[0] + c[1] + c[2]) & 1) ^ 1);  // the odd site of the pair (X even)
  for (int d = 0; d < 4; ++d) {
    bc[d] = c[d] / sg.blk[d];
    lc[d] = c[d] - bc[d] * sg.blk[d];
  }
  const int par = (c[0] + c[1] + c[2] + c[3]) & 1;
  const int to = block_linear(sg, bc) * (half ? HB : sg.bsites) + (half ? 0 : par * HB) + half_index(lc, sg.blk);
  const long p = (long)blockIdx.y * n;
  const float4 v = in[p + s];
  unsigned u[2];
  if constexpr (KIND == ST_F16) {
    const __half2 a = __float22half2_rn(make_float2(v.x, v.y)), b = __float22half2_rn(make_float2(v.z, v.w));
    memcpy(&u[0], &a, 4);
    memcpy(&u[1], &b, 4);
  } else {
    const __nv_bfloat162 a = __float22bfloat162_rn(make_float2(v.x, v.y)), b = __float22bfloat162_rn(make_float2(v.z, v.w));
    memcpy(&u[0], &a, 4);
    memcpy(&u[1], &b, 4);
  }
  out[p + to] = make_uint2(u[0], u[1]);
}

void launch_to16_blocks(const float* in, void* out, const SapGeom& sg, int planes, bool odd_only, int kind,
                        cudaStream_t st) {
  const int n = odd_only ? sg.g.V / 2 : sg.g.V;
  dim3 grid((n + 127) / 128, planes);
  if (kind == ST_F16)
    k_to16_blocks<ST_F16><<<grid, 128, 0, st>>>(reinterpret_cast<const float4*>(in), static_cast<uint2*>(out), sg, n);
  else
    k_to16_blocks<ST_BF16><<<grid, 128, 0, st>>>(reinterpret_cast<const float4*>(in), static_cast<uint2*>(out), sg, n);
}

// ===========================================================================
// D_oo^-1 for the odd-even block solve: per odd site the inverses of the two
// chiral 6x6 blocks A_h(x) + i s_h mu (s_0 = -1, s_1 = +1: gamma5 of the
// chirality), Gauss-Jordan with partial pivoting in FP64, stored row-major
// per block as 12 rows of 6 complex, chunked SoA over the V/2 odd sites
// (compact index s >> 1).
// ===========================================================================
namespace {
template <typename T>
__global__ void k_clover_inverse(const double* __restrict__ c64, T* __restrict__ dinv, Lat g, double mu, int* err,
                                 int parity) {
  const long so = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long Vh = g.V / 2;
  if (so >= Vh) return;
  // odd site with compact index so: x-row so / (X/2), x = 2 (so % (X/2)) + parity offset
  const long row = so / (g.L[3] / 2);
  const int xh = (int)(so % (g.L[3] / 2));
  int c[4];
  c[2] = (int)(row % g.L[2]);
  c[1] = (int)((row / g.L[2]) % g.L[1]);
  c[0] = (int)(row / ((long)g.L[2] * g.L[1]));
  c[3] = 2 * xh + (((c[0] + c[1] + c[2]) & 1) ^ parity);
  const int s = ((c[0] * g.L[1] + c[1]) * g.L[2] + c[2]) * g.L[3] + c[3];
  double m72[72];
  ld_re<double, 72>(c64, g.V, s, m72);
  for (int h = 0; h < 2; ++h) {
    cx<double> M[6][12];
    const double* m = m72 + 36 * h;
    for (int i = 0; i < 6; ++i)
      for (int jj = 0; jj < 12; ++jj) M[i][jj] = cx<double>{jj - 6 == i ? 1.0 : 0.0, 0.0};
    for (int i = 0; i < 6; ++i) M[i][i] = cx<double>{m[i], (h == 0 ? -mu : mu)};
    int kk = 6;
    for (int i = 0; i < 6; ++i)
      for (int jj = i + 1; jj < 6; ++jj) {
        M[i][jj] = cx<double>{m[kk], m[kk + 1]};
        M[jj][i] = cx<double>{m[kk], -m[kk + 1]};
        kk += 2;
      }
    for (int col = 0; col < 6; ++col) {
      int piv = col;
      double best = norm2(M[col][col]);
      for (int i = col + 1; i < 6; ++i)
        if (norm2(M[i][col]) > best) {
          best = norm2(M[i][col]);
          piv = i;
        }
      if (!(best > 0)) {
        atomicOr(err, ERRF_SINGULAR);
        return;
      }
      if (piv != col)
        for (int jj = 0; jj < 12; ++jj) {
          const cx<double> t = M[col][jj];
          M[col][jj] = M[piv][jj];
          M[piv][jj] = t;
        }
      const cx<double> pv = M[col][col];
      const double pn = norm2(pv);
      const cx<double> inv{pv.r / pn, -pv.i / pn};
      for (int jj = 0; jj < 12; ++jj) M[col][jj] = inv * M[col][jj];
      for (int i = 0; i < 6; ++i) {
        if (i == col) continue;
        const cx<double> f = M[i][col];
        for (int jj = 0; jj < 12; ++jj) M[i][jj] = M[i][jj] - f * M[col][jj];
      }
    }
    for (int i = 0; i < 6; ++i) {
      cx<T> row6[6];
      for (int jj = 0; jj < 6; ++jj) row6[jj] = cx<T>{(T)M[i][6 + jj].r, (T)M[i][6 + jj].i};
      st_cx<T, 6>(dinv + (long)(h * 6 + i) * 12 * Vh, Vh, so, row6);
    }
  }
}
}  // namespace

template <typename T>
void launch_clover_inverse(const double* c64, T* dinv, const Lat& g, double mu, int* err, cudaStream_t st,
                           int parity) {
  const long Vh = g.V / 2;
  k_clover_inverse<T><<<(unsigned)((Vh + 63) / 64), 64, 0, st>>>(c64, dinv, g, mu, err, parity);
}
template void launch_clover_inverse<double>(const double*, double*, const Lat&, double, int*, cudaStream_t, int);
template void launch_clover_inverse<float>(const double*, float*, const Lat&, double, int*, cudaStream_t, int);

}  // namespace tmamg
