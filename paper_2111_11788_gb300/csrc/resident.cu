// Whole batched solves on small meshes: one launch per batch, a cluster of
// CTAs per sample, every vector of the solve in shared memory.
//
// On these meshes a PCG iteration of separate kernels is bound by launches
// and by the latency of a few short warps, not by arithmetic or memory: a
// 128^2 FP64 GMG solve of one sample took 1782 us, 178 us per iteration,
// where its FP64 operations need 24 us on 8 SMs. Here the
// cluster of C CTAs that owns a sample keeps x, r, p, q, z and every
// multigrid level's b, e and output in shared memory, iterates without
// leaving the kernel (PCG and V-cycle as in the separate kernels: the same
// recurrences, damped-Jacobi V(1,1), stopping tests and refinement loop) and
// pays a cluster barrier where the separate kernels pay a launch.
//
// Layout. A level's interior node slabs (2D: rows, 3D: planes) are dealt to
// the CTAs in bands of R; a band is stored with its boundary columns (0, never
// written). A slab of a neighbouring CTA is read through distributed shared
// memory, a boundary slab is one shared array of zeros. The levels of few
// nodes run on CTA 0 alone, behind ordinary block barriers. Operator data
// (kappa, FP64 2D coefficients, smoother weights) stays in global memory,
// where the setup kernels put it: it is read through L1 / L2 once per stencil.
// Sums are formed per band of the finest level, and the bands depend on the
// mesh alone (a CTA of a larger batch takes several), in a fixed order, so a
// sample's result does not depend on the batch.
#include <cooperative_groups.h>

#include <algorithm>

#include "guess.cuh"
#include "mlmc_internal.cuh"

namespace mlmc {
namespace {

namespace cg = cooperative_groups;

constexpr int RES_THREADS = 256;
constexpr int RES_PER_SM = 3;     // CTAs per SM the registers allow

constexpr int RES_BAND = 512;     // interior nodes from which a mesh gets another band
constexpr int RES_MAX_V = 16;     // bands of a sample, hence CTAs of its cluster
constexpr int RES_PORTABLE = 8;   // CTAs of a portable cluster
constexpr int RES_MAX_LEVELS = MAX_RESIDENT_LEVELS;   // 128 .. 2 cells
constexpr size_t RES_SMEM_MAX = 224 * 1024;
constexpr size_t RES_SMEM_SHARE = 74 * 1024;   // shared memory of a CTA at RES_PER_SM of them
constexpr int64_t RES_SLOTS = 152 * RES_PER_SM;

// scalars of the iteration, formed by one thread of each CTA
struct ResScalars {
  double gamma, alpha, beta, rho, inv;
  int stop;
};

template <class T>
struct ResLevel {
  int n, N1, S;        // cells and nodes per side, nodes per slab
  int R, sh;           // slabs per CTA, log2 R (where levels meet: R a power of two)
  unsigned m1, m2;     // ceil(2^32 / (n - 1)), ceil(2^32 / (n - 1)^2)
  unsigned ob, oe, ot; // shared-memory offsets (bytes) of b, e and the output
  int64_t ns, es;
  T d0, d1;            // operator constants: 2D unused, 3D h / 3 and h / 12
  const T* kap;
  const T* coef;       // FP64 2D
  const T* w;
};

template <class T>
struct ResArgs {
  int K, C, nd;        // multigrid levels; CTAs per sample; levels split over the CTAs
  int V, nv, Rv;       // level 0: bands the sums are formed in, bands per CTA, slabs per band (most of them)
  int shv;             // log2 V
  ResLevel<T> lv[RES_MAX_LEVELS];
  unsigned ox, op, oz, ored, osw, osc;   // x, p, zeros, sums, scalars
  unsigned bytes;
  int64_t B;
  const double* kap64; // mixed: operator data of the FP64 residual
  const double* coef64;
  double tol;          // stop at ||r|| <= tol
  double bval;         // h^dim, the right-hand side at interior nodes
  int max_iter;        // CG cap (mixed: of each inner solve)
  double inner_rtol, scale0;
  int outer_max;
  const double* uc;    // nested guess: the coarse-mesh solution, or null
  int64_t ucs;
  double* u;           // solution (node arrays of the level-0 stride)
  double* r;           // mixed: the FP64 residual
  double* q;
  int32_t *iters, *iters2;
  int box, L, H;
  double qw;
};

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}

template <int DIM, class T, bool MIXED>
struct Res {
  const ResArgs<T>& a;
  unsigned char* sm;
  int rank;
  int64_t smp;
  int tid;
  int slot;
  int f0, c0;   // level 0: this CTA's first slab and its slabs

  __device__ __forceinline__ bool mine(int l) const { return l < a.nd || rank == 0; }
  // the slabs of level 0 before band v: bands of Rv slabs where levels meet, else
  // (one level, any n) even shares of the n - 1 slabs
  __device__ __forceinline__ int edge(int v) const {
    const int m = a.lv[0].n - 1;
    return a.K == 1 ? (v * m) >> a.shv : min(v * a.Rv, m);
  }
  __device__ __forceinline__ void deal() {
    f0 = edge(rank * a.nv) + 1;
    c0 = edge((rank + 1) * a.nv) + 1 - f0;
  }
  __device__ __forceinline__ int first(int l) const { return l == 0 ? f0 : l < a.nd ? rank * a.lv[l].R + 1 : 1; }
  __device__ __forceinline__ int own(int l) const {
    if (l == 0) return c0;
    const int n = a.lv[l].n;
    return max(0, min(a.lv[l].R, n - first(l)));
  }
  __device__ __forceinline__ void level_sync(int l) const {
    if (l < a.nd) cluster_barrier();
    else if (rank == 0) __syncthreads();
  }
  // every CTA of the cluster
  __device__ __forceinline__ void all_sync() const {
    if (a.C > 1) cluster_barrier();
    else __syncthreads();
  }
  template <class V>
  __device__ __forceinline__ V* at(unsigned off) const {
    return reinterpret_cast<V*>(sm + off);
  }
  template <class V>
  __device__ __forceinline__ V* remote(V* p, int r) const {
    return r == rank ? p : cg::this_cluster().map_shared_rank(p, r);
  }
  // slab z of a level-l array (boundary slabs: zeros)
  template <class V>
  __device__ __forceinline__ const V* slab(int l, unsigned off, int z) const {
    const ResLevel<T>& L = a.lv[l];
    if (z <= 0 || z >= L.n) return at<V>(a.oz);
    if (l >= a.nd) return remote(at<V>(off) + (z - 1) * L.S, 0);
    return remote(at<V>(off) + ((z - 1) & (L.R - 1)) * L.S, (z - 1) >> L.sh);
  }
  // the slabs before and after this CTA's band
  template <class V>
  __device__ __forceinline__ const V* before(int l, unsigned off) const {
    if (l >= a.nd || rank == 0) return at<V>(a.oz);
    const int last = (a.K == 1 ? f0 - 1 - edge((rank - 1) * a.nv) : a.lv[l].R) - 1;
    return remote(at<V>(off) + last * a.lv[l].S, rank - 1);
  }
  template <class V>
  __device__ __forceinline__ const V* after(int l, unsigned off) const {
    if (l >= a.nd || first(l) + own(l) >= a.lv[l].n) return at<V>(a.oz);
    return remote(at<V>(off), rank + 1);
  }
  // f(js, o, i, j): interior nodes of `cnt` slabs of this CTA from slab s0 on,
  // slab js of its band, offset o in the slab, column i (3D: row j)
  template <class F>
  __device__ __forceinline__ void slab_nodes(int l, int s0, int cnt, F&& f) const {
    const ResLevel<T>& L = a.lv[l];
    const int m = L.n - 1;
    if constexpr (DIM == 2) {
      const int total = cnt * m;
      for (int x = tid; x < total; x += RES_THREADS) {
        const int js = (int)__umulhi((unsigned)x, L.m1), i = x - js * m + 1;
        f(s0 + js, i, i, 0);
      }
    } else {
      const int total = cnt * m * m;
      for (int x = tid; x < total; x += RES_THREADS) {
        const int js = (int)__umulhi((unsigned)x, L.m2), r = x - js * m * m;
        const int j = (int)__umulhi((unsigned)r, L.m1) + 1, i = r - (j - 1) * m + 1;
        f(s0 + js, j * L.N1 + i, i, j);
      }
    }
  }
  template <class F>
  __device__ __forceinline__ void nodes(int l, F&& f) const {
    slab_nodes(l, 0, own(l), f);
  }
  // The nodes of level 0 band by band, done(v) after band v: a sum is formed
  // per band, in an order that does not depend on how many bands a CTA has.
  template <class F, class D>
  __device__ __forceinline__ void nodes0(F&& f, D&& done) const {
    for (int v = 0, s0 = 0; v < a.nv; ++v) {
      const int s1 = edge(rank * a.nv + v + 1) + 1 - f0;
      slab_nodes(0, s0, s1 - s0, f);
      done(v);
      s0 = s1;
    }
  }
  // f - (A v) at node (o, i, j) of slab z, v given by the slabs around it
  template <class V>
  __device__ __forceinline__ V resid(int n, int64_t ns, V d0, V d1, const V* __restrict__ kap,
                                     const V* __restrict__ coef, const V* vm, const V* v0, const V* vp, int z, int o,
                                     int i, int j, V f) const {
    const int N1 = n + 1;
    if constexpr (DIM == 2) {
      const int g = z * N1 + o, e = z * n + o;
      if constexpr (sizeof(V) == 8) {
        const V* cd = coef;
        const V* ce = coef + ns;
        const V* cn = coef + 2 * ns;
        const V* q = coef + 3 * ns;
        V s = fma(-__ldg(cd + g), v0[o], f);
        s = fma(-__ldg(ce + g), v0[o + 1], s);
        s = fma(-__ldg(ce + g - 1), v0[o - 1], s);
        s = fma(-__ldg(cn + g), vp[o], s);
        s = fma(-__ldg(cn + g - N1), vm[o], s);
        s = fma(-__ldg(q + e), vp[o + 1], s);
        s = fma(-__ldg(q + e - 1), vp[o - 1], s);
        s = fma(-__ldg(q + e - n), vm[o + 1], s);
        return fma(-__ldg(q + e - n - 1), vm[o - 1], s);
      } else {
        const V ksw = __ldg(kap + e - n - 1), kse = __ldg(kap + e - n), knw = __ldg(kap + e - 1), kne = __ldg(kap + e);
        const V kS = ksw + kse, kN = knw + kne, kW = ksw + knw, kE = kse + kne;
        const V edge = kE * v0[o + 1] + kW * v0[o - 1] + kN * vp[o] + kS * vm[o];
        const V corner = kne * vp[o + 1] + knw * vp[o - 1] + kse * vm[o + 1] + ksw * vm[o - 1];
        return f - (V(2) / V(3) * (kS + kN) * v0[o] - V(1) / V(6) * edge - V(1) / V(3) * corner);
      }
    } else {
      const V* K = kap + ((int64_t)(z - 1) * n + (j - 1)) * n + (i - 1);
      V k[2][2][2];
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          k[c][b][0] = __ldg(K + (c * n + b) * n);
          k[c][b][1] = __ldg(K + (c * n + b) * n + 1);
        }
      auto v = [&](int dx, int dy, int dz) -> V { return (dz < 0 ? vm : dz > 0 ? vp : v0)[o + dy * N1 + dx]; };
      V u = V(0);
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          u = fma(k[0][q][p] + k[1][q][p], v(2 * p - 1, 2 * q - 1, 0), u);
          u = fma(k[q][0][p] + k[q][1][p], v(2 * p - 1, 0, 2 * q - 1), u);
          u = fma(k[q][p][0] + k[q][p][1], v(0, 2 * p - 1, 2 * q - 1), u);
        }
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int p = 0; p < 2; ++p) u = fma(k[c][b][p], v(2 * p - 1, 2 * b - 1, 2 * c - 1), u);
      const V s = ((k[0][0][0] + k[0][0][1]) + (k[0][1][0] + k[0][1][1])) +
                  ((k[1][0][0] + k[1][0][1]) + (k[1][1][0] + k[1][1][1]));
      return fma(d1, u, fma(-d0, s * v0[o], f));
    }
  }
  // f(index in the band, node, rhs - A v) over the band of level l, v the array
  // at `off`; on level 0 band by band with done(v)
  template <class RhsF, class F, class D>
  __device__ __forceinline__ void stencil(int l, unsigned off, RhsF&& rhs, F&& f, D&& done) const {
    const ResLevel<T>& L = a.lv[l];
    const int n = L.n, S = L.S, z0 = first(l), cnt = own(l);
    const T* v = at<T>(off);
    const T* lo = before<T>(l, off);
    const T* hi = after<T>(l, off);
    const T* kap = L.kap + smp * L.es;
    const T* coef = (DIM == 2 && sizeof(T) == 8) ? L.coef + smp * (3 * L.ns + L.es) : nullptr;
    auto node = [&](int js, int o, int i, int j) {
      const T* v0 = v + js * S;
      const T* vm = js > 0 ? v0 - S : lo;
      const T* vp = js < cnt - 1 ? v0 + S : hi;
      f(js * S + o, (z0 + js) * S + o, resid<T>(n, L.ns, L.d0, L.d1, kap, coef, vm, v0, vp, z0 + js, o, i, j, rhs(js * S + o)));
    };
    if (l > 0) {
      slab_nodes(l, 0, cnt, node);
      return;
    }
    for (int v = 0, s0 = 0; v < a.nv; ++v) {
      const int s1 = edge(rank * a.nv + v + 1) + 1 - f0;
      slab_nodes(l, s0, s1 - s0, node);
      done(v);
      s0 = s1;
    }
  }
  // Sums over the sample: every thread hands in its part of each of its CTA's
  // bands (part, quantity q), then total() adds them up in a fixed order
  // (threads, warps' lanes, bands) and thread 0 of every CTA turns the sums
  // into what all threads then read (f, with a block barrier after it): the
  // additions, divisions and roots are FP64, 64 cycles of an SM partition per
  // warp instruction, so as few warps as possible execute them. Holds a
  // barrier of the cluster.
  template <class V>
  __device__ __forceinline__ void part(int q, int v, V x) const {
    at<V>(a.osw + (unsigned)((q * a.nv + v) * RES_THREADS * 8))[tid] = x;
  }
  template <class V, class F>
  __device__ __forceinline__ void total(int nq, F&& f) {
    double* red = at<double>(a.ored) + slot * 2 * RES_MAX_V;
    __syncthreads();
    const int lane = tid & 31;
    for (int w = tid >> 5; w < nq * a.nv; w += RES_THREADS / 32) {
      const V* s = at<V>(a.osw + (unsigned)(w * RES_THREADS * 8));
      double t = (double)s[lane];
#pragma unroll
      for (int k = 1; k < RES_THREADS / 32; ++k) t += (double)s[k * 32 + lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      t = __shfl_sync(0xffffffffu, t, 0);
      const int q = w >= a.nv ? 1 : 0;
      if (lane < a.C) *remote(red + q * RES_MAX_V + rank * a.nv + (w - q * a.nv), lane) = t;
    }
    all_sync();
    if (tid < 32) {
      double t = 0.0;
      if (lane < 2)
        for (int r = 0; r < a.V; ++r) t += red[lane * RES_MAX_V + r];
      const double t1 = __shfl_sync(0xffffffffu, t, 1);
      if (tid == 0) f(t, t1);
    }
    __syncthreads();
    slot = (slot + 1) & 3;
  }
  // full weighting of level l's output array into b of level l + 1; e = W b
  // there (on the coarsest grid the exact solve of its one unknown)
  __device__ __forceinline__ void restrict_to(int c) const {
    const int l = c - 1, Nf = a.lv[l].N1;
    const ResLevel<T>& L = a.lv[c];
    const T h = T(0.5);
    auto row = [&](const T* r) { return h * r[-1] + r[0] + h * r[1]; };
    auto plane = [&](const T* r) { return h * row(r - Nf) + row(r) + h * row(r + Nf); };
    auto value = [&](int z, int i, int j) -> T {
      const T* f0 = slab<T>(l, a.lv[l].ot, 2 * z - 1);
      const T* f1 = slab<T>(l, a.lv[l].ot, 2 * z);
      const T* f2 = slab<T>(l, a.lv[l].ot, 2 * z + 1);
      if constexpr (DIM == 2) return h * (row(f0 + 2 * i) + row(f2 + 2 * i)) + row(f1 + 2 * i);
      const int o = 2 * j * Nf + 2 * i;
      return h * plane(f0 + o) + plane(f1 + o) + h * plane(f2 + o);
    };
    if (c == a.K - 1) {
      if (tid == 0) {
        const T* k = L.kap + smp * L.es;
        T s = T(0);
        for (int e = 0; e < (DIM == 2 ? 4 : 8); ++e) s += k[e];
        at<T>(L.ot)[DIM == 2 ? 1 : L.N1 + 1] = value(1, 1, 1) / ((DIM == 2 ? T(2) / T(3) : L.d0) * s);
      }
      return;
    }
    T* b = at<T>(L.ob);
    T* e = at<T>(L.oe);
    const T* w = L.w + smp * L.ns;
    const int S = L.S, z0 = first(c);
    nodes(c, [&](int js, int o, int i, int j) {
      const T v = value(z0 + js, i, j);
      b[js * S + o] = v;
      e[js * S + o] = __ldg(w + (z0 + js) * S + o) * v;
    });
  }
  // (P v)(z, o) at a fine node of level l, v a coarse array given by slab(z)
  template <class V, class SlabF>
  __device__ __forceinline__ V prolong(SlabF&& cs, int C1, int z, int i, int j) const {
    const int I = i >> 1, oz = z & 1, ox = i & 1;
    const V* s0 = cs(z >> 1);
    const V* s1 = oz ? cs((z >> 1) + 1) : s0;
    if constexpr (DIM == 2) {
      V v0 = s0[I];
      if (ox) v0 = V(0.5) * (v0 + s0[I + 1]);
      if (!oz) return v0;
      V v1 = s1[I];
      if (ox) v1 = V(0.5) * (v1 + s1[I + 1]);
      return V(0.5) * (v0 + v1);
    } else {
      const int J = j >> 1, oy = j & 1;
      V t0 = V(0), t1 = V(0);
      for (int c = 0; c <= oz; ++c)
        for (int b = 0; b <= oy; ++b) {
          const V* r = (c ? s1 : s0) + (J + b) * C1;
          t0 += r[I];
          if (ox) t1 += r[I + 1];
        }
      const int rows = oy + oz;
      const V inv = rows == 0 ? V(1) : (rows == 1 ? V(0.5) : V(0.25));
      return ox ? V(0.5) * (t0 + t1) * inv : t0 * inv;
    }
  }
  // z = M r (r: level 0's b, with e = W r in place; z: its output array); hands
  // in the parts of r.z (Dot)
  template <bool Dot>
  __device__ __forceinline__ void vcycle() const {
    T dot = T(0);
    for (int l = 0; l < a.K - 1; ++l) {
      const ResLevel<T>& L = a.lv[l];
      if (mine(l)) {
        const T* b = at<T>(L.ob);
        T* t = at<T>(L.ot);
        stencil(l, L.oe, [&](int x) { return b[x]; }, [&](int x, int, T r) { t[x] = r; }, [](int) {});
      }
      level_sync(l);
      if (mine(l + 1)) restrict_to(l + 1);
      level_sync(l + 1);
    }
    for (int l = a.K - 2; l >= 0; --l) {
      const ResLevel<T>& L = a.lv[l];
      if (l == a.nd - 1) cluster_barrier();   // CTA 0 has finished its levels
      if (mine(l)) {
        const unsigned oc = a.lv[l + 1].ot;
        const int S = L.S, z0 = first(l), C1 = a.lv[l + 1].N1;
        T* e = at<T>(L.oe);
        nodes(l, [&](int js, int o, int i, int j) {
          e[js * S + o] += prolong<T>([&](int z) { return slab<T>(l + 1, oc, z); }, C1, z0 + js, i, j);
        });
      }
      level_sync(l);
      if (mine(l)) {
        const T* b = at<T>(L.ob);
        const T* e = at<T>(L.oe);
        T* t = at<T>(L.ot);
        const T* w = L.w + smp * L.ns;
        stencil(l, L.oe, [&](int x) { return b[x]; }, [&](int x, int g, T r) {
          const T v = fma(__ldg(w + g), r, e[x]);
          t[x] = v;
          if (Dot && l == 0) dot = fma(b[x], v, dot);
        }, [&](int v) {
          if constexpr (Dot) part(0, v, dot);
          dot = T(0);
        });
      }
      if (l > 0 && l != a.nd) level_sync(l);
    }
  }
  // PCG on level 0's b (overwritten by the residual) from the x in place;
  // returns the iterations, or -1 at the cap
  __device__ int pcg(double tol, int max_iter) {
    const ResLevel<T>& L = a.lv[0];
    const int S = L.S, z0 = first(0);
    const bool mg = a.K > 1;
    T* x = at<T>(a.ox);
    T* p = at<T>(a.op);
    T* r = at<T>(L.ob);
    T* q = at<T>(L.oe);
    const T* zv = at<T>(L.ot);
    const T* w = L.w + smp * L.ns;
    ResScalars& sc = *at<ResScalars>(a.osc);
    T dot = T(0), dz = T(0);
    auto hand_in = [&](int v) {
      part(0, v, dot);
      dot = T(0);
    };
    // what follows deals the nodes to the threads band by band, or all bands at
    // once, unlike the caller that wrote r
    __syncthreads();
    if (mg) {
      nodes(0, [&](int js, int o, int, int) { q[js * S + o] = __ldg(w + (z0 + js) * S + o) * r[js * S + o]; });
      all_sync();
      vcycle<true>();
    } else nodes0([&](int js, int o, int, int) {
      const T rv = r[js * S + o];
      dot = fma(rv, __ldg(w + (z0 + js) * S + o) * rv, dot);
    }, hand_in);
    total<T>(1, [&](double g, double) {
      sc.gamma = g;
      sc.beta = 0.0;
    });
    for (int it = 1;; ++it) {
      const T bb = (T)sc.beta;
      nodes(0, [&](int js, int o, int, int) {
        const int k = js * S + o;
        const T z = mg ? zv[k] : __ldg(w + (z0 + js) * S + o) * r[k];
        p[k] = bb == T(0) ? z : fma(bb, p[k], z);
      });
      all_sync();
      stencil(0, a.op, [](int) { return T(0); }, [&](int k, int, T v) {
        q[k] = -v;
        dot = fma(p[k], -v, dot);
      }, hand_in);
      total<T>(1, [&](double delta, double) { sc.alpha = delta > 0.0 ? sc.gamma / delta : 0.0; });
      const T al = (T)sc.alpha;
      nodes0([&](int js, int o, int, int) {
        const int k = js * S + o;
        x[k] = fma(al, p[k], x[k]);
        const T rv = fma(-al, q[k], r[k]);
        r[k] = rv;
        dot = fma(rv, rv, dot);
        const T wr = __ldg(w + (z0 + js) * S + o) * rv;
        if (mg) q[k] = wr;   // q's array is level 0's e
        else dz = fma(rv, wr, dz);
      }, [&](int v) {
        hand_in(v);
        if (!mg) part(1, v, dz);
        dz = T(0);
      });
      total<T>(mg ? 1 : 2, [&](double rr, double rz) {
        const double rho = sqrt(rr);
        sc.stop = rho <= tol ? 1 : (it >= max_iter || !(rho == rho) ? 2 : 0);
        if (!mg) {
          sc.beta = sc.gamma != 0.0 ? rz / sc.gamma : 0.0;
          sc.gamma = rz;
        }
      });
      if (sc.stop) return sc.stop == 1 ? it : -1;
      if (mg) {
        vcycle<true>();
        total<T>(1, [&](double rz, double) {
          sc.beta = sc.gamma != 0.0 ? rz / sc.gamma : 0.0;
          sc.gamma = rz;
        });
      }
    }
  }
  // The sample's solution in global memory, boundary included, as zeros.
  __device__ __forceinline__ double* zero_solution() const {
    const ResLevel<T>& L = a.lv[0];
    const int S = L.S, z0 = first(0), cnt = own(0);
    double* u = a.u + smp * L.ns;
    for (int k = tid; k < cnt * S; k += RES_THREADS) u[z0 * S + k] = 0.0;
    if (rank == 0)
      for (int k = tid; k < S; k += RES_THREADS) u[k] = 0.0;
    if (cnt > 0 && z0 + cnt == L.n)
      for (int k = tid; k < S; k += RES_THREADS) u[L.n * S + k] = 0.0;
    return u;
  }
  // QoI of the solution (val(js, o): its value at a node of this CTA) and the iteration count
  template <class ValF>
  __device__ __forceinline__ void finish(ValF&& val, int iters) {
    const int z0 = first(0);
    double acc = 0.0;
    auto chi = [&](int i) { return i > a.L && i < a.H ? 1.0 : (i == a.L || i == a.H ? 0.5 : 0.0); };
    nodes0([&](int js, int o, int i, int j) {
      double wt = a.qw;
      if (a.box) wt *= DIM == 2 ? chi(i) * chi(z0 + js) : chi(i) * chi(j) * chi(z0 + js);
      acc = fma(wt, val(js, o), acc);
    }, [&](int v) {
      part(0, v, acc);
      acc = 0.0;
    });
    total<double>(1, [&](double t, double) {
      if (rank != 0) return;
      a.q[smp] = t;
      a.iters[smp] = iters;
      if (a.iters2) a.iters2[smp] = iters;
    });
  }
  // set(js, o, value): the nested initial guess P uc at this CTA's nodes
  template <class SetF>
  __device__ __forceinline__ void initial(SetF&& set) const {
    const ResLevel<T>& L = a.lv[0];
    const int z0 = first(0), C1 = L.n / 2 + 1, CS = DIM == 2 ? C1 : C1 * C1;
    const double* uc = a.uc + smp * a.ucs;
    const bool cubic = C1 > CUBIC_MIN_CELLS;
    nodes(0, [&](int js, int o, int i, int j) {
      if (cubic) {
        auto row = [&](const double* r) { return cubic_at(i, C1 - 1, [&](int c) { return __ldg(r + c); }); };
        auto plane = [&](const double* p) {
          return DIM == 2 ? row(p) : cubic_at(j, C1 - 1, [&](int k) { return row(p + k * C1); });
        };
        set(js, o, cubic_at(z0 + js, C1 - 1, [&](int k) { return plane(uc + k * CS); }));
      } else {
        set(js, o, prolong<double>([&](int z) { return uc + z * CS; }, C1, z0 + js, i, j));
      }
    });
  }
  __device__ void solve_fp64() {
    const ResLevel<T>& L = a.lv[0];
    double* x = at<double>(a.ox);
    double* r = at<double>(L.ob);
    const int S = L.S, z0 = first(0), cnt = own(0);
    double* u = zero_solution();
    if (a.uc) {
      initial([&](int js, int o, double v) { x[js * S + o] = v; });
      all_sync();
      if constexpr (!MIXED)
        stencil(0, a.ox, [&](int) { return (T)a.bval; }, [&](int k, int, T v) { r[k] = v; }, [](int) {});
    } else {
      nodes(0, [&](int js, int o, int, int) { r[js * S + o] = a.bval; });
    }
    const int it = pcg(a.tol, a.max_iter);
    for (int k = tid; k < cnt * S; k += RES_THREADS) u[z0 * S + k] = x[k];
    finish([&](int js, int o) { return x[js * S + o]; }, it);
  }
  // Mixed form: FP64 refinement around the FP32 PCG. The solution and the
  // residual stay in global memory (they are touched once per refinement step,
  // and shared memory is what limits the CTAs on an SM); the residual is kept in
  // FP64 and rounded once, scaled to unit norm, into the inner right-hand side.
  __device__ void solve_mixed() {
    const ResLevel<T>& L = a.lv[0];
    const int n = L.n, S = L.S, z0 = first(0);
    double* u = zero_solution();
    double* res = a.r + smp * L.ns;
    T* x = at<T>(a.ox);
    T* b = at<T>(L.ob);
    ResScalars& sc = *at<ResScalars>(a.osc);
    const double* kap = a.kap64 + smp * L.es;
    const double* coef = DIM == 2 ? a.coef64 + smp * (3 * L.ns + L.es) : nullptr;
    const double h = 1.0 / n;
    double scale = a.scale0;
    int count = 0, iters = -1;
    // r = b - A u; stop: 1 converged (or stalled at the rounding floor of the
    // FP64 residual), 2 ended without
    auto step = [&](int outer) {
      double dot = 0.0;
      nodes0([&](int js, int o, int i, int j) {
        const double* v0 = u + (z0 + js) * S;
        const double r = resid<double>(n, L.ns, h / 3.0, h / 12.0, kap, coef, v0 - S, v0, v0 + S, z0 + js, o, i, j,
                                       a.bval);
        res[(z0 + js) * S + o] = r;
        dot = fma(r, r, dot);
      }, [&](int v) {
        part(0, v, dot);
        dot = 0.0;
      });
      total<double>(1, [&](double rr, double) {
        const double rho = sqrt(rr);
        sc.stop = rho <= a.tol || (rho > 0.5 * scale && rho <= 100.0 * a.tol)
                      ? 1
                      : (outer >= a.outer_max || !(rho == rho) ? 2 : 0);
        sc.rho = rho;
        sc.inv = 1.0 / rho;
      });
      scale = sc.rho;
      if (sc.stop == 1) iters = count;
      return sc.stop != 0;
    };
    bool done = false;
    double inv = 1.0 / scale;
    if (a.uc) {
      __syncthreads();   // the zeros of this CTA's slabs before its values
      initial([&](int js, int o, double v) { u[(z0 + js) * S + o] = v; });
      all_sync();
      done = step(0);
      inv = sc.inv;
    } else {
      nodes(0, [&](int js, int o, int, int) { res[(z0 + js) * S + o] = a.bval; });
    }
    for (int outer = 1; !done; ++outer) {
      nodes(0, [&](int js, int o, int, int) {
        const int k = js * S + o;
        b[k] = (T)(res[(z0 + js) * S + o] * inv);
        x[k] = T(0);
      });
      const int it = pcg(a.inner_rtol, a.max_iter);
      count += it > 0 ? it : a.max_iter;
      nodes(0, [&](int js, int o, int, int) {
        double* v = u + (z0 + js) * S + o;
        *v = fma(scale, (double)x[js * S + o], *v);
      });
      all_sync();
      done = step(outer);
      inv = sc.inv;
    }
    finish([&](int js, int o) { return u[(z0 + js) * S + o]; }, iters);
  }
};

// 2D: 64 registers without spills, a fourth CTA on an SM where its shared memory
// fits (300 mixed samples of 128^2: 3.82 -> 3.01 ms)
template <int DIM, class T, bool MIXED>
__global__ void __launch_bounds__(RES_THREADS, DIM == 2 ? RES_PER_SM + 1 : RES_PER_SM)
    k_resident(const __grid_constant__ ResArgs<T> a) {
  extern __shared__ __align__(16) unsigned char res_sm[];
  const int tid = threadIdx.x;
  for (int64_t smp = blockIdx.x / a.C; smp < a.B; smp += gridDim.x / a.C) {
    Res<DIM, T, MIXED> s{a, res_sm, (int)(blockIdx.x % a.C), smp, tid, 0, 0, 0};
    s.deal();
    for (unsigned k = tid; k < a.bytes / 8; k += RES_THREADS) reinterpret_cast<double*>(res_sm)[k] = 0.0;
    s.all_sync();   // the cluster has started and every array is zero
    if constexpr (MIXED) s.solve_mixed();
    else s.solve_fp64();
    s.all_sync();   // no CTA goes on while another may read its arrays
  }
}

// The levels of at most 64^2 (2D) or 16^3 (3D) cells below the finest of a
// larger mesh's V-cycle, for a PCG of separate kernels: from b on the finest of
// them to the post-smoothed correction out, with the same vcycle(). `cycles` 2:
// a second cycle on the residual of the first.
template <int DIM, class T>
__global__ void __launch_bounds__(RES_THREADS, RES_PER_SM) k_bottom(const __grid_constant__ ResArgs<T> a,
                                                                    const T* __restrict__ Bv, T* __restrict__ Out,
                                                                    const int32_t* __restrict__ active, int cycles,
                                                                    Prof prof) {
  extern __shared__ __align__(16) unsigned char res_sm[];
  const int tid = threadIdx.x;
  Res<DIM, T, false> s{a, res_sm, (int)(blockIdx.x % a.C), (int64_t)(blockIdx.x / a.C), tid, 0, 0, 0};
  s.deal();
  if (!active[s.smp]) return;   // the whole cluster
  for (unsigned k = tid; k < a.bytes / 8; k += RES_THREADS) reinterpret_cast<double*>(res_sm)[k] = 0.0;
  __syncthreads();
  const ResLevel<T>& L = a.lv[0];
  const int S = L.S, z0 = s.first(0), cnt = s.own(0);
  T* b = s.template at<T>(L.ob);
  T* e = s.template at<T>(L.oe);
  const T* t = s.template at<T>(L.ot);
  const T* w = L.w + s.smp * L.ns;
  const T* src = Bv + s.smp * L.ns;
  T* out = Out + s.smp * L.ns;
  s.nodes(0, [&](int js, int o, int, int) {
    const int g = (z0 + js) * S + o;
    const T v = src[g];
    b[js * S + o] = v;
    e[js * S + o] = __ldg(w + g) * v;
  });
  s.all_sync();   // the cluster has started and every array is in place
  s.template vcycle<false>();
  if (cycles > 1) {
    s.all_sync();
    for (int k = tid; k < cnt * S; k += RES_THREADS) out[z0 * S + k] = t[k];
    s.stencil(0, L.ot, [&](int x) { return b[x]; },
              [&](int x, int g, T r) {
                b[x] = r;
                e[x] = __ldg(w + g) * r;
              }, [](int) {});
    s.all_sync();
    s.template vcycle<false>();
  }
  __syncthreads();
  for (int k = tid; k < cnt * S; k += RES_THREADS) out[z0 * S + k] = cycles > 1 ? out[z0 * S + k] + t[k] : t[k];
  if (s.rank == 0)
    for (int k = tid; k < S; k += RES_THREADS) out[k] = T(0);
  if (cnt > 0 && z0 + cnt == L.n)
    for (int k = tid; k < S; k += RES_THREADS) out[L.n * S + k] = T(0);
  if (prof.acc && s.rank == 0 && tid == 0) atomicAdd(prof.acc, prof.per_sample);
  s.all_sync();   // no CTA leaves while another may read its arrays
}

// Setup, first launch: one CTA per sample makes the kappa hierarchy (mixed
// form: the FP32 kappa of the finest mesh too, unless it is given).
template <class T>
struct ResKappa {
  int K, dim;
  int n[RES_MAX_LEVELS];
  int64_t es[RES_MAX_LEVELS];
  T* kap[RES_MAX_LEVELS];
  const double* kap64;   // mixed: rounded into kap[0]; else null
};
template <class T>
__global__ void __launch_bounds__(512) k_res_kappa(const __grid_constant__ ResKappa<T> a) {
  const int64_t b = blockIdx.x;
  if (a.kap64) {
    const int ne = a.dim == 2 ? a.n[0] * a.n[0] : a.n[0] * a.n[0] * a.n[0];
    for (int e = threadIdx.x; e < ne; e += 512) a.kap[0][b * a.es[0] + e] = (T)a.kap64[b * a.es[0] + e];
    __syncthreads();
  }
  for (int l = 1; l < a.K; ++l) {
    const T* f = a.kap[l - 1] + b * a.es[l - 1];
    T* c = a.kap[l] + b * a.es[l];
    const int nc = a.n[l], nf = 2 * nc, pl = nf * nf;
    const int ne = a.dim == 2 ? nc * nc : nc * nc * nc;
    for (int e = threadIdx.x; e < ne; e += 512) {
      if (a.dim == 2) {
        const int J = e / nc, I = e - J * nc;
        const T* g = f + 2 * J * nf + 2 * I;
        c[e] = T(0.25) * ((g[0] + g[1]) + (g[nf] + g[nf + 1]));
      } else {
        const int Z = e / (nc * nc), r = e - Z * nc * nc, J = r / nc, I = r - J * nc;
        const T* g = f + 2 * Z * pl + 2 * J * nf + 2 * I;
        const T s0 = (g[0] + g[1]) + (g[nf] + g[nf + 1]);
        const T s1 = (g[pl] + g[pl + 1]) + (g[pl + nf] + g[pl + nf + 1]);
        c[e] = T(0.125) * (s0 + s1);
      }
    }
    __syncthreads();
  }
}

// Setup, second launch: smoother weights of every level and the FP64 2D
// operator coefficients, a thread per node of any level.
template <class T>
struct ResCoefs {
  int kw, dim;           // levels
  int n[RES_MAX_LEVELS];
  int64_t off[RES_MAX_LEVELS + 1];   // first thread of each level
  int64_t ns[RES_MAX_LEVELS], es[RES_MAX_LEVELS];
  const T* kap[RES_MAX_LEVELS];
  T* w[RES_MAX_LEVELS];
  T* coef[RES_MAX_LEVELS];   // FP64 2D: coefficient blocks, else null
  const double* kap64;       // mixed 2D: the finest mesh's FP64 coefficients too
  double* coef64;
  double omega;
};
template <class V>
__device__ __forceinline__ V res_coefs(const V* __restrict__ k, int n, int64_t ns, int x, V* __restrict__ cb) {
  const int N1 = n + 1, j = x / N1, i = x - j * N1;
  auto at = [&](int c, int r) -> V { return (c >= 0 && c < n && r >= 0 && r < n) ? k[r * n + c] : V(0); };
  const V ksw = at(i - 1, j - 1), kse = at(i, j - 1), knw = at(i - 1, j), kne = at(i, j);
  const bool in = i > 0 && i < n && j > 0 && j < n;
  const V d = in ? V(2) / V(3) * ((ksw + kse) + (knw + kne)) : V(0);
  if (cb) {
    cb[x] = d;
    cb[ns + x] = -(V(1) / V(6)) * (kse + kne);
    cb[2 * ns + x] = -(V(1) / V(6)) * (knw + kne);
    if (i < n && j < n) cb[3 * ns + j * n + i] = -(V(1) / V(3)) * kne;
  }
  return d;
}
template <class T>
__global__ void __launch_bounds__(256) k_res_coefs(const __grid_constant__ ResCoefs<T> a) {
  const int64_t b = blockIdx.y;
  const int64_t g = (int64_t)blockIdx.x * 256 + threadIdx.x;
  int l = 0;
  while (l < a.kw && g >= a.off[l + 1]) ++l;
  if (l >= a.kw) return;
  const int x = (int)(g - a.off[l]), n = a.n[l], N1 = n + 1;
  const T* k = a.kap[l] + b * a.es[l];
  T d = T(0);
  if (a.dim == 2) {
    d = res_coefs<T>(k, n, a.ns[l], x, a.coef[l] ? a.coef[l] + b * (3 * a.ns[l] + a.es[l]) : nullptr);
    if (l == 0 && a.coef64)
      res_coefs<double>(a.kap64 + b * a.es[0], n, a.ns[0], x, a.coef64 + b * (3 * a.ns[0] + a.es[0]));
  } else {
    const int z = x / (N1 * N1), r = x - z * N1 * N1, j = r / N1, i = r - j * N1;
    if (i > 0 && i < n && j > 0 && j < n && z > 0 && z < n) {
      const T* q = k + ((int64_t)(z - 1) * n + (j - 1)) * n + (i - 1);
      const int p = n * n;
      d = T(1.0 / n / 3.0) * (((q[0] + q[1]) + (q[n] + q[n + 1])) + ((q[p] + q[p + 1]) + (q[p + n] + q[p + n + 1])));
    }
  }
  a.w[l][b * a.ns[l] + x] = d != T(0) ? T(a.omega) / d : T(0);
}

}  // namespace

// Fills the geometry and the shared-memory layout of `a` for C CTAs per
// sample; returns the dynamic shared memory of a CTA.
template <class T>
static size_t resident_layout(int dim, int n, int K, int V, int C, ResArgs<T>& a, bool solve = true) {
  unsigned off = 0;
  auto take = [&](int64_t count, size_t size) {
    off = (off + 15u) / 16u * 16u;
    const unsigned o = off;
    off += (unsigned)(count * (int64_t)size);
    return o;
  };
  a.K = K;
  a.C = C;
  a.V = V;
  a.nv = V / C;
  a.Rv = K > 1 ? std::max(1, n / V) : (n - 1 + V - 1) / V;
  a.shv = 0;
  while ((1 << a.shv) < V) ++a.shv;
  a.nd = 0;
  int64_t band0 = 0;
  for (int l = 0; l < K; ++l) {
    ResLevel<T>& L = a.lv[l];
    L.n = n >> l;
    L.N1 = L.n + 1;
    L.S = dim == 2 ? L.N1 : L.N1 * L.N1;
    // a level is dealt to the CTAs while it has a slab for each and more than
    // a block's worth of work (2D above 16 rows, 3D above 4 planes)
    const bool split = C > 1 && a.nd == l && (l == 0 || (L.n >= C && L.n > (dim == 2 ? 16 : 4)));
    if (split) a.nd = l + 1;
    L.R = split ? (K > 1 ? std::max(1, L.n / C) : (a.nv * (n - 1) + V - 1) / V) : L.n - 1;
    L.sh = 0;
    while (K > 1 && (1 << (L.sh + 1)) <= L.R) ++L.sh;
    const uint64_t m = (uint64_t)std::max(1, L.n - 1), two32 = (uint64_t)1 << 32;
    L.m1 = (unsigned)((two32 + m - 1) / m);
    L.m2 = (unsigned)((two32 + m * m - 1) / (m * m));
    const double h = 1.0 / L.n;
    L.d0 = T(h / 3.0);
    L.d1 = T(h / 12.0);
    const int64_t band = (int64_t)L.R * L.S;
    if (l == 0) band0 = band;
    const bool last = K > 1 && l == K - 1;
    L.ob = last ? 0 : take(band, sizeof(T));
    L.oe = last ? 0 : take(band, sizeof(T));
    L.ot = K > 1 ? take(band, sizeof(T)) : 0;
  }
  a.oz = take(a.lv[0].S, sizeof(T));
  if (solve) {
    a.ox = take(band0, sizeof(T));
    a.op = take(band0, sizeof(T));
    a.ored = take(4 * 2 * RES_MAX_V, 8);
    a.osw = take((int64_t)(K > 1 ? 1 : 2) * a.nv * RES_THREADS, 8);
    a.osc = take(1, sizeof(ResScalars));
  }
  a.bytes = (off + 15u) / 16u * 16u;
  return a.bytes;
}

static size_t resident_bytes(int dim, int n, int K, int V, int C, bool mixed) {
  ResArgs<float> f{};
  ResArgs<double> d{};
  return mixed ? resident_layout(dim, n, K, V, C, f) : resident_layout(dim, n, K, V, C, d);
}

// Largest mesh (cells per side) whose solves run resident. The rule looks at the
// mesh alone, so that a sample's bits do not depend on its batch, and takes a
// mesh where 100 samples are no slower than on the separate kernels (one sample
// is 1.7 to 4 times as fast). ms resident / separate kernels:
//   2D FP64 GMG 128^2: 1 sample 0.68/1.19, 100 2.8/3.6, 256 7.0/7.2, 400 10.7/9.7, 1000 25.8/21.6
//   2D mixed GMG 128^2: 1 0.56/0.96, 100 1.3/1.9, 400 3.9/4.2, 1000 9.1/8.6
//   2D FP64 GMG 64^2: 1000 6.5/7.2, 4000 24.9/23.6; mixed: 4000 9.9/9.8
//   3D GMG 16^3: FP64 1000 12.4/15.6, mixed 3000 10.5/15.3; 32^3 mixed: 200 8.4/4.9
//   2D FP64 Jacobi: 150^2 100 50.5/60.4, 300 140/129; 170^2 100 79.2/82.5, 300 234/182; 179^2 100 91.4/89.7
//   2D mixed Jacobi: 200^2 300 147/155, 256^2 100 134/144, 300 372/333
//   3D FP64 Jacobi 24^3: 300 33.0/33.5; 32^3: 64 29.6/18.5
//   3D mixed Jacobi: 30^3 100 6.8/9.5, 300 19.9/20.8; 31^3 100 11.5/10.0, 32^3 12.3/9.8
// So on the largest meshes batches of several hundred samples and more take
// longer than they would on the separate kernels, up to 30%.
static int resident_cells(int dim, int K, bool mixed) {
  if (K > 1) return dim == 2 ? 128 : 16;
  return dim == 2 ? (mixed ? 256 : 170) : (mixed ? 30 : 24);
}

// Bands of the resident solve on a mesh of n cells per side with K multigrid
// levels (1: Jacobi), or 0 where it does not run: one per 512 interior nodes, at
// most a portable cluster. Jacobi, whose hundreds of iterations are one stencil
// and two sums each, goes on to 16 (one sample of 100^2 3.86 -> 2.93 ms, 20
// samples 5.49 -> 4.7); with multigrid the second band of a CTA cost large
// batches 5%.
int resident_bands(int dim, int n, int K, bool mixed) {
  if (n < 2 || K < 1 || K > RES_MAX_LEVELS || n > resident_cells(dim, K, mixed)) return 0;
  const int64_t in = ipow(n - 1, dim);
  int V = 1;
  while (V < RES_PORTABLE && in > (int64_t)V * RES_BAND && 2 * V <= n) V *= 2;
  if (K == 1 && V == RES_PORTABLE && in > (int64_t)V * RES_BAND && RES_MAX_V <= n) V = RES_MAX_V;
  return resident_bytes(dim, n, K, V, V, mixed) <= RES_SMEM_MAX ? V : 0;
}

// CTAs per sample for a batch: one per band while the batch leaves room on the
// SMs, else as few as keep RES_PER_SM CTAs on an SM (a CTA then takes several
// bands in turn, in the same order of sums).
static int resident_ctas(int dim, int n, int K, int V, bool mixed, int64_t B, int64_t slots) {
  int C = V;
  while (C > 1 && B * C > slots && resident_bytes(dim, n, K, V, C / 2, mixed) <= RES_SMEM_SHARE) C /= 2;
  return C;
}

template <int DIM, class T, bool MIXED>
static cudaError_t launch_res(cudaStream_t s, const ResArgs<T>& a, int64_t B) {
  static std::atomic<uint64_t> opted{0};
  cudaError_t e = once_per_device(opted, [] {
    const cudaError_t e1 = cudaFuncSetAttribute(k_resident<DIM, T, MIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)RES_SMEM_MAX);
    return e1 != cudaSuccess ? e1
                             : cudaFuncSetAttribute(k_resident<DIM, T, MIXED>,
                                                    cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(B * a.C), 1, 1);
  cfg.blockDim = dim3(RES_THREADS, 1, 1);
  cfg.dynamicSmemBytes = a.bytes;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)a.C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, k_resident<DIM, T, MIXED>, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// The two setup launches: kappa hierarchy, then weights and coefficients.
template <class T>
static cudaError_t launch_res_setup(cudaStream_t s, const ResidentSolve<T>& r, int64_t B, int* launches) {
  const int dim = r.g[0].dim;
  *launches = 0;
  if (r.K > 1 || r.round_kappa) {
    ResKappa<T> k{};
    k.K = r.K;
    k.dim = dim;
    for (int l = 0; l < r.K; ++l) {
      k.n[l] = r.g[l].n;
      k.es[l] = r.g[l].es;
      k.kap[l] = r.kap[l];
    }
    k.kap64 = r.round_kappa ? r.kap64 : nullptr;
    k_res_kappa<T><<<(unsigned)B, 512, 0, s>>>(k);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ++*launches;
  }
  ResCoefs<T> c{};
  c.kw = r.K > 1 ? r.K - 1 : 1;
  c.dim = dim;
  for (int l = 0; l < c.kw; ++l) {
    c.n[l] = r.g[l].n;
    c.off[l + 1] = c.off[l] + ipow(r.g[l].n + 1, dim);
    c.ns[l] = r.g[l].ns;
    c.es[l] = r.g[l].es;
    c.kap[l] = r.kap[l];
    c.w[l] = r.w[l];
    c.coef[l] = dim == 2 ? r.coef[l] : nullptr;
  }
  c.kap64 = r.kap64;
  c.coef64 = dim == 2 ? r.coef64 : nullptr;
  c.omega = r.omega;
  k_res_coefs<T><<<dim3((unsigned)((c.off[c.kw] + 255) / 256), (unsigned)B), 256, 0, s>>>(c);
  ++*launches;
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_resident(cudaStream_t s, const ResidentSolve<T>& r, int64_t B, int64_t slots, int* launches) {
  constexpr bool mixed = sizeof(T) == 4;
  if (B <= 0) return cudaSuccess;
  const int dim = r.g[0].dim, n = r.g[0].n;
  const int V = resident_bands(dim, n, r.K, mixed);
  if (V == 0) return cudaErrorInvalidValue;
  const bool limited = slots > 0;
  if (!limited) slots = RES_SLOTS;
  const int C = resident_ctas(dim, n, r.K, V, mixed, B, slots);
  cudaError_t e = launch_res_setup<T>(s, r, B, launches);
  if (e != cudaSuccess) return e;
  ResArgs<T> a{};
  if (resident_layout(dim, n, r.K, V, C, a) > RES_SMEM_MAX) return cudaErrorInvalidValue;
  for (int l = 0; l < r.K; ++l) {
    a.lv[l].ns = r.g[l].ns;
    a.lv[l].es = r.g[l].es;
    a.lv[l].kap = r.kap[l];
    a.lv[l].coef = r.coef[l];
    a.lv[l].w = r.w[l];
  }
  a.kap64 = r.kap64;
  a.coef64 = r.coef64;
  a.tol = r.tol;
  a.bval = dim == 2 ? r.g[0].h * r.g[0].h : r.g[0].h * r.g[0].h * r.g[0].h;
  a.max_iter = r.max_iter;
  a.inner_rtol = r.inner_rtol;
  a.scale0 = r.scale0;
  a.outer_max = r.outer_max;
  a.uc = r.uc;
  a.ucs = r.ucs;
  a.u = r.u;
  a.r = r.r;
  a.q = r.q;
  a.iters = r.iters;
  a.iters2 = r.iters2;
  a.box = r.box;
  a.L = r.L;
  a.H = r.H;
  a.qw = a.bval * r.inv_vol;
  ++*launches;
  a.B = B;
  const int64_t clusters = limited ? std::min(B, std::max<int64_t>(1, slots / C)) : B;
  return dim == 2 ? launch_res<2, T, mixed>(s, a, clusters) : launch_res<3, T, mixed>(s, a, clusters);
}
template cudaError_t launch_resident<double>(cudaStream_t, const ResidentSolve<double>&, int64_t, int64_t, int*);
template cudaError_t launch_resident<float>(cudaStream_t, const ResidentSolve<float>&, int64_t, int64_t, int*);

template <int DIM, class T>
static cudaError_t launch_bottom_dim(cudaStream_t s, const ResArgs<T>& a, const T* b, T* out, const int32_t* active,
                                     int cycles, int64_t B, Prof p) {
  static std::atomic<uint64_t> opted{0};
  cudaError_t e = once_per_device(opted, [] {
    return cudaFuncSetAttribute(k_bottom<DIM, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RES_SMEM_MAX);
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(B * a.C), 1, 1);
  cfg.blockDim = dim3(RES_THREADS, 1, 1);
  cfg.dynamicSmemBytes = a.bytes;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)a.C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, k_bottom<DIM, T>, a, b, out, active, cycles, p);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <class T>
cudaError_t launch_bottom(cudaStream_t s, const BottomLevels<T>& lv, const T* b, T* out, const int32_t* active,
                          int64_t B, Prof p) {
  const int dim = lv.g[0].dim, n = lv.g[0].n;
  if (lv.L < 2 || lv.L > RES_MAX_LEVELS || lv.g[lv.L - 1].n != 2) return cudaErrorInvalidValue;
  // as many CTAs per sample as the batch leaves room for (nothing is summed
  // over a sample here, so the result does not depend on it), at least as
  // many as its arrays need
  int C = 1;
  while (C < RES_PORTABLE && ipow(n - 1, dim) > (int64_t)C * RES_THREADS && 2 * C <= n) C *= 2;
  ResArgs<T> a{};
  while (C > 1 && B * C > RES_SLOTS && resident_layout(dim, n, lv.L, C / 2, C / 2, a, false) <= RES_SMEM_SHARE) C /= 2;
  if (resident_layout(dim, n, lv.L, C, C, a, false) > RES_SMEM_MAX) return cudaErrorInvalidValue;
  for (int l = 0; l < lv.L; ++l) {
    a.lv[l].ns = lv.g[l].ns;
    a.lv[l].es = lv.g[l].es;
    a.lv[l].kap = lv.kap[l];
    a.lv[l].coef = lv.coef[l];
    a.lv[l].w = lv.w[l];
  }
  return dim == 2 ? launch_bottom_dim<2, T>(s, a, b, out, active, lv.cycles, B, p)
                  : launch_bottom_dim<3, T>(s, a, b, out, active, lv.cycles, B, p);
}
template cudaError_t launch_bottom<double>(cudaStream_t, const BottomLevels<double>&, const double*, double*,
                                           const int32_t*, int64_t, Prof);
template cudaError_t launch_bottom<float>(cudaStream_t, const BottomLevels<float>&, const float*, float*,
                                          const int32_t*, int64_t, Prof);
}  // namespace mlmc
