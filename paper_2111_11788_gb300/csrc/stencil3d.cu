// 3D matrix-free Q1 operator, PCG and geometric multigrid kernels,
// templated on the value type.
//
// Operator (Eq. (model), Sec. 2.1, trilinear Q1, kappa constant per element,
// homogeneous Dirichlet). The reference element matrix has the entries
// h/3 (diagonal), 0 (vertices differing in one coordinate), -h/12 (two or
// three coordinates). Node c = (x, y, z) is shared by the 8 elements
// (x-1+a, y-1+b, z-1+c'), a, b, c' in {0, 1}; a neighbour at offset
// d in {-1, 0, 1}^3 shares the elements whose index bit is 1 where d = +1,
// 0 where d = -1 and free where d = 0. Hence the row of A at c has
//   diagonal              h/3 * (sum of the 8 kappa)
//   12 edge neighbours    -h/12 * (sum of the 2 shared kappa)
//   8 corner neighbours   -h/12 * (the 1 shared kappa)
// and no face coupling.
//
// Stencil kernels march along z: a CTA owns a 32 x 16 tile of node columns
// and a chunk of zc planes; a thread owns two rows of one column. Each step
// stages one plane of the input field (with a one-node halo) and one layer
// of kappa (with a one-element halo) in shared memory, double buffered,
// while the next plane is fetched into registers. A plane p feeds three
// outputs of a column: p - 1 (the 8 couplings across layer p - 1, after
// which output p - 1 is complete and goes to the epilogue), p (the centre
// and its 4 in-plane diagonal edge neighbours) and p + 1 (the 8 couplings
// across layer p). So a node costs about one coalesced load of the field and
// of kappa, a few shared-memory reads and one store, instead of 27 + 8
// cached global loads. The field a stencil acts on is formed by a loader
// while its plane is staged (z + beta p for A p, omega D^-1 b for the
// multigrid residual), so those need no pointwise pre-pass. In FP32 the two
// rows of a thread are 8 apart and stored as pairs, so the stencil runs on
// paired FP32 instructions (or, on 32..256 cells per side, on full-width
// tiles staged by TMA bulk copies, k_zm3w). In FP64, where the plan has the
// per-node kappa sums of the level, the same march runs on element sums
// (k_zm3q: about 19 instead of 33 FP64 operations per node). The remaining pointwise kernels run one thread
// per node column of a 32 x 8 tile over 8 z-planes on grids of 64 and more
// cells per side, else over one (the prolongation: one thread per fine
// x-pair over 8 planes); the initialisation and the QoI run
// one CTA per z-plane. Node arrays carry the boundary nodes (always 0).
// Partials: one per CTA (g.tiles_s per sample for the stencil kernels,
// g.tiles_q = N1 for the QoI). The multigrid levels of at most
// 16^3 cells below the finest run as one kernel per V-cycle (resident.cu,
// k_bottom).
#include "guess.cuh"
#include "mlmc_internal.cuh"

#include <type_traits>

namespace mlmc {
namespace {

constexpr int BX = 32, BY = 8;

struct Node3 {
  int i, j, k;
  bool valid, interior;
  int64_t idx;  // (k * N1 + j) * N1 + i
};


// Node tiles with a z-loop: CTA (zg, tile) covers the 32 x 8 node tile in
// planes zg * pz .. zg * pz + pz - 1 (one thread per column, pz planes
// each), so a pointwise kernel on a large grid runs few, large CTAs
// (pz = NODE_PZ) and one on a small grid keeps one plane per thread
// (node_pz).
constexpr int NODE_PZ = 8;
inline int node_pz(int n) { return n >= 64 ? NODE_PZ : 1; }
struct NodeCol {
  int i, j, k0, k1;   // column (i, j), planes [k0, k1)
  bool valid;         // the column lies in the mesh
};
__device__ __forceinline__ NodeCol node_col3(int n, int pz) {
  const int N1 = n + 1;
  const int tx = (N1 + BX - 1) / BX, ty = (N1 + BY - 1) / BY;
  const int tiles = tx * ty;
  const int zg = blockIdx.x / tiles;
  const int t = blockIdx.x - zg * tiles;
  const int ty_ = t / tx;
  NodeCol c;
  c.i = (t - ty_ * tx) * BX + threadIdx.x;
  c.j = ty_ * BY + threadIdx.y;
  c.k0 = zg * pz;
  c.k1 = min(c.k0 + pz, N1);
  c.valid = c.i <= n && c.j <= n;
  return c;
}
inline unsigned node_col3_blocks(int n, int pz) {
  const int N1 = n + 1;
  return (unsigned)(((N1 + BX - 1) / BX) * ((N1 + BY - 1) / BY) * ((N1 + pz - 1) / pz));
}

template <class T>
__device__ __forceinline__ T warp_sum3(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Sum of the CTA (256 threads) into part[b * tiles + blockIdx.x].
__device__ __forceinline__ void cta_partial3(double v, double* __restrict__ part, int64_t tiles) {
  __shared__ double s_w[BY];
  v = warp_sum3(v);
  if (threadIdx.x == 0) s_w[threadIdx.y] = v;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    double r = 0.0;
#pragma unroll
    for (int w = 0; w < BY; ++w) r += s_w[w];
    part[(int64_t)blockIdx.y * tiles + blockIdx.x] = r;
  }
}

__device__ __forceinline__ void prof_tick3(const Prof& p) {
  if (p.acc && blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) atomicAdd(p.acc, p.per_sample);
}

// kappa of the 8 elements around interior node q: kk[c'][b][a].
template <class T>
__device__ __forceinline__ void load_k8(const T* __restrict__ K, int n, const Node3& q, T kk[2][2][2]) {
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const T* r = K + ((int64_t)(q.k - 1 + c) * n + (q.j - 1 + b)) * n + (q.i - 1);
      kk[c][b][0] = __ldg(r);
      kk[c][b][1] = __ldg(r + 1);
    }
}

template <class T>
__device__ __forceinline__ T diag3(const T kk[2][2][2], double c3) {
  const T s = ((kk[0][0][0] + kk[0][0][1]) + (kk[0][1][0] + kk[0][1][1])) +
              ((kk[1][0][0] + kk[1][0][1]) + (kk[1][1][0] + kk[1][1][1]));
  return T(c3) * s;
}

// ---------------------------------------------------------------- z-march

constexpr int ZTX = 32, ZTY = 16;          // node columns per CTA (x, y)
constexpr int ZRY = 2;                     // y-rows per thread
constexpr int ZTHREADS = ZTX * (ZTY / ZRY);
constexpr int ZSX = ZTX + 2, ZSY = ZTY + 2, ZNV = ZSX * ZSY;   // vector plane + halo
constexpr int ZKX = ZTX + 1, ZKY = ZTY + 1, ZNK = ZKX * ZKY;   // kappa layer + halo
constexpr int ZSLOTS = ((ZNV > ZNK ? ZNV : ZNK) + ZTHREADS - 1) / ZTHREADS;
static_assert(ZNV <= ZSLOTS * ZTHREADS && ZNK <= ZSLOTS * ZTHREADS, "staging slots per thread");
static_assert(ZTHREADS == BX * BY, "the z-march CTA has the node-tile thread count");

struct ZTile {
  int tx0, ty0, z0, z1;   // column origin; output planes [z0, z1)
};

__device__ __forceinline__ ZTile ztile(const Grid& g) {
  const int txn = (g.n + ZTX - 1) / ZTX, tyn = (g.n + ZTY - 1) / ZTY;
  int t = blockIdx.x;
  const int zq = t / (txn * tyn);
  t -= zq * txn * tyn;
  const int ty = t / txn;
  ZTile z;
  z.tx0 = (t - ty * txn) * ZTX;
  z.ty0 = ty * ZTY;
  z.z0 = zq * g.zc;
  z.z1 = min(z.z0 + g.zc, g.n + 1);
  return z;
}

// Generic z-marching stencil kernel: y = A(kappa) x at every node of the
// CTA's columns and planes, handed to the epilogue with the centre value of
// x; the epilogue's returned values are summed (in T per thread, in FP64
// across the CTA) into one partial per CTA (part may be null). A thread owns
// two adjacent y-rows of one x-column. The epilogue's own inputs for a node
// are fetched one plane ahead (Epi::Pre). Tiles cover node columns
// [0, 32 ceil(n/32)) x [0, 16 ceil(n/16)); when n is a multiple of the tile
// width, the column n (boundary) is written by the thread of column n - 1
// (epi.zero). Offsets inside one sample fit 32 bits ((n + 1)^3 < 2^31).
template <class T, class Ld, class Epi>
__global__ void __launch_bounds__(ZTHREADS, 2) k_zm3(Grid g, const T* __restrict__ Kap, Ld ld,
                                                  const int32_t* __restrict__ active, Epi epi,
                                                  double* __restrict__ part, Prof prof) {
  const int64_t b = blockIdx.y;
  if (active && !active[b]) return;
  __shared__ T sv[2][ZNV];
  __shared__ T sk[2][ZNK];
  const ZTile t = ztile(g);
  const int n = g.n, N1 = n + 1, P = N1 * N1, KP = n * n;
  const int tid = threadIdx.y * ZTX + threadIdx.x;
  const T* __restrict__ kp = Kap + b * g.es;
  ld.bind(b);
  epi.bind(b);
  // staging slots: plane entries tid + q * ZTHREADS, with their in-plane
  // offsets and whether they lie inside (interior nodes for x, whose
  // boundary values are ignored; mesh elements for kappa)
  int vo[ZSLOTS], ko[ZSLOTS];
  bool vok[ZSLOTS], kok[ZSLOTS], vin[ZSLOTS], kin[ZSLOTS];
#pragma unroll
  for (int q = 0; q < ZSLOTS; ++q) {
    const int sidx = tid + q * ZTHREADS;
    vin[q] = sidx < ZNV;
    kin[q] = sidx < ZNK;
    const int vx = t.tx0 - 1 + sidx % ZSX, vy = t.ty0 - 1 + sidx / ZSX;
    vok[q] = vin[q] && vx >= 1 && vx < n && vy >= 1 && vy < n;
    vo[q] = vok[q] ? vy * N1 + vx : 0;
    const int kx = t.tx0 - 1 + sidx % ZKX, ky = t.ty0 - 1 + sidx / ZKX;
    kok[q] = kin[q] && kx >= 0 && kx < n && ky >= 0 && ky < n;
    ko[q] = kok[q] ? ky * n + kx : 0;
  }
  T rv[ZSLOTS], rk[ZSLOTS];
  auto fetch = [&](int pp) {
    const bool pv = pp >= 1 && pp < n, pk = pp >= 0 && pp < n;
#pragma unroll
    for (int q = 0; q < ZSLOTS; ++q) {
      rv[q] = (pv && vok[q]) ? ld(pp * P + vo[q]) : T(0);
      rk[q] = (pk && kok[q]) ? __ldg(kp + pp * KP + ko[q]) : T(0);
    }
  };
  int p = t.z0 - 1;
  fetch(p);

  const int i = t.tx0 + threadIdx.x;
  const int j0 = t.ty0 + ZRY * threadIdx.y;
  bool cvalid[ZRY], cint[ZRY], ey[ZRY];
  int ocol[ZRY];
#pragma unroll
  for (int r = 0; r < ZRY; ++r) {
    const int j = j0 + r;
    cvalid[r] = i <= n && j <= n;
    cint[r] = i >= 1 && i < n && j >= 1 && j < n;
    ey[r] = j == n - 1 && n % ZTY == 0;
    ocol[r] = j * N1 + i;
  }
  const bool ex = i == n - 1 && n % ZTX == 0;
  const T c3 = T(g.c3), c12 = T(g.c12);
  // Per output row: U = unscaled coupling sum and D = (sum of the 8 kappa) x
  // centre of the output of plane p - 1 so far, N = the couplings of the
  // output of plane p with plane p - 1; output = c3 D - c12 U. Pair sums of a
  // kappa layer (X: along x per element row, Y: along y per column, S: the 4
  // elements around an output row) are formed once per layer and reused by
  // both rows and by the next plane; every coupling is one FMA into U.
  T U[ZRY], D[ZRY], N[ZRY], vc[ZRY];
  typename Epi::Pre pre[ZRY];    // epilogue inputs of plane p - 1
#pragma unroll
  for (int r = 0; r < ZRY; ++r) U[r] = D[r] = N[r] = vc[r] = T(0);
  T kb[ZRY + 1][2];              // kappa layer p - 1, element rows j0 - 1 .. j0 + ZRY - 1
  T Xb[ZRY + 1], Yb[ZRY][2], Sb[ZRY];
#pragma unroll
  for (int r = 0; r <= ZRY; ++r) kb[r][0] = kb[r][1] = Xb[r] = T(0);
#pragma unroll
  for (int r = 0; r < ZRY; ++r) Yb[r][0] = Yb[r][1] = Sb[r] = T(0);
  T dot = T(0);
  const int vbase = (ZRY * threadIdx.y + 1) * ZSX + threadIdx.x + 1;
  const int kbase = ZRY * threadIdx.y * ZKX + threadIdx.x;
  int buf = 0;
  for (; p <= t.z1; ++p) {
    T* svb = sv[buf];
    T* skb = sk[buf];
#pragma unroll
    for (int q = 0; q < ZSLOTS; ++q) {
      if (vin[q]) svb[tid + q * ZTHREADS] = rv[q];
      if (kin[q]) skb[tid + q * ZTHREADS] = rk[q];
    }
    __syncthreads();
    if (p < t.z1) fetch(p + 1);   // the next plane is in flight while this one is used
    typename Epi::Pre nxt[ZRY];
#pragma unroll
    for (int r = 0; r < ZRY; ++r)
      if (cint[r] && p >= t.z0 && p < t.z1 && p >= 1 && p < n) nxt[r] = epi.load(p * P + ocol[r]);
    T v[ZRY + 2][3], ka[ZRY + 1][2];
#pragma unroll
    for (int r = 0; r < ZRY + 2; ++r)
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) v[r][dx] = svb[vbase + (r - 1) * ZSX + (dx - 1)];
#pragma unroll
    for (int r = 0; r <= ZRY; ++r)
#pragma unroll
      for (int a = 0; a < 2; ++a) ka[r][a] = skb[kbase + r * ZKX + a];
    T Xa[ZRY + 1], Ya[ZRY][2], Sa[ZRY];
#pragma unroll
    for (int r = 0; r <= ZRY; ++r) Xa[r] = ka[r][0] + ka[r][1];
#pragma unroll
    for (int r = 0; r < ZRY; ++r) {
      Ya[r][0] = ka[r][0] + ka[r + 1][0];
      Ya[r][1] = ka[r][1] + ka[r + 1][1];
      Sa[r] = Xa[r] + Xa[r + 1];
    }
    const int m = p - 1;
#pragma unroll
    for (int r = 0; r < ZRY; ++r) {
      const T* v0 = v[r];
      const T* v1 = v[r + 1];
      const T* v2 = v[r + 2];
      // couplings of output p - 1 with plane p across layer p - 1: complete
      T u = U[r];
      u = fma(Yb[r][0], v1[0], u);
      u = fma(Yb[r][1], v1[2], u);
      u = fma(Xb[r], v0[1], u);
      u = fma(Xb[r + 1], v2[1], u);
      u = fma(kb[r][0], v0[0], u);
      u = fma(kb[r][1], v0[2], u);
      u = fma(kb[r + 1][0], v2[0], u);
      u = fma(kb[r + 1][1], v2[2], u);
      // A x = c3 D - c12 U, or f - A x = f - c3 D + c12 U for a residual epilogue
      T done;
      if constexpr (Epi::kRes) done = fma(c12, u, fma(-c3, D[r], T(epi.rhs(pre[r]))));
      else done = fma(-c12, u, c3 * D[r]);
      if (cvalid[r] && m >= t.z0) {
        const int o = m * P + ocol[r];
        dot += epi(o, cint[r] && m >= 1 && m < n, done, vc[r], pre[r]);
        if (ex) epi.zero(o + 1);
        if (ey[r]) epi.zero(o + N1);
        if (ex && ey[r]) epi.zero(o + N1 + 1);
      }
      // output p: couplings with plane p - 1 (N) and the in-plane diagonal
      // edges (free axis z: one kappa of each layer), and the diagonal part
      u = N[r];
      u = fma(kb[r][0] + ka[r][0], v0[0], u);
      u = fma(kb[r][1] + ka[r][1], v0[2], u);
      u = fma(kb[r + 1][0] + ka[r + 1][0], v2[0], u);
      u = fma(kb[r + 1][1] + ka[r + 1][1], v2[2], u);
      U[r] = u;
      D[r] = (Sb[r] + Sa[r]) * v1[1];
      // output p + 1: couplings with plane p across layer p
      u = Ya[r][0] * v1[0];
      u = fma(Ya[r][1], v1[2], u);
      u = fma(Xa[r], v0[1], u);
      u = fma(Xa[r + 1], v2[1], u);
      u = fma(ka[r][0], v0[0], u);
      u = fma(ka[r][1], v0[2], u);
      u = fma(ka[r + 1][0], v2[0], u);
      N[r] = fma(ka[r + 1][1], v2[2], u);
      vc[r] = v1[1];
      pre[r] = nxt[r];
    }
#pragma unroll
    for (int r = 0; r <= ZRY; ++r) {
      kb[r][0] = ka[r][0];
      kb[r][1] = ka[r][1];
      Xb[r] = Xa[r];
    }
#pragma unroll
    for (int r = 0; r < ZRY; ++r) {
      Yb[r][0] = Ya[r][0];
      Yb[r][1] = Ya[r][1];
      Sb[r] = Sa[r];
    }
    buf ^= 1;
  }
  if (part) cta_partial3((double)dot, part, g.tiles_s);
  prof_tick3(prof);
}

// FP64 z-march on precomputed kappa sums (k_zm3q). With K_n the sum of the 8
// kappa around node n and K_{n,n+d} the sum of the 4 elements sharing the
// edge (n, n+d), the Q1 row of node n (element stiffness h/12 (4, 0, -1,
// -1) by the number of differing coordinates, Sec. 5.1 of the FE setting)
// is
//   (A u)_n = h/12 [5 u_n K_n - sum_{e ni n} kappa_e S_e + sum_{6 d} u_{n+d} K_{n,n+d}],
// S_e the sum of u over the 8 nodes of element e. Per plane p a CTA forms,
// for every element position of its tile (33 x 17 with the halo), the sum
// of u over the element's 4 nodes in plane p (PXY), and Q = kappa * S for
// the layer below plane p (S = PXY(p) + PXY(p - 1)), once per element, in
// shared memory; a node takes the 2 x 2 sums of Q of the two layers around
// it (B, one carried from the plane before) and its 6 face neighbours
// weighted by the edge sums. About 17.5 FP64 operations per node instead of
// the 33 of k_zm3 (the kernel is bound by the FP64 pipe; the 4 node arrays
// of kappa sums, [5 K_n | K_x | K_y | K_z] per sample, are computed once per
// solve by k_ksum3). Same tiles, chunks, loaders, epilogues and boundary
// rule as k_zm3.
template <class Ld, class Epi>
__global__ void __launch_bounds__(ZTHREADS, 2) k_zm3q(Grid g, const double* __restrict__ Kap,
                                                   const double* __restrict__ Ks, int64_t kss, Ld ld,
                                                   const int32_t* __restrict__ active, Epi epi,
                                                   double* __restrict__ part, Prof prof) {
  const int64_t b = blockIdx.y;
  if (active && !active[b]) return;
  __shared__ double sv[3][ZNV];   // field planes with halo (p, p - 1, and the one being refilled)
  __shared__ double sk[2][ZNK];   // kappa layers with halo
  __shared__ double sp[2][ZNK];   // PXY of the plane, per element position
  __shared__ double sq[ZNK];      // Q of the layer below the current plane
  const ZTile t = ztile(g);
  const int n = g.n, N1 = n + 1, P = N1 * N1, KP = n * n;
  const int tid = threadIdx.y * ZTX + threadIdx.x;
  const double* __restrict__ kp = Kap + b * g.es;
  const double* __restrict__ Kn = Ks + b * kss;
  const double* __restrict__ Kx = Kn + g.ns;
  const double* __restrict__ Ky = Kn + 2 * g.ns;
  const double* __restrict__ Kz = Kn + 3 * g.ns;
  ld.bind(b);
  epi.bind(b);
  for (int e = tid; e < ZNK; e += ZTHREADS) sp[1][e] = sk[1][e] = 0.0;
  for (int e = tid; e < ZNV; e += ZTHREADS) sv[2][e] = 0.0;
  int vo[ZSLOTS], ko[ZSLOTS];
  bool vok[ZSLOTS], kok[ZSLOTS], vin[ZSLOTS], kin[ZSLOTS];
#pragma unroll
  for (int q = 0; q < ZSLOTS; ++q) {
    const int sidx = tid + q * ZTHREADS;
    vin[q] = sidx < ZNV;
    kin[q] = sidx < ZNK;
    const int vx = t.tx0 - 1 + sidx % ZSX, vy = t.ty0 - 1 + sidx / ZSX;
    vok[q] = vin[q] && vx >= 1 && vx < n && vy >= 1 && vy < n;
    vo[q] = vok[q] ? vy * N1 + vx : 0;
    const int kx = t.tx0 - 1 + sidx % ZKX, ky = t.ty0 - 1 + sidx / ZKX;
    kok[q] = kin[q] && kx >= 0 && kx < n && ky >= 0 && ky < n;
    ko[q] = kok[q] ? ky * n + kx : 0;
  }
  double rv[ZSLOTS], rk[ZSLOTS];
  auto fetch = [&](int pp) {
    const bool pv = pp >= 1 && pp < n, pk = pp >= 0 && pp < n;
#pragma unroll
    for (int q = 0; q < ZSLOTS; ++q) {
      rv[q] = (pv && vok[q]) ? ld(pp * P + vo[q]) : 0.0;
      rk[q] = (pk && kok[q]) ? __ldg(kp + pp * KP + ko[q]) : 0.0;
    }
  };
  int p = t.z0 - 1;
  fetch(p);

  const int i = t.tx0 + threadIdx.x;
  const int j0 = t.ty0 + ZRY * threadIdx.y;
  bool cvalid[ZRY], cint[ZRY], ey[ZRY];
  int ocol[ZRY];
#pragma unroll
  for (int r = 0; r < ZRY; ++r) {
    const int j = j0 + r;
    cvalid[r] = i <= n && j <= n;
    cint[r] = i >= 1 && i < n && j >= 1 && j < n;
    ey[r] = j == n - 1 && n % ZTY == 0;
    ocol[r] = j * N1 + i;
  }
  const bool ex = i == n - 1 && n % ZTX == 0;
  const double h12 = g.c12;   // h / 12
  // per output row: B of the layer below the current output plane, the
  // centre u and K_z of the plane below it, the kappa sums of the output
  // plane (5 K_n, K_x(i), K_x(i - 1), K_y(j), K_y(j - 1), K_z) loaded a plane
  // ahead, and the epilogue inputs
  double Bprev[ZRY], ucar[ZRY], kzcar[ZRY], ks[ZRY][6];
  typename Epi::Pre pre[ZRY];
#pragma unroll
  for (int r = 0; r < ZRY; ++r) {
    Bprev[r] = ucar[r] = kzcar[r] = 0.0;
#pragma unroll
    for (int c = 0; c < 6; ++c) ks[r][c] = 0.0;
  }
  double dot = 0.0;
  const int vbase = (ZRY * threadIdx.y + 1) * ZSX + threadIdx.x + 1;   // node (i, j0)
  const int kbase = ZRY * threadIdx.y * ZKX + threadIdx.x;             // element (i - 1, j0 - 1)
  // sv: plane p in sv[cur], plane p - 1 in sv[prv]; a buffer is refilled
  // two steps after its last read, with the barriers of a step between
  int buf = 0, cur = 0, prv = 2;
  for (; p <= t.z1; ++p) {
    double* svb = sv[cur];
    double* skb = sk[buf];
#pragma unroll
    for (int q = 0; q < ZSLOTS; ++q) {
      if (vin[q]) svb[tid + q * ZTHREADS] = rv[q];
      if (kin[q]) skb[tid + q * ZTHREADS] = rk[q];
    }
    __syncthreads();   // plane p and kappa layer p staged
    if (p < t.z1) fetch(p + 1);
    // kappa sums and epilogue inputs of plane p (an output plane at the next step)
    typename Epi::Pre nxt[ZRY];
    double kn[ZRY][6];
#pragma unroll
    for (int r = 0; r < ZRY; ++r) {
      const bool out = cint[r] && p >= 1 && p < n;
      if (out && p >= t.z0 && p < t.z1) nxt[r] = epi.load(p * P + ocol[r]);
      const int o = p * P + ocol[r];
      kn[r][0] = out ? __ldg(Kn + o) : 0.0;
      kn[r][1] = out ? __ldg(Kx + o) : 0.0;
      kn[r][2] = out ? __ldg(Kx + o - 1) : 0.0;
      kn[r][3] = out ? __ldg(Ky + o) : 0.0;
      kn[r][4] = out ? __ldg(Ky + o - N1) : 0.0;
      kn[r][5] = (cint[r] && p >= 0 && p < n) ? __ldg(Kz + o) : 0.0;
    }
    // element sums of plane p and Q of layer p - 1, once per element position
    const double* svo = sv[prv];
    for (int e = tid; e < ZNK; e += ZTHREADS) {
      const int ex_ = e % ZKX, ey_ = e / ZKX;
      const double* v = svb + ey_ * ZSX + ex_;
      const double pxy = (v[0] + v[1]) + (v[ZSX] + v[ZSX + 1]);
      sq[e] = sk[buf ^ 1][e] * (pxy + sp[buf ^ 1][e]);
      sp[buf][e] = pxy;
    }
    __syncthreads();   // Q of layer p - 1 complete
    const int m = p - 1;
    // Q x-pair sums of the element rows j0 - 1 .. j0 + ZRY - 1 at columns i - 1, i
    double qx[ZRY + 1];
#pragma unroll
    for (int r = 0; r <= ZRY; ++r) qx[r] = sq[kbase + r * ZKX] + sq[kbase + r * ZKX + 1];
#pragma unroll
    for (int r = 0; r < ZRY; ++r) {
      const double Bcur = qx[r] + qx[r + 1];
      const double* v = svo + vbase + r * ZSX;   // node (i, j0 + r) of plane m
      const double uc = v[0];
      if (cvalid[r] && m >= t.z0) {
        const int o = m * P + ocol[r];
        const bool in = cint[r] && m >= 1 && m < n;
        double acc = 0.0;
        if (in) {
          // - sum kappa_e S_e, the six face neighbours by their edge sums, 5 u K_n
          double sx = fma(ks[r][1], v[1], -(Bprev[r] + Bcur));
          sx = fma(ks[r][2], v[-1], sx);
          sx = fma(ks[r][3], v[ZSX], sx);
          sx = fma(ks[r][4], v[-ZSX], sx);
          sx = fma(ks[r][5], svb[vbase + r * ZSX], sx);
          sx = fma(kzcar[r], ucar[r], sx);
          acc = fma(uc, ks[r][0], sx);
        }
        double done;
        if constexpr (Epi::kRes) done = fma(-h12, acc, epi.rhs(pre[r]));
        else done = h12 * acc;
        dot += epi(o, in, done, uc, pre[r]);
        if (ex) epi.zero(o + 1);
        if (ey[r]) epi.zero(o + N1);
        if (ex && ey[r]) epi.zero(o + N1 + 1);
      }
      Bprev[r] = Bcur;
      ucar[r] = uc;
      kzcar[r] = ks[r][5];
#pragma unroll
      for (int c = 0; c < 6; ++c) ks[r][c] = kn[r][c];
      pre[r] = nxt[r];
    }
    buf ^= 1;
    prv = cur;
    cur = cur == 2 ? 0 : cur + 1;
  }
  if (part) cta_partial3(dot, part, g.tiles_s);
  prof_tick3(prof);
}

// Kappa sums of every node (0 outside the mesh), per sample [5 K_n | K_x | K_y
// | K_z] in node strides: K_n the 8 elements around the node, K_x the 4
// elements sharing the edge to the +x neighbour (element column i, rows j-1
// and j, layers k-1 and k), K_y and K_z likewise. Once per solve and level. With
// W also the smoother weights omega / D, D = h/3 K_n (the same values as
// k_winv3's, without a second pass that sums the 8 elements again: 6 samples of
// 128^3 644 -> 477 us, bound by the FP64 pipe, the division most of it).
__global__ void __launch_bounds__(256) k_ksum3(Grid g, const double* __restrict__ K, double* __restrict__ Ks,
                                               int64_t kss, int pz, double omega, double* __restrict__ W) {
  const int64_t b = blockIdx.y;
  const NodeCol c = node_col3(g.n, pz);
  if (!c.valid) return;
  const int n = g.n, N1 = n + 1;
  const double* k = K + b * g.es;
  double* kn = Ks + b * kss;
  auto el = [&](int z, int y, int x) -> double {
    return (z >= 0 && z < n && y >= 0 && y < n && x >= 0 && x < n) ? __ldg(k + ((int64_t)z * n + y) * n + x) : 0.0;
  };
  // per element layer z, around this node column: L = the 4 elements, X =
  // the 2 elements of row j (x-pair, for K_y), Y = the 2 of column i
  // (y-pair, for K_x); a node adds the sums of the layers below and above
  auto layer = [&](int z, double& L, double& X, double& Y) {
    const double a = el(z, c.j - 1, c.i - 1), bq = el(z, c.j - 1, c.i);
    const double cq = el(z, c.j, c.i - 1), d = el(z, c.j, c.i);
    X = cq + d;
    Y = bq + d;
    L = (a + bq) + X;
  };
  double L0, X0, Y0;
  layer(c.k0 - 1, L0, X0, Y0);
  for (int kz = c.k0; kz < c.k1; ++kz) {
    double L1, X1, Y1;
    layer(kz, L1, X1, Y1);
    const int64_t o = ((int64_t)kz * N1 + c.j) * N1 + c.i;
    kn[o] = 5.0 * (L0 + L1);
    kn[g.ns + o] = Y0 + Y1;
    kn[2 * g.ns + o] = X0 + X1;
    kn[3 * g.ns + o] = L1;
    if (W) {
      const bool in = c.i > 0 && c.i < n && c.j > 0 && c.j < n && kz > 0 && kz < n;
      W[b * g.ns + o] = in ? omega / (g.c3 * (L0 + L1)) : 0.0;
    }
    L0 = L1;
    X0 = X1;
    Y0 = Y1;
  }
}

// Loaders: the value the stencil acts on at an interior node, formed while
// the plane is staged (bind(sample) offsets the arrays to the sample), so a
// pointwise pre-pass is not needed.
template <class T>
struct LdX {   // x
  const T* x;
  int64_t ns;
  __device__ void bind(int64_t b) { x += b * ns; }
  __device__ T operator()(int o) const { return __ldg(x + o); }
};

template <class T>
struct LdPupd {   // the new CG direction z + beta p (beta == 0: z)
  const T* z;
  const T* pold;
  const double* beta;
  int64_t ns;
  T bb;
  __device__ void bind(int64_t b) {
    z += b * ns;
    pold += b * ns;
    bb = (T)beta[b];
  }
  __device__ T operator()(int o) const {
    const T zv = __ldg(z + o);
    return bb == T(0) ? zv : fma(bb, __ldg(pold + o), zv);
  }
};

template <class T>
struct LdWb {   // the pre-smoothed iterate from zero: omega D^-1 b
  const T* W;
  const T* Bv;
  int64_t ns;
  __device__ void bind(int64_t b) {
    W += b * ns;
    Bv += b * ns;
  }
  __device__ T operator()(int o) const { return __ldg(W + o) * __ldg(Bv + o); }
};

// Epilogues: bind(sample) offsets their arrays to the sample; load(node)
// fetches the node's own inputs (Pre) one plane ahead; then (node offset,
// interior?, y, x at the node, Pre) -> contribution to the CTA partial;
// zero() writes a boundary node. y is (A x) at the node, or, for an epilogue
// with kRes (the FP64 residual forms, k_zm3 only), f - (A x) with f =
// rhs(Pre): the FP64 kernel then folds f into its last two FMAs instead of a
// multiply, an FMA and a subtraction.
struct NoPre {};


template <class T>
struct EpiApply {   // y = A x
  using Pre = NoPre;
  static constexpr bool kRes = false;
  __device__ T rhs(const Pre&) const { return T(0); }
  T* Y;
  int64_t ns;
  __device__ void bind(int64_t b) { Y += b * ns; }
  __device__ Pre load(int) const { return Pre{}; }
  __device__ T operator()(int o, bool in, T ax, T, const Pre&) const {
    Y[o] = in ? ax : T(0);
    return T(0);
  }
  __device__ void zero(int o) const { Y[o] = T(0); }
};

template <class T>
struct EpiAq {   // q = A p, partial of p.q; p itself stored (Pn) when formed by the loader
  using Pre = NoPre;
  static constexpr bool kRes = false;
  __device__ T rhs(const Pre&) const { return T(0); }
  T* Q;
  T* Pn;
  int64_t ns;
  __device__ void bind(int64_t b) {
    Q += b * ns;
    if (Pn) Pn += b * ns;
  }
  __device__ Pre load(int) const { return Pre{}; }
  __device__ T operator()(int o, bool in, T ax, T xc, const Pre&) const {
    const T qv = in ? ax : T(0);
    Q[o] = qv;
    if (Pn) Pn[o] = in ? xc : T(0);
    return xc * qv;
  }
  __device__ void zero(int o) const {
    Q[o] = T(0);
    if (Pn) Pn[o] = T(0);
  }
};

template <class T>
struct PreB {
  T b;
};

template <class T>
struct EpiMgRes {   // residual of the pre-smoothed iterate: b - A e; e stored (E) when formed by the loader
  using Pre = PreB<T>;
  static constexpr bool kRes = sizeof(T) == 8;
  __device__ T rhs(const Pre& pr) const { return pr.b; }
  const T* Bv;
  T* R1;
  T* E;
  int64_t ns;
  __device__ void bind(int64_t b) {
    Bv += b * ns;
    R1 += b * ns;
    if (E) E += b * ns;
  }
  __device__ Pre load(int o) const { return Pre{__ldg(Bv + o)}; }
  __device__ T operator()(int o, bool in, T y, T xc, const Pre& pr) const {
    R1[o] = in ? (kRes ? y : pr.b - y) : T(0);
    if (E) E[o] = in ? xc : T(0);
    return T(0);
  }
  __device__ void zero(int o) const {
    R1[o] = T(0);
    if (E) E[o] = T(0);
  }
};

template <class T>
struct PreBW {
  T b, w;
};

template <class T>
struct EpiMgPost {   // post-smoothing: e + W (b - A e), partial of b.out
  using Pre = PreBW<T>;
  static constexpr bool kRes = sizeof(T) == 8;
  __device__ T rhs(const Pre& pr) const { return pr.b; }
  const T* W;
  const T* Bv;
  T* Out;
  int64_t ns;
  __device__ void bind(int64_t b) {
    W += b * ns;
    Bv += b * ns;
    Out += b * ns;
  }
  __device__ Pre load(int o) const { return Pre{__ldg(Bv + o), __ldg(W + o)}; }
  __device__ T operator()(int o, bool in, T y, T ec, const Pre& pr) const {
    const T ov = in ? fma(pr.w, kRes ? y : pr.b - y, ec) : T(0);
    Out[o] = ov;
    return in ? pr.b * ov : T(0);
  }
  __device__ void zero(int o) const { Out[o] = T(0); }
};

struct EpiResid {   // outer FP64 residual h^3 - A u, partial of its square
  using Pre = NoPre;
  static constexpr bool kRes = true;
  double* R;
  int64_t ns;
  double h3;
  __device__ double rhs(const Pre&) const { return h3; }
  __device__ void bind(int64_t b) { R += b * ns; }
  __device__ Pre load(int) const { return Pre{}; }
  __device__ double operator()(int o, bool in, double rv_in, double, const Pre&) const {
    const double rv = in ? rv_in : 0.0;
    R[o] = rv;
    return rv * rv;
  }
  __device__ void zero(int o) const { R[o] = 0.0; }
};

// ------------------------------------------------ FP32 z-march, packed pairs
//
// The FP32 form of k_zm3 on Blackwell's paired FP32 instructions (FFMA2 and
// friends, __ffma2_rn / __fadd2_rn / __fmul2_rn): a thread owns rows j and
// j + 8 of one column of the 32 x 16 tile, and shared memory holds each
// staged plane as pairs (value at row r, value at row r + 8), so one 64-bit
// shared load brings the same neighbour of both outputs and every stencil
// operation serves both. Same tile, chunks, boundary rule and epilogues as
// k_zm3.
constexpr int ZPY = ZTY / 2 + 2, ZNVP = ZSX * ZPY;   // 34 x 10 pairs
constexpr int ZKPY = ZTY / 2 + 1, ZNKP = ZKX * ZKPY; // 33 x 9 pairs
static_assert(ZNVP <= 2 * ZTHREADS && ZNKP <= 2 * ZTHREADS, "two paired staging slots per thread");

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Asynchronous 4-byte global -> shared copy to a shared-window address
// (zero-filled when src_bytes = 0).
__device__ __forceinline__ void cp_async4s(unsigned sa, const void* gmem, int src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sa), "l"(gmem), "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

constexpr int ZSTAGES = 4;   // planes in flight: the current one and ZSTAGES - 1 ahead

// Paired FP32 loaders for k_zm3f: kArrays node arrays are staged per plane
// and combined pairwise into the field once the plane has arrived.
struct LdXf {   // x
  static constexpr int kArrays = 1;
  static constexpr bool kCoarse = false;
  const float* a0;
  int64_t ns;
  __device__ void bind(int64_t b) { a0 += b * ns; }
  __device__ const float* src(int) const { return a0; }
  __device__ float2 combine(float2 x, float2) const { return x; }
  __device__ float combine1(float x, float) const { return x; }
  bool aligned16() const { return ((uintptr_t)a0 & 15) == 0; }
};

struct LdPupdf {   // z + beta p (beta == 0: z)
  static constexpr int kArrays = 2;
  static constexpr bool kCoarse = false;
  const float* z;
  const float* pold;
  const double* beta;
  int64_t ns;
  float bb;
  __device__ void bind(int64_t b) {
    z += b * ns;
    pold += b * ns;
    bb = (float)beta[b];
  }
  __device__ const float* src(int k) const { return k ? pold : z; }
  __device__ float2 combine(float2 zv, float2 pv) const {
    return bb == 0.0f ? zv : fma2(make_float2(bb, bb), pv, zv);
  }
  __device__ float combine1(float zv, float pv) const { return bb == 0.0f ? zv : fmaf(bb, pv, zv); }
  bool aligned16() const { return (((uintptr_t)z | (uintptr_t)pold) & 15) == 0; }
};

struct LdWbf {   // omega D^-1 b
  static constexpr int kArrays = 2;
  static constexpr bool kCoarse = false;
  const float* W;
  const float* Bv;
  int64_t ns;
  __device__ void bind(int64_t b) {
    W += b * ns;
    Bv += b * ns;
  }
  __device__ const float* src(int k) const { return k ? Bv : W; }
  __device__ float2 combine(float2 w, float2 bv) const { return mul2(w, bv); }
  __device__ float combine1(float w, float bv) const { return w * bv; }
  bool aligned16() const { return (((uintptr_t)W | (uintptr_t)Bv) & 15) == 0; }
};

// The corrected iterate omega D^-1 b + P e_c (k_zm3n only): W and b are staged
// and the pre-smoothed iterate formed from them again, P e_c added from coarse
// rows kept in shared memory. Neither the iterate nor its sum with the
// correction is stored by a pass of its own.
struct LdPostf {
  static constexpr int kArrays = 2;
  static constexpr bool kCoarse = true;
  const float* W;
  const float* Bv;
  const float* ec;
  int64_t ns, nsc;
  __device__ void bind(int64_t b) {
    W += b * ns;
    Bv += b * ns;
    ec += b * nsc;
  }
  __device__ const float* src(int k) const { return k ? Bv : W; }
};

template <class Ld>
struct LdPaired;
template <>
struct LdPaired<LdX<float>> {
  using type = LdXf;
  static LdXf make(const LdX<float>& l) { return LdXf{l.x, l.ns}; }
};
template <>
struct LdPaired<LdPupd<float>> {
  using type = LdPupdf;
  static LdPupdf make(const LdPupd<float>& l) { return LdPupdf{l.z, l.pold, l.beta, l.ns, 0.0f}; }
};
template <>
struct LdPaired<LdWb<float>> {
  using type = LdWbf;
  static LdWbf make(const LdWb<float>& l) { return LdWbf{l.W, l.Bv, l.ns}; }
};

template <class Ld, class Epi>
__global__ void __launch_bounds__(ZTHREADS, 2) k_zm3f(Grid g, const float* __restrict__ Kap, Ld ld,
                                                      const int32_t* __restrict__ active, Epi epi,
                                                      double* __restrict__ part, Prof prof) {
  static_assert(!Epi::kRes, "the FP32 z-march hands A x to its epilogues");
  constexpr int NA = Ld::kArrays;
  const int64_t b = blockIdx.y;
  if (active && !active[b]) return;
  __shared__ __align__(16) float2 sv[ZSTAGES][NA][ZNVP];
  __shared__ __align__(16) float2 sk[ZSTAGES][ZNKP];
  const ZTile t = ztile(g);
  const int n = g.n, N1 = n + 1, P = N1 * N1, KP = n * n;
  const int tid = threadIdx.y * ZTX + threadIdx.x;
  const float* __restrict__ kp = Kap + b * g.es;
  ld.bind(b);
  epi.bind(b);
  // copy slots: pair entries tid and tid + 256; entry (xx, yy) holds rows
  // r = ty0 - 1 + yy and r + 8 of column tx0 - 1 + xx
  int vo[2][2], ko[2][2];
  bool vok[2][2], kok[2][2], vin[2], kin[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int e = tid + q * ZTHREADS;
    vin[q] = e < ZNVP;
    kin[q] = e < ZNKP;
    const int vx = t.tx0 - 1 + e % ZSX, vy = t.ty0 - 1 + e / ZSX;
    const int kx = t.tx0 - 1 + e % ZKX, ky = t.ty0 - 1 + e / ZKX;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int ry = vy + 8 * h, rk = ky + 8 * h;
      vok[q][h] = vin[q] && vx >= 1 && vx < n && ry >= 1 && ry < n;
      vo[q][h] = vok[q][h] ? ry * N1 + vx : 0;
      kok[q][h] = kin[q] && kx >= 0 && kx < n && rk >= 0 && rk < n;
      ko[q][h] = kok[q][h] ? rk * n + kx : 0;
    }
  }
  // stage plane pp into ring slot st (one commit group per plane; empty
  // groups past the chunk keep the group count uniform)
  // shared addresses of this thread's copy slots in ring slot 0 (slot st is
  // st * stage bytes further); global reads of masked slots point at a plane
  // inside the sample and copy 0 bytes
  const unsigned sv0 = (unsigned)__cvta_generic_to_shared(&sv[0][0][0]);
  const unsigned sk0 = (unsigned)__cvta_generic_to_shared(&sk[0][0]);
  constexpr unsigned SV_ARR = ZNVP * 8, SV_STAGE = NA * ZNVP * 8, SK_STAGE = ZNKP * 8;
  auto issue = [&](int pp, int st) {
    if (pp <= t.z1) {
      const bool pv = pp >= 1 && pp < n, pk = pp >= 0 && pp < n;
      const int pc = min(max(pp, 0), n - 1);
      const unsigned svs = sv0 + st * SV_STAGE, sks = sk0 + st * SK_STAGE;
      const float* kpl = kp + pc * KP;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const unsigned e8 = (unsigned)(tid + q * ZTHREADS) * 8u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (vin[q]) {
#pragma unroll
            for (int a = 0; a < NA; ++a)
              cp_async4s(svs + a * SV_ARR + e8 + 4u * h, ld.src(a) + pc * P + vo[q][h],
                         (pv && vok[q][h]) ? 4 : 0);
          }
          if (kin[q]) cp_async4s(sks + e8 + 4u * h, kpl + ko[q][h], (pk && kok[q][h]) ? 4 : 0);
        }
      }
    }
    cp_async_commit();
  };
  int p = t.z0 - 1;
#pragma unroll
  for (int j = 0; j < ZSTAGES - 1; ++j) issue(p + j, j);

  const int i = t.tx0 + threadIdx.x;
  const int jr[2] = {t.ty0 + (int)threadIdx.y, t.ty0 + (int)threadIdx.y + 8};
  bool cvalid[2], cint[2], ey[2];
  int ocol[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    cvalid[r] = i <= n && jr[r] <= n;
    cint[r] = i >= 1 && i < n && jr[r] >= 1 && jr[r] < n;
    ey[r] = jr[r] == n - 1 && n % ZTY == 0;
    ocol[r] = jr[r] * N1 + i;
  }
  const bool ex = i == n - 1 && n % ZTX == 0;
  const float c3s = (float)g.c3, c12s = (float)g.c12;
  const float2 c3 = make_float2(c3s, c3s), mc12 = make_float2(-c12s, -c12s);
  // as in k_zm3: U unscaled couplings and D diagonal part of the output of
  // plane p - 1, N couplings of the output of plane p with plane p - 1; the
  // kappa pair sums of a layer (X along x, Y along y, S of the 4 elements)
  // are formed once and reused for the next plane
  const float2 z2 = make_float2(0.f, 0.f);
  float2 U = z2, D = z2, Nn = z2, vc = z2;
  float2 kb[2][2] = {{z2, z2}, {z2, z2}};
  float2 Xb[2] = {z2, z2}, Yb[2] = {z2, z2}, Sb = z2;
  typename Epi::Pre pre[2];
  float dot = 0.0f;
  const int vbase = (threadIdx.y + 1) * ZSX + threadIdx.x + 1;
  const int kbase = threadIdx.y * ZKX + threadIdx.x;
  int st = 0;
  for (; p <= t.z1; ++p) {
    cp_async_wait<ZSTAGES - 2>();   // this thread's copies of plane p have landed
    if (NA > 1) {                   // combine this thread's entries into the field
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (vin[q]) {
          const int e = tid + q * ZTHREADS;
          sv[st][0][e] = ld.combine(sv[st][0][e], sv[st][NA - 1][e]);
        }
    }
    __syncthreads();                // plane p complete; slot of plane p - 1 free
    issue(p + ZSTAGES - 1, (st + ZSTAGES - 1) % ZSTAGES);
    typename Epi::Pre nxt[2];
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (cint[r] && p >= t.z0 && p < t.z1 && p >= 1 && p < n) nxt[r] = epi.load(p * P + ocol[r]);
    const float2* svb = sv[st][0];
    const float2* skb = sk[st];
    float2 v[3][3], ka[2][2];
#pragma unroll
    for (int dy = 0; dy < 3; ++dy)
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) v[dy][dx] = svb[vbase + (dy - 1) * ZSX + (dx - 1)];
#pragma unroll
    for (int bq = 0; bq < 2; ++bq)
#pragma unroll
      for (int a = 0; a < 2; ++a) ka[bq][a] = skb[kbase + bq * ZKX + a];
    float2 Xa[2], Ya[2];
    Xa[0] = add2(ka[0][0], ka[0][1]);
    Xa[1] = add2(ka[1][0], ka[1][1]);
    Ya[0] = add2(ka[0][0], ka[1][0]);
    Ya[1] = add2(ka[0][1], ka[1][1]);
    const float2 Sa = add2(Xa[0], Xa[1]);
    // outputs of plane p - 1 are complete: couplings with plane p across layer p - 1
    float2 u = fma2(Yb[0], v[1][0], U);
    u = fma2(Yb[1], v[1][2], u);
    u = fma2(Xb[0], v[0][1], u);
    u = fma2(Xb[1], v[2][1], u);
    u = fma2(kb[0][0], v[0][0], u);
    u = fma2(kb[0][1], v[0][2], u);
    u = fma2(kb[1][0], v[2][0], u);
    u = fma2(kb[1][1], v[2][2], u);
    const float2 done = fma2(mc12, u, mul2(c3, D));
    const int m = p - 1;
    if (m >= t.z0) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (!cvalid[r]) continue;
        const int o = m * P + ocol[r];
        dot += epi(o, cint[r] && m >= 1 && m < n, r ? done.y : done.x, r ? vc.y : vc.x, pre[r]);
        if (ex) epi.zero(o + 1);
        if (ey[r]) epi.zero(o + N1);
        if (ex && ey[r]) epi.zero(o + N1 + 1);
      }
    }
    // output p: couplings with plane p - 1 and the in-plane diagonal edges
    u = fma2(add2(kb[0][0], ka[0][0]), v[0][0], Nn);
    u = fma2(add2(kb[0][1], ka[0][1]), v[0][2], u);
    u = fma2(add2(kb[1][0], ka[1][0]), v[2][0], u);
    U = fma2(add2(kb[1][1], ka[1][1]), v[2][2], u);
    D = mul2(add2(Sb, Sa), v[1][1]);
    // output p + 1: couplings with plane p across layer p
    u = mul2(Ya[0], v[1][0]);
    u = fma2(Ya[1], v[1][2], u);
    u = fma2(Xa[0], v[0][1], u);
    u = fma2(Xa[1], v[2][1], u);
    u = fma2(ka[0][0], v[0][0], u);
    u = fma2(ka[0][1], v[0][2], u);
    u = fma2(ka[1][0], v[2][0], u);
    Nn = fma2(ka[1][1], v[2][2], u);
#pragma unroll
    for (int bq = 0; bq < 2; ++bq)
#pragma unroll
      for (int a = 0; a < 2; ++a) kb[bq][a] = ka[bq][a];
    Xb[0] = Xa[0];
    Xb[1] = Xa[1];
    Yb[0] = Ya[0];
    Yb[1] = Ya[1];
    Sb = Sa;
    vc = v[1][1];
    pre[0] = nxt[0];
    pre[1] = nxt[1];
    st = (st + 1) % ZSTAGES;
  }
  cp_async_wait<0>();
  if (part) cta_partial3((double)dot, part, g.tiles_s);
  prof_tick3(prof);
}

// ------------------------------------ FP32 z-march, TMA bulk-copy staging
//
// k_zm3w is k_zm3f with its planes staged by the copy engine instead of by
// per-element cp.async, for the meshes with n in {32, 64, 128, 256}: a CTA
// covers the full width of the mesh (n threads across x, one column each)
// and R = 256 RT / n node rows, RT = 2 rows per thread (the CTAs per sample
// are those of the 32 x 16 tiles; k_zm3n takes four rows per thread and half
// as many CTAs), so the halo slab of a plane (rows ty0 - 1 ..
// ty0 + R, every column) is one contiguous range of a node array; the kappa
// slab (rows ty0 - 1 .. ty0 + R - 1) is one contiguous range of an element
// array. Each plane of each array is then ONE asynchronous bulk copy
// (cp.async.bulk, global -> shared, completing on the slot's mbarrier),
// issued by one thread: no per-element address, predicate or register work.
// Node rows have an odd pitch n + 1, so a slab starts sh = (offset mod 4)
// floats past a 16-byte boundary; the copy starts at that boundary and lands
// at a slot offset that keeps the destination 16-byte aligned, which shifts
// the slab by OFF (0..3 floats, one value per plane) inside the slot.
// Values that feed only boundary outputs (row -1, column -1, the kappa halo
// and the layers -1 and n) may be stale; planes 0 and n are not copied, and
// the boundary nodes of the field (rows, columns and planes 0 and n) are
// read as 0 by the threads next to them, whatever the array holds there.
// A thread's two rows are one float2 pair. Waits are
// bounded: a wait that gives up counts a timeout in g_zt_timeouts (read by
// the host at its sync points), lets the copies still in flight land
// (bounded again) and ends the CTA.
constexpr int ZW_S = 4;                             // ring slots, ZW_S - 1 planes in flight
constexpr int ZW_WAIT_TRIES = 1 << 22;              // bounded waits: tries and SM cycles (~2 s)
constexpr long long ZW_WAIT_CYCLES = 1ll << 32;

// rows per CTA and slot sizes (floats) of a node slab and of a kappa slab
// for cells per side n and rows per thread rt
__host__ __device__ constexpr int zw_rows(int n, int rt) { return 256 * rt / n; }
__host__ __device__ constexpr int zw_vslot(int n, int rt) {
  return (12 + (zw_rows(n, rt) + 2) * (n + 1) + 3) / 4 * 4;
}
__host__ __device__ constexpr int zw_kslot(int n, int rt) { return (8 + (zw_rows(n, rt) + 1) * n + 3) / 4 * 4; }
inline bool zw_mesh(int n) { return n == 32 || n == 64 || n == 128 || n == 256; }

__device__ unsigned int g_zt_timeouts;

__device__ __forceinline__ void mbar_init(unsigned addr, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(addr), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(unsigned addr, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(addr), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned addr, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(addr), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait for the completion of phase `parity`; false if it gave up.
__device__ __forceinline__ bool mbar_wait(unsigned addr, unsigned parity) {
  if (mbar_try_wait(addr, parity)) return true;
  const long long t0 = clock64();
  for (int k = 0; k < ZW_WAIT_TRIES; ++k) {
    if (mbar_try_wait(addr, parity)) return true;
    if (clock64() - t0 > ZW_WAIT_CYCLES) break;
  }
  return false;
}
__device__ __forceinline__ void bulk_g2s(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}

template <class Ld, class Epi>
__global__ void __launch_bounds__(ZTHREADS, 3) k_zm3w(Grid g, const float* __restrict__ Kap, Ld ld,
                                                                   const int32_t* __restrict__ active, Epi epi,
                                                                   double* __restrict__ part, Prof prof) {
  static_assert(!Epi::kRes, "the FP32 z-march hands A x to its epilogues");
  constexpr int NA = Ld::kArrays;
  constexpr int RT = 2, NP = 1;   // rows and float2 row pairs per thread
  const int64_t b = blockIdx.y;
  if (active && !active[b]) return;
  extern __shared__ __align__(16) float zw_smem[];
  const int n = g.n, N1 = n + 1, P = N1 * N1, KPn = n * n;
  const int R = zw_rows(n, RT), VS = zw_vslot(n, RT), KS = zw_kslot(n, RT), SS = NA * VS + KS;
  float* ring = zw_smem;                                              // ZW_S slots of SS floats
  unsigned long long* sbar = reinterpret_cast<unsigned long long*>(zw_smem + ZW_S * SS);
  __shared__ double s_w[ZTHREADS / 32];
  const int tyn = n / R;
  int t = blockIdx.x;
  const int zq = t / tyn;
  const int ty0 = (t - zq * tyn) * R;
  const int z0 = zq * g.zc, z1 = min(z0 + g.zc, n + 1);
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  const float* __restrict__ kp = Kap + b * g.es;
  ld.bind(b);
  epi.bind(b);
  for (int e = tid; e < ZW_S * SS / 4; e += ZTHREADS)
    reinterpret_cast<float4*>(ring)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  const unsigned bar0 = (unsigned)__cvta_generic_to_shared(sbar);
  const unsigned ring0 = (unsigned)__cvta_generic_to_shared(ring);
  if (tid == 0) {
#pragma unroll
    for (int s = 0; s < ZW_S; ++s) mbar_init(bar0 + 8u * s, 1u);
    fence_mbar_init();
  }
  fence_proxy_async_smem();
  __syncthreads();

  // slabs: node rows ylo..yhi of a plane, kappa rows kylo..ty0 + R - 1 of a layer
  const int ylo = max(ty0 - 1, 0), yhi = min(ty0 + R, n), r0 = ylo - ty0 + 1;
  const int kylo = max(ty0 - 1, 0), kr0 = kylo - ty0 + 1;
  const unsigned kbytes = 4u * (unsigned)((ty0 + R - kylo) * n);
  // shift of plane pp's slab inside its slot (the slab's 16-byte alignment)
  auto voff = [&](int pp) {
    const int sh = (pp * P + ylo * N1) & 3;
    return (sh - r0 * N1) & 3;
  };
  // stage plane pp (field) and layer pp (kappa) into slot st: one bulk copy per array
  auto issue = [&](int pp, int st) {
    if (tid != 0) return;
    const bool pv = pp >= 1 && pp < n, pk = pp >= 0 && pp < n;
    const unsigned bar = bar0 + 8u * st;
    const int G0 = pp * P + ylo * N1, G1 = pp * P + (yhi + 1) * N1;
    const int Ga = G0 & ~3, Gb = (G1 + 3) & ~3;
    const unsigned vbytes = 4u * (unsigned)(Gb - Ga);
    mbar_arrive_tx(bar, (pv ? NA * vbytes : 0u) + (pk ? kbytes : 0u));
    if (pv) {
      const int dst = 4 + voff(pp) + r0 * N1 - (G0 - Ga);
#pragma unroll
      for (int a = 0; a < NA; ++a)
        bulk_g2s(ring0 + 4u * (unsigned)(st * SS + a * VS + dst), ld.src(a) + Ga, vbytes, bar);
    }
    if (pk)
      bulk_g2s(ring0 + 4u * (unsigned)(st * SS + NA * VS + 4 + kr0 * n), kp + (pp * KPn + kylo * n), kbytes,
               bar);
  };

  int p = z0 - 1;
  unsigned pend = 0;   // slots with copies issued and not yet waited for
#pragma unroll
  for (int j = 0; j < ZW_S - 1; ++j)
    if (p + j <= z1) {
      issue(p + j, j);
      pend |= 1u << j;
    }

  const int i = threadIdx.x;
  const int jr0 = ty0 + RT * (int)threadIdx.y;   // this thread's rows jr0 .. jr0 + RT - 1
  bool cint[RT], ey[RT];
  int ocol[RT];
#pragma unroll
  for (int r = 0; r < RT; ++r) {
    cint[r] = i >= 1 && i < n && jr0 + r >= 1 && jr0 + r < n;
    ey[r] = jr0 + r == n - 1;
    ocol[r] = (jr0 + r) * N1 + i;
  }
  const bool ex = i == n - 1;
  // field boundary nodes next to this thread's stencils (columns i - 1 .. i + 1,
  // rows jr0 - 1 .. jr0 + RT) read as 0
  bool cok[3], rok[RT + 2];
#pragma unroll
  for (int dx = 0; dx < 3; ++dx) cok[dx] = i - 1 + dx >= 1 && i - 1 + dx <= n - 1;
#pragma unroll
  for (int r = 0; r < RT + 2; ++r) rok[r] = jr0 - 1 + r >= 1 && jr0 - 1 + r <= n - 1;
  const bool edge = !(cok[0] && cok[2] && rok[0] && rok[RT + 1]);
  const float c3s = (float)g.c3, c12s = (float)g.c12;
  const float2 c3 = make_float2(c3s, c3s), mc12 = make_float2(-c12s, -c12s);
  const float2 z2 = make_float2(0.f, 0.f);
  // per row pair q (rows jr0 + 2q, jr0 + 2q + 1), as in k_zm3f: U unscaled
  // couplings and D diagonal part of the output of plane p - 1, N couplings
  // of the output of plane p with plane p - 1, the kappa pair sums of the
  // layer below (X along x, Y along y, S of the 4 elements)
  float2 U[NP], D[NP], Nn[NP], vc[NP], kb[NP][2][2], Xb[NP][2], Yb[NP][2], Sb[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    U[q] = D[q] = Nn[q] = vc[q] = Sb[q] = z2;
    kb[q][0][0] = kb[q][0][1] = kb[q][1][0] = kb[q][1][1] = z2;
    Xb[q][0] = Xb[q][1] = Yb[q][0] = Yb[q][1] = z2;
  }
  typename Epi::Pre pre[RT];
  float dot = 0.0f;
  const int vrow = 4 + RT * (int)threadIdx.y * N1 + i - 1;    // + OFF: row jr0 - 1, column i - 1
  const int krow = 4 + RT * (int)threadIdx.y * n + i - 1;     // row jr0 - 1, element i - 1
  int st = 0;
  unsigned par = 0;    // phase parity of each slot's next completion
  bool timed_out = false;
#pragma unroll 2
  for (; p <= z1; ++p) {
    const bool landed = mbar_wait(bar0 + 8u * st, (par >> st) & 1u);
    if (landed) {
      pend &= ~(1u << st);
      par ^= 1u << st;
    }
    float* slot = ring + st * SS;
    if (NA > 1 && landed && p >= 1 && p < n) {   // combine the arrays into the field
      for (int e = tid; e < VS; e += ZTHREADS) slot[e] = ld.combine1(slot[e], slot[VS + e]);
    }
    fence_proxy_async_smem();       // this thread's shared-memory writes before later copies
    // plane p complete; the slot of plane p - 1 is free (or a wait gave up:
    // every thread leaves the loop together)
    if (__syncthreads_or(!landed)) {
      timed_out = true;
      break;
    }
    if (p + ZW_S - 1 <= z1) {
      const int sn = (st + ZW_S - 1) % ZW_S;
      issue(p + ZW_S - 1, sn);
      pend |= 1u << sn;
    }
    typename Epi::Pre nxt[RT];
#pragma unroll
    for (int r = 0; r < RT; ++r)
      if (cint[r] && p >= z0 && p < z1 && p >= 1 && p < n) nxt[r] = epi.load(p * P + ocol[r]);
    const float* svb = slot + voff(p) + vrow;
    const float* skb = slot + NA * VS + krow;
    float sv[RT + 2][3], kv[RT + 1][2];
#pragma unroll
    for (int r = 0; r < RT + 2; ++r)
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) sv[r][dx] = svb[r * N1 + dx];
#pragma unroll
    for (int r = 0; r < RT + 1; ++r)
#pragma unroll
      for (int a = 0; a < 2; ++a) kv[r][a] = skb[r * n + a];
    if (p <= 0 || p >= n) {
#pragma unroll
      for (int r = 0; r < RT + 2; ++r)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) sv[r][dx] = 0.f;
    } else if (edge) {
#pragma unroll
      for (int r = 0; r < RT + 2; ++r)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx)
          if (!rok[r] || !cok[dx]) sv[r][dx] = 0.f;
    }
    const int m = p - 1;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      float2 v[3][3], ka[2][2];
#pragma unroll
      for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) v[dy][dx] = make_float2(sv[2 * q + dy][dx], sv[2 * q + dy + 1][dx]);
#pragma unroll
      for (int bq = 0; bq < 2; ++bq)
#pragma unroll
        for (int a = 0; a < 2; ++a) ka[bq][a] = make_float2(kv[2 * q + bq][a], kv[2 * q + bq + 1][a]);
      float2 Xa[2], Ya[2];
      Xa[0] = add2(ka[0][0], ka[0][1]);
      Xa[1] = add2(ka[1][0], ka[1][1]);
      Ya[0] = add2(ka[0][0], ka[1][0]);
      Ya[1] = add2(ka[0][1], ka[1][1]);
      const float2 Sa = add2(Xa[0], Xa[1]);
      // outputs of plane p - 1 are complete: couplings with plane p across layer p - 1
      float2 u = fma2(Yb[q][0], v[1][0], U[q]);
      u = fma2(Yb[q][1], v[1][2], u);
      u = fma2(Xb[q][0], v[0][1], u);
      u = fma2(Xb[q][1], v[2][1], u);
      u = fma2(kb[q][0][0], v[0][0], u);
      u = fma2(kb[q][0][1], v[0][2], u);
      u = fma2(kb[q][1][0], v[2][0], u);
      u = fma2(kb[q][1][1], v[2][2], u);
      const float2 done = fma2(mc12, u, mul2(c3, D[q]));
      if (m >= z0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = 2 * q + h;
          const int o = m * P + ocol[r];
          dot += epi(o, cint[r] && m >= 1 && m < n, h ? done.y : done.x, h ? vc[q].y : vc[q].x, pre[r]);
          if (ex) epi.zero(o + 1);
          if (ey[r]) epi.zero(o + N1);
          if (ex && ey[r]) epi.zero(o + N1 + 1);
        }
      }
      // output p: couplings with plane p - 1 and the in-plane diagonal edges
      u = fma2(add2(kb[q][0][0], ka[0][0]), v[0][0], Nn[q]);
      u = fma2(add2(kb[q][0][1], ka[0][1]), v[0][2], u);
      u = fma2(add2(kb[q][1][0], ka[1][0]), v[2][0], u);
      U[q] = fma2(add2(kb[q][1][1], ka[1][1]), v[2][2], u);
      D[q] = mul2(add2(Sb[q], Sa), v[1][1]);
      // output p + 1: couplings with plane p across layer p
      u = mul2(Ya[0], v[1][0]);
      u = fma2(Ya[1], v[1][2], u);
      u = fma2(Xa[0], v[0][1], u);
      u = fma2(Xa[1], v[2][1], u);
      u = fma2(ka[0][0], v[0][0], u);
      u = fma2(ka[0][1], v[0][2], u);
      u = fma2(ka[1][0], v[2][0], u);
      Nn[q] = fma2(ka[1][1], v[2][2], u);
#pragma unroll
      for (int bq = 0; bq < 2; ++bq)
#pragma unroll
        for (int a = 0; a < 2; ++a) kb[q][bq][a] = ka[bq][a];
      Xb[q][0] = Xa[0];
      Xb[q][1] = Xa[1];
      Yb[q][0] = Ya[0];
      Yb[q][1] = Ya[1];
      Sb[q] = Sa;
      vc[q] = v[1][1];
    }
#pragma unroll
    for (int r = 0; r < RT; ++r) pre[r] = nxt[r];
    st = (st + 1) % ZW_S;
  }
  if (timed_out) {
    // record the timeout, let the copies still in flight land (bounded), end the CTA
    if (tid == 0) atomicAdd(&g_zt_timeouts, 1u);
    for (int s2 = 0; s2 < ZW_S; ++s2)
      if (pend & (1u << s2)) mbar_wait(bar0 + 8u * s2, (par >> s2) & 1u);
    return;
  }
  if (part) {
    double v = warp_sum3((double)dot);
    if ((tid & 31) == 0) s_w[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
      double r = 0.0;
#pragma unroll
      for (int w = 0; w < ZTHREADS / 32; ++w) r += s_w[w];
      part[(int64_t)blockIdx.y * g.tiles_s + blockIdx.x] = r;
    }
  }
  prof_tick3(prof);
}

// k_zm3n: the z-march of k_zm3w with four rows per thread and the mesh's width a
// compile-time constant, so that every shared-memory and node offset inside a
// plane is an immediate. Bound by instruction issue: the form with a run-time
// width spent 109 warp instructions per 32 nodes on the FP32 operator (63% of
// the issue slots, 159 us for 16 samples of 128^3), 33 of which are its
// arithmetic. What else changed: the two rows of a pair are 2 apart (rows
// jr0 + q and jr0 + q + 2 of output pair q), so the pairs of one output pair
// serve the other's neighbours and need no register moves; boundary values of
// a field that may be nonzero there are cleared in shared memory once per
// plane by the few threads next to the barrier instead of being selected
// away by every thread; the slab's shift is carried (a plane has an odd number
// of nodes, N1^2 = 1 mod 4: one float further each plane); the epilogue's own
// inputs are read without a test, boundary nodes included. 109 us then, 55% of
// the copy bandwidth (registers allow two CTAs per SM).
template <int N, class Ld, class Epi>
__global__ void __launch_bounds__(ZTHREADS, 2) k_zm3n(Grid g, const float* __restrict__ Kap, Ld ld,
                                                      const int32_t* __restrict__ active, Epi epi,
                                                      double* __restrict__ part, Prof prof) {
  static_assert(!Epi::kRes, "the FP32 z-march hands A x to its epilogues");
  constexpr int NA = Ld::kArrays, RT = 4;
  constexpr int N1 = N + 1, P = N1 * N1, KPn = N * N;
  constexpr int R = zw_rows(N, RT), VS = zw_vslot(N, RT), KS = zw_kslot(N, RT), SS = NA * VS + KS;
  static_assert((P & 3) == 1, "the slab's shift grows by one float a plane");
  const int64_t b = blockIdx.y;
  if (active && !active[b]) return;
  extern __shared__ __align__(16) float zw_smem[];
  float* ring = zw_smem;                                              // ZW_S slots of SS floats
  unsigned long long* sbar = reinterpret_cast<unsigned long long*>(zw_smem + ZW_S * SS);
  __shared__ double s_w[ZTHREADS / 32];
  // P e_c: the coarse rows under a slab, interpolated along z to plane p, in
  // scz[p & 1] (rows J0 .. J0 + CR - 1 of CC nodes)
  constexpr int C1 = N / 2 + 1, CR = R / 2 + 2, CE = Ld::kCoarse ? CR * C1 : 1;
  constexpr int CPT = (CE + ZTHREADS - 1) / ZTHREADS;
  float* scz = reinterpret_cast<float*>(sbar + ZW_S);
  constexpr int tyn = N / R;
  const int zq = blockIdx.x / tyn;
  const int ty0 = (blockIdx.x - zq * tyn) * R;
  const int z0 = zq * g.zc, z1 = min(z0 + g.zc, N1);
  const int i = threadIdx.x, tid = threadIdx.y * N + i;
  const float* __restrict__ kp_ = Kap + b * g.es;
  ld.bind(b);
  epi.bind(b);
  for (int e = tid; e < ZW_S * SS / 4; e += ZTHREADS)
    reinterpret_cast<float4*>(ring)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  const unsigned bar0 = (unsigned)__cvta_generic_to_shared(sbar);
  const unsigned ring0 = (unsigned)__cvta_generic_to_shared(ring);
  if (tid == 0) {
#pragma unroll
    for (int s = 0; s < ZW_S; ++s) mbar_init(bar0 + 8u * s, 1u);
    fence_mbar_init();
  }
  fence_proxy_async_smem();
  __syncthreads();

  // slabs: node rows ylo..yhi of a plane, kappa rows kylo..ty0 + R - 1 of a layer
  const int ylo = max(ty0 - 1, 0), yhi = min(ty0 + R, N), r0 = ylo - ty0 + 1;
  const int kylo = max(ty0 - 1, 0), kr0 = kylo - ty0 + 1;
  const unsigned kbytes = 4u * (unsigned)((ty0 + R - kylo) * N);
  auto voff = [&](int pp) { return ((pp * P + ylo * N1) - r0 * N1) & 3; };
  // stage plane pp (field) and layer pp (kappa) into slot st: one bulk copy per array
  auto issue = [&](int pp, int st) {
    if (tid != 0) return;
    const bool pv = pp >= 1 && pp < N, pk = pp >= 0 && pp < N;
    const unsigned bar = bar0 + 8u * st;
    const int G0 = pp * P + ylo * N1, G1 = pp * P + (yhi + 1) * N1;
    const int Ga = G0 & ~3, Gb = (G1 + 3) & ~3;
    const unsigned vbytes = 4u * (unsigned)(Gb - Ga);
    mbar_arrive_tx(bar, (pv ? NA * vbytes : 0u) + (pk ? kbytes : 0u));
    if (pv) {
      const int dst = 4 + voff(pp) + r0 * N1 - (G0 - Ga);
#pragma unroll
      for (int a = 0; a < NA; ++a)
        bulk_g2s(ring0 + 4u * (unsigned)(st * SS + a * VS + dst), ld.src(a) + Ga, vbytes, bar);
    }
    if (pk)
      bulk_g2s(ring0 + 4u * (unsigned)(st * SS + NA * VS + 4 + kr0 * N), kp_ + (pp * KPn + kylo * N), kbytes, bar);
  };

  int p = z0 - 1;
  unsigned pend = 0;   // slots with copies issued and not yet waited for
#pragma unroll
  for (int j = 0; j < ZW_S - 1; ++j)
    if (p + j <= z1) {
      issue(p + j, j);
      pend |= 1u << j;
    }

  float cn[CPT];   // this thread's entries of the next plane's coarse rows
  const int J0 = ty0 / 2 - 1;
  auto coarse_fetch = [&](int pp) {
    if constexpr (Ld::kCoarse) {
      const bool pv = pp >= 1 && pp < N;
#pragma unroll
      for (int q = 0; q < CPT; ++q) {
        const int e = tid + q * ZTHREADS, J = J0 + e / C1;
        float v = 0.f;
        if (pv && e < CE && J >= 0 && J < C1) {
          const float* c = ld.ec + ((pp >> 1) * C1 + J) * C1 + e % C1;
          v = __ldg(c);
          if (pp & 1) v = 0.5f * (v + __ldg(c + C1 * C1));
        }
        cn[q] = v;
      }
    }
  };
  auto coarse_store = [&](int pp) {
    if constexpr (Ld::kCoarse) {
#pragma unroll
      for (int q = 0; q < CPT; ++q)
        if (tid + q * ZTHREADS < CE) scz[(pp & 1) * CE + tid + q * ZTHREADS] = cn[q];
    }
  };
  if constexpr (Ld::kCoarse) {   // the first plane's rows, the second's on their way
    coarse_fetch(p);
    coarse_store(p);
    coarse_fetch(p + 1);
    __syncthreads();
  }

  const int jr0 = ty0 + RT * (int)threadIdx.y;   // this thread's rows jr0 .. jr0 + 3
  const bool ci = i >= 1, c0 = ci && jr0 > 0;    // interior column; interior node of row jr0
  const bool ex = i == N - 1, ey = jr0 + RT == N;
  const float c3s = (float)g.c3, c12s = (float)g.c12;
  const float2 c3 = make_float2(c3s, c3s), mc12 = make_float2(-c12s, -c12s);
  const float2 z2 = make_float2(0.f, 0.f);
  // output pair q: rows jr0 + q and jr0 + q + 2. As in k_zm3f: U unscaled
  // couplings and D diagonal part of the output of plane p - 1, Nn couplings
  // of the output of plane p with plane p - 1; of the kappa layer below, the
  // element pairs (kb), their sums along x (Xb), along y (Yb) and of four (Sb)
  float2 U[2], D[2], Nn[2], vc[2], kb[3][2], Xb[3], Yb[2][2], Sb[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) U[q] = D[q] = Nn[q] = vc[q] = Sb[q] = Yb[q][0] = Yb[q][1] = z2;
#pragma unroll
  for (int k = 0; k < 3; ++k) kb[k][0] = kb[k][1] = Xb[k] = z2;
  typename Epi::Pre pre[RT];
  float dot = 0.0f;
  const float* vthr = ring + 4 + RT * (int)threadIdx.y * N1 + i - 1;            // + shift: row jr0 - 1, column i - 1
  const float* kthr = ring + NA * VS + 4 + RT * (int)threadIdx.y * N + i - 1;   // row jr0 - 1, element i - 1
  const int o0 = jr0 * N1 + i;
  int sh = voff(p);
  int st = 0;
  unsigned par = 0;    // phase parity of each slot's next completion
  bool timed_out = false;
#pragma unroll 2
  for (; p <= z1; ++p) {
    const bool landed = mbar_wait(bar0 + 8u * st, (par >> st) & 1u);
    if (landed) {
      pend &= ~(1u << st);
      par ^= 1u << st;
    }
    float* slot = ring + st * SS;
    if (landed && p >= 1 && p < N) {
      if constexpr (Ld::kCoarse) {   // W b + P e_c (0 on the boundary, as W, b and e_c are)
        const float* cz = scz + (p & 1) * CE + (i >> 1);
        const int ox = i & 1;
#pragma unroll
        for (int rr = (int)threadIdx.y; rr < R + 2; rr += ZTHREADS / N) {
          const int jj = rr + 1;                     // fine row ty0 - 1 + rr = 2 J0 + jj
          const float* c = cz + (jj >> 1) * C1;
          float h = c[0] + c[ox];                    // twice the value along x
          h = (jj & 1) ? 0.25f * (h + (c[C1] + c[C1 + ox])) : 0.5f * h;
          float* e = slot + 4 + sh + rr * N1 + i;
          e[0] = fmaf(e[0], e[VS], h);
        }
      } else if constexpr (NA > 1) {   // combine the arrays into the field (both are 0 on the boundary)
        for (int e = tid; e < VS; e += ZTHREADS) slot[e] = ld.combine1(slot[e], slot[VS + e]);
      } else {                  // clear the field's boundary columns and rows
        float* row = slot + 4 + sh;
        if (tid < R + 2) row[tid * N1] = row[tid * N1 + N] = 0.f;
        if (ty0 == 0 && threadIdx.y == 0) row[N1 + i] = 0.f;
        if (ty0 + R == N && threadIdx.y == 0) row[(R + 1) * N1 + i] = 0.f;
      }
    }
    coarse_store(p + 1);
    fence_proxy_async_smem();       // this thread's shared-memory writes before later copies
    // plane p complete; the slot of plane p - 1 is free (or a wait gave up:
    // every thread leaves the loop together)
    if (__syncthreads_or(!landed)) {
      timed_out = true;
      break;
    }
    coarse_fetch(p + 2);
    if (p + ZW_S - 1 <= z1) {
      const int sn = (st + ZW_S - 1) % ZW_S;
      issue(p + ZW_S - 1, sn);
      pend |= 1u << sn;
    }
    typename Epi::Pre nxt[RT];
    if (p >= z0 && p < z1 && p >= 1 && p < N) {
#pragma unroll
      for (int r = 0; r < RT; ++r) nxt[r] = epi.load(p * P + o0 + r * N1);
    }
    // node row pairs (jr0 - 1 + k, jr0 + 1 + k), element row pairs likewise
    float2 v[4][3], ka[3][2];
    if (p >= 1 && p < N) {
      const float* sv = vthr + st * SS + sh;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) v[k][dx] = make_float2(sv[k * N1 + dx], sv[(k + 2) * N1 + dx]);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) v[k][dx] = z2;
    }
    {
      const float* sk = kthr + st * SS;
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int a = 0; a < 2; ++a) ka[k][a] = make_float2(sk[k * N + a], sk[(k + 2) * N + a]);
    }
    float2 Xa[3], Ya[2][2], Sa[2], ks[3][2];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      Xa[k] = add2(ka[k][0], ka[k][1]);
      ks[k][0] = add2(kb[k][0], ka[k][0]);
      ks[k][1] = add2(kb[k][1], ka[k][1]);
    }
    const int m = p - 1;
    const bool mi = m >= 1 && m < N;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      Ya[q][0] = add2(ka[q][0], ka[q + 1][0]);
      Ya[q][1] = add2(ka[q][1], ka[q + 1][1]);
      Sa[q] = add2(Xa[q], Xa[q + 1]);
      const float2 *v0 = v[q], *v1 = v[q + 1], *v2 = v[q + 2];
      // outputs of plane p - 1 are complete: couplings with plane p across layer p - 1
      float2 u = fma2(Yb[q][0], v1[0], U[q]);
      u = fma2(Yb[q][1], v1[2], u);
      u = fma2(Xb[q], v0[1], u);
      u = fma2(Xb[q + 1], v2[1], u);
      u = fma2(kb[q][0], v0[0], u);
      u = fma2(kb[q][1], v0[2], u);
      u = fma2(kb[q + 1][0], v2[0], u);
      u = fma2(kb[q + 1][1], v2[2], u);
      const float2 done = fma2(mc12, u, mul2(c3, D[q]));
      if (m >= z0) {
        const int o = m * P + o0;
        dot += epi(o + q * N1, (q ? ci : c0) && mi, done.x, vc[q].x, pre[q]);
        dot += epi(o + (q + 2) * N1, ci && mi, done.y, vc[q].y, pre[q + 2]);
      }
      // output p: couplings with plane p - 1 and the in-plane diagonal edges
      u = fma2(ks[q][0], v0[0], Nn[q]);
      u = fma2(ks[q][1], v0[2], u);
      u = fma2(ks[q + 1][0], v2[0], u);
      U[q] = fma2(ks[q + 1][1], v2[2], u);
      D[q] = mul2(add2(Sb[q], Sa[q]), v1[1]);
      // output p + 1: couplings with plane p across layer p
      u = mul2(Ya[q][0], v1[0]);
      u = fma2(Ya[q][1], v1[2], u);
      u = fma2(Xa[q], v0[1], u);
      u = fma2(Xa[q + 1], v2[1], u);
      u = fma2(ka[q][0], v0[0], u);
      u = fma2(ka[q][1], v0[2], u);
      u = fma2(ka[q + 1][0], v2[0], u);
      Nn[q] = fma2(ka[q + 1][1], v2[2], u);
      vc[q] = v1[1];
    }
    if (m >= z0) {   // boundary nodes beyond the tile's last column and row
      const int o = m * P + o0;
      if (ex) {
#pragma unroll
        for (int r = 0; r < RT; ++r) epi.zero(o + r * N1 + 1);
      }
      if (ey) {
        epi.zero(o + RT * N1);
        if (ex) epi.zero(o + RT * N1 + 1);
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      kb[k][0] = ka[k][0];
      kb[k][1] = ka[k][1];
      Xb[k] = Xa[k];
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      Yb[q][0] = Ya[q][0];
      Yb[q][1] = Ya[q][1];
      Sb[q] = Sa[q];
    }
#pragma unroll
    for (int r = 0; r < RT; ++r) pre[r] = nxt[r];
    st = (st + 1) % ZW_S;
    sh = (sh + 1) & 3;
  }
  if (timed_out) {
    // record the timeout, let the copies still in flight land (bounded), end the CTA
    if (tid == 0) atomicAdd(&g_zt_timeouts, 1u);
    for (int s2 = 0; s2 < ZW_S; ++s2)
      if (pend & (1u << s2)) mbar_wait(bar0 + 8u * s2, (par >> s2) & 1u);
    return;
  }
  if (part) {
    // the partial sits where the first 32 x 16 tile of this CTA's rows puts
    // it; the other tile it covers gets 0
    double v = warp_sum3((double)dot);
    if ((tid & 31) == 0) s_w[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
      double r = 0.0;
#pragma unroll
      for (int w = 0; w < ZTHREADS / 32; ++w) r += s_w[w];
      constexpr int R2 = zw_rows(N, 2);
      double* pt = part + (int64_t)blockIdx.y * g.tiles_s + (int64_t)zq * (N / R2) + ty0 / R2;
      pt[0] = r;
      pt[1] = 0.0;
    }
  }
  prof_tick3(prof);
}

inline dim3 gridz(const Grid& g, int64_t B) { return dim3((unsigned)g.zx, (unsigned)B, 1); }

// Full-width tiles staged by bulk copies: n in 32..256 and the partials'
// layout of whole tiles (every grid of make_grid with stencil_tile 0 or 2).
inline bool zm_wide(const Grid& g) {
  return g.zt != 1 && zw_mesh(g.n) && g.ns % 4 == 0 && g.es % 4 == 0 &&
         (g.zx == (int64_t)(g.n / zw_rows(g.n, 2)) * ((g.n + 1 + g.zc - 1) / g.zc));
}

// The grid with the z-chunks of a launch that leaves no partial sums (A x, the
// pre-smoother, the post-smoother below the finest level). A CTA takes about
// as long as its planes and two more (halo planes, filling its pipeline) and
// the CTAs run in waves of two per SM, so the chunk height is the one with the
// least waves x planes; every node's value is the same for any height. With
// the 16 planes of the partial sums' layout, 6 samples of 32^3 were 36 CTAs
// (FP64 pre-smoother: 74 us): a coupled FP64 batch of 6 samples of 128^3 went
// from 26.9 to 24.3 ms, 16 mixed solves of 64^3 from 3.87 to 3.55 ms (one CTA
// per SM as a wave: 24.7 and 3.65, three: 24.7 and 3.59).
constexpr int64_t CHUNK_WAVE = 2 * 152;
template <class T>
inline Grid flat_chunks(Grid g, int64_t B) {
  if (g.zset) return g;
  // the four-row FP32 kernel takes two 32 x 16 tiles per CTA
  const int64_t tiles = ((g.n + 31) / 32) * ((g.n + 15) / 16) / (sizeof(T) == 4 && zm_wide(g) && g.zt == 0 ? 2 : 1);
  const int64_t N1 = g.n + 1;
  int64_t best = -1;
  for (int64_t c = 1; 2 * c <= N1; ++c) {
    const int64_t zc = (N1 + c - 1) / c;
    if ((N1 + zc - 1) / zc != c) continue;
    const int64_t t = (tiles * B * c + CHUNK_WAVE - 1) / CHUNK_WAVE * (zc + 2);
    if (best < 0 || t < best) {
      best = t;
      g.zc = (int)zc;
    }
  }
  g.zx = ((g.n + 31) / 32) * ((g.n + 15) / 16) * (int)((N1 + g.zc - 1) / g.zc);
  return g;
}

template <int N, class LP, class Epi>
inline void launch_zm3n_at(cudaStream_t s, const Grid& g, int64_t B, const float* kappa, const LP& lp,
                           const int32_t* active, const Epi& epi, double* part, Prof p) {
  constexpr int NA = LP::kArrays, R = zw_rows(N, 4);
  // up to 76 KB of ring and coarse rows per CTA (opt-in above 48 KB)
  constexpr int smem = (int)sizeof(float) * ZW_S * (NA * zw_vslot(N, 4) + zw_kslot(N, 4)) + 8 * ZW_S +
                       (LP::kCoarse ? (int)sizeof(float) * 2 * (R / 2 + 2) * (N / 2 + 1) : 0);
  static std::atomic<uint64_t> opted{0};
  if (once_per_device(opted, [] {
        return cudaFuncSetAttribute(k_zm3n<N, LP, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      }) != cudaSuccess)
    return;   // the launcher's cudaGetLastError reports it
  k_zm3n<N, LP, Epi><<<dim3((unsigned)(g.zx / 2), (unsigned)B, 1), dim3(N, ZTHREADS / N, 1), smem, s>>>(
      g, kappa, lp, active, epi, part, p);
}
template <class LP, class Epi>
inline void launch_zm3n(cudaStream_t s, const Grid& g, int64_t B, const float* kappa, const LP& lp,
                        const int32_t* active, const Epi& epi, double* part, Prof p) {
  if (g.n == 32) launch_zm3n_at<32>(s, g, B, kappa, lp, active, epi, part, p);
  else if (g.n == 64) launch_zm3n_at<64>(s, g, B, kappa, lp, active, epi, part, p);
  else if (g.n == 128) launch_zm3n_at<128>(s, g, B, kappa, lp, active, epi, part, p);
  else launch_zm3n_at<256>(s, g, B, kappa, lp, active, epi, part, p);
}

// The z-march launch of an epilogue: the paired FP32 kernel for float.
template <class T, class Ld, class Epi>
inline void launch_zm3(cudaStream_t s, const Grid& g, int64_t B, const T* kappa, const Ld& ld,
                       const int32_t* active, const Epi& epi, double* part, Prof p,
                       const T* ks = nullptr) {
  if constexpr (std::is_same<T, double>::value) {
    if (ks) {   // FP64 on the element sums and the per-node kappa sums
      k_zm3q<Ld, Epi><<<gridz(g, B), dim3(ZTX, ZTY / ZRY, 1), 0, s>>>(g, kappa, ks, 4 * g.ns, ld, active, epi,
                                                                        part, p);
      return;
    }
  }
  if constexpr (std::is_same<T, float>::value) {
    using LP = LdPaired<Ld>;
    const typename LP::type lp = LP::make(ld);
    // bulk-copy staging: full-width tiles (n in 32..256), 16-byte aligned arrays;
    // stencil_tile 0: four rows per thread, 2: two rows per thread
    if (zm_wide(g) && lp.aligned16() && ((uintptr_t)kappa & 15) == 0) {
      constexpr int NA = LP::type::kArrays;
      if (g.zt == 0) {
        launch_zm3n(s, g, B, kappa, lp, active, epi, part, p);
      } else {
        const size_t smem = sizeof(float) * ZW_S * (NA * zw_vslot(g.n, 2) + zw_kslot(g.n, 2)) + 8 * ZW_S;
        k_zm3w<typename LP::type, Epi><<<gridz(g, B), dim3(g.n, ZTHREADS / g.n, 1), smem, s>>>(
            g, kappa, lp, active, epi, part, p);
      }
    }
    else
      k_zm3f<typename LP::type, Epi><<<gridz(g, B), dim3(ZTX, ZTY / ZRY, 1), 0, s>>>(g, kappa, lp, active,
                                                                                   epi, part, p);
  }
  else
    k_zm3<T, Ld, Epi><<<gridz(g, B), dim3(ZTX, ZTY / ZRY, 1), 0, s>>>(g, kappa, ld, active, epi, part, p);
}


template <class T>
__global__ void __launch_bounds__(256) k_winv3(Grid g, const T* __restrict__ K, double omega,
                                               T* __restrict__ W, int pz) {
  const int64_t b = blockIdx.y;
  const NodeCol c = node_col3(g.n, pz);
  if (!c.valid) return;
  const int n = g.n, N1 = n + 1;
  for (int k = c.k0; k < c.k1; ++k) {
    Node3 q;
    q.i = c.i;
    q.j = c.j;
    q.k = k;
    q.valid = true;
    q.interior = q.i > 0 && q.i < n && q.j > 0 && q.j < n && k > 0 && k < n;
    q.idx = ((int64_t)k * N1 + q.j) * N1 + q.i;
    T w = T(0);
    if (q.interior) {
      T kk[2][2][2];
      load_k8(K + b * g.es, g.n, q, kk);
      w = T(omega) / diag3(kk, g.c3);
    }
    W[b * g.ns + q.idx] = w;
  }
}

// x = 0 at every node, r = h^3 at interior nodes and 0 on the boundary
// (r may be null): one CTA per z-plane, threads along x, so the stores are
// row-contiguous and the CTA count is N1 per sample.
template <class T>
__global__ void __launch_bounds__(256) k_init3(Grid g, T* __restrict__ X, T* __restrict__ R, Prof prof) {
  const int64_t b = blockIdx.y;
  const int n = g.n, N1 = n + 1, k = blockIdx.x;
  const int64_t plane = b * g.ns + (int64_t)k * N1 * N1;
  const T h3 = T(g.h * g.h * g.h);
  const bool kin = k > 0 && k < n;
  for (int j = threadIdx.y; j <= n; j += blockDim.y) {
    const bool jin = kin && j > 0 && j < n;
    T* x = X + plane + (int64_t)j * N1;
    T* r = R ? R + plane + (int64_t)j * N1 : nullptr;
    for (int i = threadIdx.x; i <= n; i += blockDim.x) {
      x[i] = T(0);
      if (r) r[i] = (jin && i > 0 && i < n) ? h3 : T(0);
    }
  }
  prof_tick3(prof);
}

// Full weighting: bc(I) = sum_{d in {-1,0,1}^3} w(dx) w(dy) w(dz) r1(2I + d).
// A thread walks coarse planes and keeps the weighted odd fine plane between two
// of them: 2 fine planes a coarse one instead of 3 (18 loads and about 18 FP64
// operations instead of 27 and 30; bound by the FP64 pipe and L2 latency).
// FP64, 6 samples of 128^3: 146 -> 104 us.
template <class T>
__global__ void __launch_bounds__(256) k_restrict3(Grid gc, int64_t nsf, const T* __restrict__ R1,
                                                   T* __restrict__ Bc, const int32_t* __restrict__ active,
                                                   Prof prof, int pz) {
  const int64_t b = blockIdx.y;
  if (!active[b]) return;
  prof_tick3(prof);
  const NodeCol c = node_col3(gc.n, pz);
  if (!c.valid) return;
  const int nc = gc.n, C1 = nc + 1;
  const int64_t N1 = 2 * gc.n + 1, P = N1 * N1;
  const T wt[3] = {T(0.5), T(1), T(0.5)};
  const bool col_in = c.i > 0 && c.i < nc && c.j > 0 && c.j < nc;
  const T* col = R1 + b * nsf + (int64_t)(2 * c.j) * N1 + 2 * c.i;
  // the fine plane z weighted in x and y; an odd plane serves the coarse
  // planes on both sides of it
  auto plane = [&](int z) -> T {
    T pl = T(0);
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      const T* rr = col + (int64_t)z * P + dy * N1;
      pl += wt[dy + 1] * (T(0.5) * __ldg(rr - 1) + __ldg(rr) + T(0.5) * __ldg(rr + 1));
    }
    return pl;
  };
  T below = col_in && c.k0 > 0 ? plane(2 * c.k0 - 1) : T(0);
  for (int k = c.k0; k < c.k1; ++k) {
    T v = T(0);
    if (col_in && k < nc) {
      const T mid = k > 0 ? plane(2 * k) : T(0), above = plane(2 * k + 1);
      if (k > 0) v = T(0.5) * below + mid + T(0.5) * above;
      below = above;
    }
    Bc[b * gc.ns + ((int64_t)k * C1 + c.j) * C1 + c.i] = v;
  }
}

// Coarsest grid (n = 2, one unknown at (1,1,1)): e = b / D exactly.
template <class T>
__global__ void k_coarse3(Grid g, const T* __restrict__ K, const T* __restrict__ Bv, T* __restrict__ E,
                          const int32_t* __restrict__ active, int64_t B) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B || !active[b]) return;
  const T* k = K + b * g.es;
  T s = T(0);
  for (int e = 0; e < 8; ++e) s += k[e];
  const T d = T(g.c3) * s;
  for (int t = 0; t < 27; ++t) E[b * g.ns + t] = T(0);
  E[b * g.ns + 13] = Bv[b * g.ns + 13] / d;
}

// Pointwise: tmp = e + P ec (trilinear prolongation of the coarse
// correction; E == nullptr: tmp = P ec, the nested initial guess). A thread
// takes the fine nodes 2I and 2I + 1 of one fine row y in PROLONG_PZ
// consecutive z-planes. Per coarse plane the coarse rows under it (1 or 2 by
// the parity of y) are summed at coarse columns I and I + 1 once; an even fine
// plane takes these sums, the odd plane after it the sums of two coarse planes;
// the even node takes the first column's, the odd node both, each divided by
// the number of values. 2.25 FP64 operations per node (4.5 with the sums of
// every fine plane formed anew; FP64, 6 samples of 128^3: 147 -> 90 us, bound
// by the FP64 pipe and latency). Warps run along I with uniform parities, so
// the gathers do not diverge; several planes per thread keep the CTAs few and
// large. PROLONG_PZ is even: a thread starts on a coarse plane.
constexpr int PROLONG_PZ = 8;

template <class T>
__global__ void __launch_bounds__(256) k_prolong3(Grid g, int64_t nsc, const T* __restrict__ E,
                                                  const T* __restrict__ Ec, T* __restrict__ Tmp,
                                                  const int32_t* __restrict__ active, Prof prof) {
  const int64_t b = blockIdx.z;
  if (!active[b]) return;
  const int n = g.n, nc = n / 2, N1 = n + 1, C1 = nc + 1;
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int ry = blockIdx.y * blockDim.y + threadIdx.y;   // (z-group, y) index
  const int rows_y = ((N1 + 7) / 8) * 8;
  const int zg = ry / rows_y, y = ry - zg * rows_y;
  if (prof.acc && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0)
    atomicAdd(prof.acc, prof.per_sample);
  if (I > nc || y > n) return;
  const T* ec = Ec + b * nsc + (int64_t)(y >> 1) * C1 + I;
  const T* ep = E ? E + b * g.ns + (int64_t)y * N1 + 2 * I : nullptr;
  T* tp = Tmp + b * g.ns + (int64_t)y * N1 + 2 * I;
  const int64_t P = (int64_t)N1 * N1;
  const bool oy = y & 1, odd = I < nc;
  const bool in0 = y >= 1 && y < n && I >= 1 && odd, in1 = y >= 1 && y < n && odd;
  // coarse plane Kc under the row, at coarse columns I and I + 1
  auto rows = [&](int Kc, T& s0, T& s1) {
    const T* row = ec + (int64_t)Kc * C1 * C1;
    s0 = __ldg(row);
    s1 = odd ? __ldg(row + 1) : T(0);
    if (oy) {
      s0 += __ldg(row + C1);
      if (odd) s1 += __ldg(row + C1 + 1);
    }
  };
  auto put = [&](int z, T s0, T s1, T inv) {
    const bool zin = z >= 1 && z < n;
    const int64_t o = z * P;
    const T e0 = ep ? ep[o] : T(0), e1 = ep && odd ? ep[o + 1] : T(0);
    tp[o] = zin && in0 ? fma(s0, inv, e0) : T(0);
    if (odd) tp[o + 1] = zin && in1 ? fma(s0 + s1, T(0.5) * inv, e1) : T(0);
  };
  const int z0 = zg * PROLONG_PZ, z1 = min(z0 + PROLONG_PZ, n + 1);
  const T inv = oy ? T(0.5) : T(1);
  T a0, a1;
  rows(z0 >> 1, a0, a1);
  for (int z = z0; z < z1; z += 2) {
    put(z, a0, a1, inv);
    if (z + 1 >= z1) break;
    T b0, b1;
    rows((z >> 1) + 1, b0, b1);
    put(z + 1, a0 + b0, a1 + b1, T(0.5) * inv);
    a0 = b0;
    a1 = b1;
  }
}

// grid of k_prolong3 for fine mesh g and B samples
inline dim3 prolong3_grid(const Grid& g, int64_t B) {
  const int nc = g.n / 2, rows_y = ((g.n + 1 + 7) / 8) * 8;
  const int zgroups = (g.n + 1 + PROLONG_PZ - 1) / PROLONG_PZ;
  return dim3((unsigned)((nc + 1 + 31) / 32), (unsigned)(rows_y / 8 * zgroups), (unsigned)B);
}

// Nested initial guess by cubic interpolation of the coarse-mesh solution: a
// warp makes one fine row of GUESS_COLS coarse columns, a lane two fine
// columns (2I from its own values, 2I + 1 from its neighbours'), walking
// GUESS_PZ fine planes with the values of four coarse planes in registers:
// 3.5 FP64 operations per node.
constexpr int GUESS_PZ = 32, GUESS_WARPS = 8;
__global__ void __launch_bounds__(32 * GUESS_WARPS) k_guess3(Grid g, int64_t nsc, const double* __restrict__ Uc,
                                                             double* __restrict__ X,
                                                             const int32_t* __restrict__ active, Prof prof) {
  const int64_t b = blockIdx.z;
  if (!active[b]) return;
  const int n = g.n, N1 = n + 1, nc = n / 2, C1 = nc + 1, lane = threadIdx.x;
  const int rows = (N1 + GUESS_WARPS - 1) / GUESS_WARPS;   // row groups per plane chunk
  const int zg = blockIdx.y / rows, j = (blockIdx.y - zg * rows) * GUESS_WARPS + threadIdx.y;
  if (j > n) return;
  const int I = blockIdx.x * GUESS_COLS - GUESS_HALO + lane;
  const bool in = I >= 0 && I <= nc;
  const bool out = in && lane >= GUESS_HALO && lane < GUESS_HALO + GUESS_COLS;
  const double* uc = Uc + b * nsc + (in ? I : 0);
  double* x = X + b * g.ns;
  // the coarse plane K at this fine row: column I, and the odd column beside it
  auto even = [&](int K) -> double {
    return in ? cubic_at(j, nc, [&](int J) { return __ldg(uc + (K * C1 + J) * C1); }) : 0.0;
  };
  const int z0 = zg * GUESS_PZ, z1 = min(z0 + GUESS_PZ, N1);
  CubicWindow we, wo;
  we.start(z0, nc, even);
  wo.b = we.b;
#pragma unroll
  for (int k = 0; k < 4; ++k) wo.v[k] = guess_odd(I, nc, we.v[k]);
  for (int z = z0; z < z1; ++z) {
    // one coarse plane further on every second fine plane (uniform across the warp)
    const int nb = cubic_base(z >> 1, nc);
    while (we.b < nb) {
      we.advance((we.b + 2) * 2, nc, even);
      wo.v[0] = wo.v[1];
      wo.v[1] = wo.v[2];
      wo.v[2] = wo.v[3];
      wo.v[3] = guess_odd(I, nc, we.v[3]);
      wo.b = we.b;
    }
    const bool rin = j > 0 && j < n && z > 0 && z < n;
    if (out) {
      const int64_t o = ((int64_t)z * N1 + j) * N1 + 2 * I;
      x[o] = rin && I > 0 && I < nc ? we.value(z, nc) : 0.0;
      if (I < nc) x[o + 1] = rin ? wo.value(z, nc) : 0.0;
    }
  }
  if (prof.acc && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0)
    atomicAdd(prof.acc, prof.per_sample);
}

// QoI partials, one per z-plane (g.tiles_q = N1 per sample): domain: w =
// h^3 at interior nodes; box [L, H]^3 in node indices: w = h^3 chi_x chi_y
// chi_z / |box|, chi = 1 inside, 1/2 on a face. A CTA reads only the nodes
// of its plane inside the region, one FP64 add per node: each row is summed
// with its column weights (1, or 1/2 on the two face columns), each row sum
// is added with its row weight and the plane sum is scaled once.
template <class T>
__global__ void __launch_bounds__(256) k_qoi3(Grid g, int box, int L, int H, double inv_vol,
                                              const T* __restrict__ X, double* __restrict__ part, Prof prof) {
  const int64_t b = blockIdx.y;
  const int n = g.n, N1 = n + 1, k = blockIdx.x;
  const int lo = box ? L : 1, hi = box ? H : n - 1;
  double acc = 0.0;
  if (k >= lo && k <= hi) {
    const T* x = X + b * g.ns + (int64_t)k * N1 * N1;
    for (int j = lo + threadIdx.y; j <= hi; j += blockDim.y) {
      double row = 0.0;
      for (int i = lo + threadIdx.x; i <= hi; i += blockDim.x) {
        const double v = (double)x[(int64_t)j * N1 + i];
        row = (box && (i == lo || i == hi)) ? fma(0.5, v, row) : row + v;
      }
      acc = (box && (j == lo || j == hi)) ? fma(0.5, row, acc) : acc + row;
    }
    double wk = g.h * g.h * g.h;
    if (box) wk *= ((k == lo || k == hi) ? 0.5 : 1.0) * inv_vol;
    acc *= wk;
  }
  cta_partial3(acc, part, g.tiles_q);
  prof_tick3(prof);
}

inline dim3 block3() { return dim3(BX, BY, 1); }


}  // namespace

namespace d3 {

bool post32_is_fused(const Grid& g) { return zm_wide(g) && g.zt == 0; }

template <class T>
cudaError_t apply(cudaStream_t s, const Grid& g, const T* kappa, const T* x, T* y, int64_t B, Prof p) {
  launch_zm3<T>(s, flat_chunks<T>(g, B), B, kappa, LdX<T>{x, g.ns}, nullptr, EpiApply<T>{y, g.ns}, nullptr, p);
  return cudaGetLastError();
}
template <class T>
cudaError_t winv(cudaStream_t s, const Grid& g, const T* kappa, double omega, T* w, int64_t B) {
  const int pz = node_pz(g.n);
  k_winv3<T><<<dim3(node_col3_blocks(g.n, pz), (unsigned)B, 1), block3(), 0, s>>>(g, kappa, omega, w, pz);
  return cudaGetLastError();
}
template <class T>
cudaError_t pcg_init(cudaStream_t s, const Grid& g, T* x, T* r, int64_t B, Prof p) {
  if (!r) return d2::zero_nodes<T>(s, g, x, B, p);   // flat: node layout does not matter
  k_init3<T><<<dim3((unsigned)(g.n + 1), (unsigned)B, 1), block3(), 0, s>>>(g, x, r, p);
  return cudaGetLastError();
}
template <class T>
cudaError_t pcg_pq(cudaStream_t s, const Grid& g, const T* kappa, const T* z, const T* p_old, T* p_new,
                   T* q, const Scalars& sc, double* part, int64_t B, Prof p, const T* ks) {
  launch_zm3<T>(s, g, B, kappa, LdPupd<T>{z, p_old, sc.beta, g.ns, T(0)}, sc.active,
                EpiAq<T>{q, p_new, g.ns}, part, p, ks);
  return cudaGetLastError();
}
template <class T>
cudaError_t mg_pre(cudaStream_t s, const Grid& g, const T* kappa, const T* w, const T* b, T* e, T* r1,
                   const int32_t* active, int64_t B, Prof p, const T* ks) {
  launch_zm3<T>(s, flat_chunks<T>(g, B), B, kappa, LdWb<T>{w, b, g.ns}, active, EpiMgRes<T>{b, r1, e, g.ns}, nullptr, p,
                ks);
  return cudaGetLastError();
}
template <class T>
cudaError_t restrict_(cudaStream_t s, const Grid& fine, const Grid& coarse, const T* r1, T* bc,
                      const int32_t* active, int64_t B, Prof p) {
  const int pz = node_pz(coarse.n);
  k_restrict3<T><<<dim3(node_col3_blocks(coarse.n, pz), (unsigned)B, 1), block3(), 0, s>>>(coarse, fine.ns, r1,
                                                                                          bc, active, p, pz);
  return cudaGetLastError();
}
template <class T>
cudaError_t coarse_solve(cudaStream_t s, const Grid& g, const T* kappa, const T* b, T* e,
                         const int32_t* active, int64_t B) {
  k_coarse3<T><<<(unsigned)((B + 127) / 128), 128, 0, s>>>(g, kappa, b, e, active, B);
  return cudaGetLastError();
}
template <class T>
cudaError_t mg_post(cudaStream_t s, const Grid& g, const Grid& coarse, const T* kappa, const T* w,
                    const T* b, const T* e, const T* ec, T* out, T* tmp, const int32_t* active,
                    double* part, int64_t B, Prof p, const T* ks) {
  const Grid h = part ? g : flat_chunks<T>(g, B);
  if constexpr (std::is_same<T, float>::value) {
    // one kernel, which forms e itself (the arrays are a plan's, 256-byte aligned)
    if (!e) {
      if (!post32_is_fused(g) || (((uintptr_t)w | (uintptr_t)b | (uintptr_t)kappa) & 15) != 0)
        return cudaErrorInvalidValue;
      launch_zm3n(s, h, B, kappa, LdPostf{w, b, ec, g.ns, coarse.ns}, active, EpiMgPost<float>{w, b, out, g.ns}, part,
                  p);
      return cudaGetLastError();
    }
  }
  k_prolong3<T><<<prolong3_grid(g, B), dim3(32, 8, 1), 0, s>>>(g, coarse.ns, e, ec, tmp, active,
                                                                 Prof{nullptr, 0.0});
  launch_zm3<T>(s, h, B, kappa, LdX<T>{tmp, g.ns}, active, EpiMgPost<T>{w, b, out, g.ns}, part, p, ks);
  return cudaGetLastError();
}
template <class T>
cudaError_t qoi(cudaStream_t s, const Grid& g, int box, int L, int H, double inv_vol, const T* x,
                double* part, int64_t B, Prof p) {
  k_qoi3<T><<<dim3((unsigned)(g.n + 1), (unsigned)B, 1), block3(), 0, s>>>(g, box, L, H, inv_vol, x, part, p);
  return cudaGetLastError();
}
cudaError_t prolong_guess(cudaStream_t s, const Grid& g, const Grid& coarse, const double* uc,
                          double* x, const int32_t* active, int64_t B, Prof p) {
  if (coarse.n >= CUBIC_MIN_CELLS) {
    const int rows = (g.n + GUESS_WARPS) / GUESS_WARPS, zgroups = (g.n + GUESS_PZ) / GUESS_PZ;
    k_guess3<<<dim3((unsigned)((coarse.n + GUESS_COLS) / GUESS_COLS), (unsigned)(rows * zgroups), (unsigned)B),
               dim3(32, GUESS_WARPS, 1), 0, s>>>(g, coarse.ns, uc, x, active, p);
  } else {
    k_prolong3<double><<<prolong3_grid(g, B), dim3(32, 8, 1), 0, s>>>(g, coarse.ns, nullptr, uc, x, active, p);
  }
  return cudaGetLastError();
}

cudaError_t resid64(cudaStream_t s, const Grid& g, const double* kappa, const double* u, double* r,
                    const int32_t* active, double* part, int64_t B, Prof p, const double* ks) {
  if (ks)
    k_zm3q<LdX<double>, EpiResid><<<gridz(g, B), dim3(ZTX, ZTY / ZRY, 1), 0, s>>>(
        g, kappa, ks, 4 * g.ns, LdX<double>{u, g.ns}, active, EpiResid{r, g.ns, g.h * g.h * g.h}, part, p);
  else
    launch_zm3<double>(s, g, B, kappa, LdX<double>{u, g.ns}, active, EpiResid{r, g.ns, g.h * g.h * g.h},
                       part, p);
  return cudaGetLastError();
}

cudaError_t ksum(cudaStream_t s, const Grid& g, const double* kappa, double* ks, int64_t B, double omega,
                 double* w) {
  const int pz = node_pz(g.n);
  k_ksum3<<<dim3(node_col3_blocks(g.n, pz), (unsigned)B, 1), block3(), 0, s>>>(g, kappa, ks, 4 * g.ns, pz, omega, w);
  return cudaGetLastError();
}

// Waits of the bulk-copy z-march that gave up since the last call on this
// device (the counter is reset); read on `s` after the caller's own sync.
cudaError_t take_wait_timeouts(cudaStream_t s, unsigned* out) {
  unsigned h = 0;
  cudaError_t e = cudaMemcpyFromSymbolAsync(&h, g_zt_timeouts, sizeof(unsigned), 0, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess && h != 0) {
    const unsigned zero = 0;
    e = cudaMemcpyToSymbolAsync(g_zt_timeouts, &zero, sizeof(unsigned), 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  }
  *out = h;
  return e;
}

#define MLMC_INST3(T)                                                                              \
  template cudaError_t apply<T>(cudaStream_t, const Grid&, const T*, const T*, T*, int64_t, Prof); \
  template cudaError_t winv<T>(cudaStream_t, const Grid&, const T*, double, T*, int64_t);          \
  template cudaError_t pcg_init<T>(cudaStream_t, const Grid&, T*, T*, int64_t, Prof);              \
  template cudaError_t pcg_pq<T>(cudaStream_t, const Grid&, const T*, const T*, const T*, T*, T*,  \
                                 const Scalars&, double*, int64_t, Prof, const T*);                \
  template cudaError_t mg_pre<T>(cudaStream_t, const Grid&, const T*, const T*, const T*, T*, T*,  \
                                 const int32_t*, int64_t, Prof, const T*);                         \
  template cudaError_t restrict_<T>(cudaStream_t, const Grid&, const Grid&, const T*, T*,          \
                                    const int32_t*, int64_t, Prof);                                \
  template cudaError_t coarse_solve<T>(cudaStream_t, const Grid&, const T*, const T*, T*,          \
                                       const int32_t*, int64_t);                                   \
  template cudaError_t mg_post<T>(cudaStream_t, const Grid&, const Grid&, const T*, const T*,      \
                                  const T*, const T*, const T*, T*, T*, const int32_t*, double*,   \
                                  int64_t, Prof, const T*);                                        \
  template cudaError_t qoi<T>(cudaStream_t, const Grid&, int, int, int, double, const T*, double*, \
                              int64_t, Prof);

MLMC_INST3(double)
MLMC_INST3(float)

}  // namespace d3
}  // namespace mlmc
