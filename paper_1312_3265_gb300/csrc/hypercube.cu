// Hypercube transports W(x,s) of the staggered Wilson term (Sec. 3: the 16
// hypercube neighbours of the "8+16" stencil): the average over the 24
// orderings of the 4-link path from x to x+s, for the 8 stored displacements
// s = (s0, s1, s2, +1).
//
// The sum over orderings is built by dynamic programming over the walked
// directions, forward from x: for a set S of directions with signs s_S,
//   F(S) = sum_{mu in S} F(S \ mu) L_mu(x + s_{S \ mu}),   F({mu}) = L_mu(x),
// with L_mu(y) = U_mu(y) for s_mu = +1 and U_mu(y - mu)^+ for s_mu = -1, and
// W(x,s) = F({0,1,2,3}) / 24.  F(S) depends only on the signs inside S, so the
// 8 displacements share it: 18 two-direction and 20 three-direction partial
// sums (the signs of directions 0-2 free, direction 3 always +1) and the 8
// full ones take 36 + 60 + 32 = 128 matrix products per site, against 8 x 28
// = 224 when each displacement is built on its own.
//
// Eight threads per site, in one warp: each builds some of the partial sums
// in shared memory, then thread k assembles W(x, s_k).  FP64 throughout.
#include <algorithm>

#include "internal.h"
#include "common.cuh"

namespace swc {

namespace {

// The partial sums of a site: (direction mask S, sign bits on S), bit mu of
// the sign bits set when s_mu = -1; level 2 then level 3, masks increasing,
// sign patterns increasing.  pred: for each direction mu in S (increasing),
// the slot of F(S \ mu) among the level-2 sums (level 3) or the level-3 sums
// (the full sums, one per stored displacement k).
struct HcTables {
  unsigned char mask2[18], sg2[18];
  unsigned char mask3[20], sg3[20], mu3[20][3], pred3[20][3];
  unsigned char pred4[8][4];
};

constexpr int popc4(int m) { return (m & 1) + ((m >> 1) & 1) + ((m >> 2) & 1) + ((m >> 3) & 1); }

constexpr HcTables make_hc_tables() {
  HcTables t{};
  int n2 = 0, n3 = 0;
  for (int S = 0; S < 16; ++S) {
    const int lv = popc4(S);
    if (lv != 2 && lv != 3) continue;
    const int free = S & 7;  // directions whose sign varies
    for (int sg = 0; sg < 8; ++sg) {
      if (sg & ~free) continue;
      if (lv == 2) {
        t.mask2[n2] = (unsigned char)S;
        t.sg2[n2] = (unsigned char)sg;
        ++n2;
      } else {
        t.mask3[n3] = (unsigned char)S;
        t.sg3[n3] = (unsigned char)sg;
        ++n3;
      }
    }
  }
  for (int j = 0; j < 20; ++j) {
    int q = 0;
    for (int mu = 0; mu < 4; ++mu) {
      if (!((t.mask3[j] >> mu) & 1)) continue;
      const int T = t.mask3[j] & ~(1 << mu), sg = t.sg3[j] & T;
      int slot = 0;
      for (int i = 0; i < 18; ++i)
        if (t.mask2[i] == T && t.sg2[i] == sg) slot = i;
      t.mu3[j][q] = (unsigned char)mu;
      t.pred3[j][q] = (unsigned char)slot;
      ++q;
    }
  }
  for (int k = 0; k < 8; ++k)
    for (int mu = 0; mu < 4; ++mu) {
      const int T = 15 & ~(1 << mu), sg = k & T;
      int slot = 0;
      for (int j = 0; j < 20; ++j)
        if (t.mask3[j] == T && t.sg3[j] == sg) slot = j;
      t.pred4[k][mu] = (unsigned char)slot;
    }
  return t;
}

__constant__ HcTables kHc = make_hc_tables();

constexpr int kHcSites = 8;  // sites per 64-thread block (8 threads per site)

}  // namespace

__global__ void __launch_bounds__(64) hypercube_kernel(Geom g, GaugeC64 U, double2* __restrict__ W) {
  __shared__ double2 part[kHcSites][38][9];  // level-2 sums in 0..17, level-3 sums in 18..37
  const int ls = threadIdx.x >> 3, t = threadIdx.x & 7;
  const int n = blockIdx.x * kHcSites + ls;
  const bool valid = n < g.V;
  int x[4] = {0, 0, 0, 0}, df[4] = {0, 0, 0, 0}, db[4] = {0, 0, 0, 0};
  if (valid) {
    coords(g, n, x);
    hop_deltas(g, n, x, df, db);
  }
  // L_mu(y) for sign bit neg; a hop along mu from y reads only x_mu, which the
  // walked directions (never mu itself) leave unchanged, so db[mu] applies at y
  auto link = [&](int mu, int neg, int y) -> M3<double> {
    return neg ? dag(U.link(y + db[mu], mu)) : U.link(y, mu);
  };
  // x + s_T for the directions in T with the signs sg
  auto pos = [&](int T, int sg) {
    int y = n;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu)
      if ((T >> mu) & 1) y += ((sg >> mu) & 1) ? db[mu] : df[mu];
    return y;
  };
  auto store = [&](int slot, const M3<double>& M) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) part[ls][slot][i * 3 + j] = make_double2(M.e[i][j].re, M.e[i][j].im);
  };
  auto load = [&](int slot) {
    M3<double> M;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double2 v = part[ls][slot][i * 3 + j];
        M.e[i][j] = {v.x, v.y};
      }
    return M;
  };
  if (valid) {
    // two directions a < b: F = L_a(x) L_b(x + s_a) + L_b(x) L_a(x + s_b)
    for (int i = t; i < 18; i += 8) {
      const int S = kHc.mask2[i], sg = kHc.sg2[i];
      const int a = __ffs(S) - 1, b = __ffs(S & ~(1 << a)) - 1;
      const int na = (sg >> a) & 1, nb = (sg >> b) & 1;
      M3<double> M = mm(link(a, na, n), link(b, nb, pos(1 << a, sg)));
      madd(M, mm(link(b, nb, n), link(a, na, pos(1 << b, sg))));
      store(i, M);
    }
  }
  __syncwarp();
  if (valid) {
    // three directions: F(S) = sum_mu F(S \ mu) L_mu(x + s_{S \ mu})
    for (int j = (t + 6) & 7; j < 20; j += 8) {
      const int S = kHc.mask3[j], sg = kHc.sg3[j];
      M3<double> M;
#pragma unroll 1
      for (int q = 0; q < 3; ++q) {
        const int mu = kHc.mu3[j][q];
        const M3<double> term = mm(load(kHc.pred3[j][q]), link(mu, (sg >> mu) & 1, pos(S & ~(1 << mu), sg)));
        if (q == 0) M = term; else madd(M, term);
      }
      store(18 + j, M);
    }
  }
  __syncwarp();
  if (valid) {
    // all four directions for displacement k = t
    const int k = t;
    M3<double> M;
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
      const M3<double> term = mm(load(18 + kHc.pred4[k][mu]), link(mu, (k >> mu) & 1, pos(15 & ~(1 << mu), k)));
      if (mu == 0) M = term; else madd(M, term);
    }
    double2* out = W + ((size_t)n * 8 + k) * 9;
    const double w = 1.0 / 24.0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) out[i * 3 + j] = make_double2(w * M.e[i][j].re, w * M.e[i][j].im);
  }
}

// ---------------------------------------------------------------- by two-link sums
// The sum over the 24 orderings splits by the pair of directions walked
// first: with F2(S; x) the sum of the two orderings of a two-link path over
// the pair S,
//   24 W(x, s) = sum over the 6 pairs S of F2(S; x) F2(S^c; x + s_S),
// and the F2 of a lattice are shared: walked backwards, a two-link path is the
// adjoint of one based at its other end, so two fields per pair of directions
// serve every sign -- (+a,+b) and (+a,-b) for the spatial pairs, (+a,+3) and
// (-a,+3) for the pairs with direction 3.  12 sums of 2 products and 8 x 6
// products: 72 3x3 products per site, where hypercube_kernel takes 128.
//
// Bound by the FP64 pipe (7776 FMAs per site; 1.62 ms at 16^3x32 at the
// measured 1.26 TFLOP/s).  One thread computes one row of one matrix, so that
// a small lattice still fills the chip: a warp's FP64 FMA takes 64 clocks of
// its scheduler's pipe, and whole-matrix threads would run 648 of them in
// series.  The F2 fields (1728 B per site) go through a workspace a slab of
// time slices at a time.
// Measured against hypercube_kernel: 4^4 25 for 93 us, 8^4 80 for 176,
// 12^3x24 636 for 1467, 16^3x32 1.96 for 4.47 ms, 24^3x48 10.1 for 22.5 ms.
namespace {

__constant__ unsigned char kPairA[6] = {0, 0, 1, 0, 1, 2}, kPairB[6] = {1, 2, 2, 3, 3, 3};

// M or M^+ in memory (double2[9]).
struct MatRef {
  const double2* p;
  bool dag;
};
// acc += row i of A B
__device__ __forceinline__ void row_mm(cx<double> acc[3], const MatRef& A, const MatRef& B, int i) {
  const double sa = A.dag ? -1.0 : 1.0, sb = B.dag ? -1.0 : 1.0;
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const double2 a = __ldg(A.p + (A.dag ? m * 3 + i : i * 3 + m));
    const cx<double> av = {a.x, sa * a.y};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double2 b = __ldg(B.p + (B.dag ? j * 3 + m : m * 3 + j));
      cmac(acc[j].re, acc[j].im, av, cx<double>{b.x, sb * b.y});
    }
  }
}

}  // namespace

// F2 of the slab's slices: type 2 pair + variant (blockIdx.y), layout
// [12][sites][9].  Slice l of the slab is time slice (t0 + l) mod L3; the one
// after the slab's nt is needed for the spatial pairs only.
__global__ void __launch_bounds__(128) two_link_kernel(Geom g, GaugeC64 U, double2* __restrict__ F, int t0, int nt,
                                                     int sites) {
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  const int ls = id / 3, i = id - ls * 3;
  const int type = blockIdx.y, pr = type >> 1;
  const int S = g.stride[3], l = ls / S;
  if (ls >= sites || (l >= nt && pr >= 3)) return;
  int t = t0 + l;
  if (t >= g.L[3]) t -= g.L[3];
  const int n = t * S + (ls - l * S);
  int x[4], df[4], db[4];
  coords(g, n, x);
  hop_deltas(g, n, x, df, db);
  const int a = kPairA[pr], b = kPairB[pr];
  int dfa = 0, dba = 0, dfb = 0, dbb = 0;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    if (mu == a) dfa = df[mu], dba = db[mu];
    if (mu == b) dfb = df[mu], dbb = db[mu];
  }
  auto at = [&](int y, int mu) { return U.p + ((size_t)y * 4 + mu) * 9; };
  cx<double> acc[3] = {{0, 0}, {0, 0}, {0, 0}};
  if (!(type & 1)) {  // (+a, +b)
    row_mm(acc, {at(n, a), false}, {at(n + dfa, b), false}, i);
    row_mm(acc, {at(n, b), false}, {at(n + dfb, a), false}, i);
  } else if (pr < 3) {  // (+a, -b)
    row_mm(acc, {at(n, a), false}, {at(n + dfa + dbb, b), true}, i);
    row_mm(acc, {at(n + dbb, b), true}, {at(n + dbb, a), false}, i);
  } else {  // (-a, +3)
    row_mm(acc, {at(n + dba, a), true}, {at(n + dba, 3), false}, i);
    row_mm(acc, {at(n, 3), false}, {at(n + dfb + dba, a), true}, i);
  }
  double2* out = F + ((size_t)type * sites + ls) * 9 + i * 3;
#pragma unroll
  for (int j = 0; j < 3; ++j) out[j] = make_double2(acc[j].re, acc[j].im);
}

// W of the slab's nt slices from its F2.  full: the slab is the whole lattice
// (the slice after the last is the first).
__global__ void __launch_bounds__(128) pair_products_kernel(Geom g, const double2* __restrict__ F,
                                                          double2* __restrict__ W, int t0, int nt, int sites,
                                                          int full) {
  const long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int S = g.stride[3];
  const int ls = (int)(id / 24), r = (int)(id - (long long)ls * 24), k = r / 3, i = r - k * 3;
  if (ls >= nt * S) return;
  const int n = t0 * S + ls;
  int x[4], df[4], db[4];
  coords(g, n, x);
  hop_deltas(g, n, x, df, db);
  const int up = full ? df[3] : S;
  // F2 of spatial pair pr with the signs of k at slab site y; of (c, +3)
  auto spatial = [&](int pr, int y) -> MatRef {
    const int a = pr == 2 ? 1 : 0, b = pr == 0 ? 1 : 2;
    const bool na = (k >> a) & 1, nb = (k >> b) & 1;
    // (-a,-b): adjoint of (+a,+b) at y - a - b; (-a,+b): adjoint of (+a,-b) at y - a + b
    if (na) y += (a == 0 ? db[0] : db[1]) + (nb ? (b == 1 ? db[1] : db[2]) : (b == 1 ? df[1] : df[2]));
    return {F + ((size_t)(2 * pr + (na != nb)) * sites + y) * 9, na};
  };
  auto timelike = [&](int c, int y) -> MatRef {
    return {F + ((size_t)(6 + 2 * c + ((k >> c) & 1)) * sites + y) * 9, false};
  };
  auto step = [&](int mu) { return ((k >> mu) & 1) ? (mu == 0 ? db[0] : mu == 1 ? db[1] : db[2])
                                                   : (mu == 0 ? df[0] : mu == 1 ? df[1] : df[2]); };
  cx<double> acc[3] = {{0, 0}, {0, 0}, {0, 0}};
#pragma unroll 1
  for (int pr = 0; pr < 3; ++pr) {
    const int a = pr == 2 ? 1 : 0, b = pr == 0 ? 1 : 2, c = 2 - pr;
    row_mm(acc, spatial(pr, ls), timelike(c, ls + step(a) + step(b)), i);
    row_mm(acc, timelike(c, ls), spatial(pr, ls + step(c) + up), i);
  }
  double2* out = W + ((size_t)n * 8 + k) * 9 + i * 3;
  const double w = 1.0 / 24.0;
#pragma unroll
  for (int j = 0; j < 3; ++j) out[j] = make_double2(w * acc[j].re, w * acc[j].im);
}

int hypercube_build_f64(const Geom& g, const double2* U, double2* W, cudaStream_t st) {
  constexpr size_t kSite = 12 * 9 * sizeof(double2);
  // workspace: 256 MB, or an eighth of W where that is more (slices of a large
  // lattice: a slab computes the spatial sums of one slice twice)
  const size_t kCap = std::max(size_t(256) << 20, (size_t)g.V * 144);
  const int S = g.stride[3];
  // whole lattice, or slabs of nt slices and the one after
  int nt = g.L[3];
  bool full = kSite * g.V <= kCap;
  if (!full) nt = (int)std::max<size_t>(1, std::min<size_t>(g.L[3] - 1, kCap / (kSite * S) > 1 ? kCap / (kSite * S) - 1 : 1));
  const int sites = full ? g.V : (nt + 1) * S;
  // A stream that is being captured, or a device without room for the
  // workspace, takes the kernel that needs none.
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const bool plain = cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
  double2* F = nullptr;
  cudaMemPool_t pool = plain ? nullptr : lib_pool();
  if (!pool || cudaMallocFromPoolAsync((void**)&F, kSite * sites, pool, st) != cudaSuccess) {
    cudaGetLastError();
    const long long grid = ((long long)g.V + kHcSites - 1) / kHcSites;
    hypercube_kernel<<<(unsigned)grid, 64, 0, st>>>(g, GaugeC64{U}, W);
    note_launches(1);
  } else {
    for (int t0 = 0; t0 < g.L[3]; t0 += nt) {
      const int m = std::min(nt, g.L[3] - t0), ms = full ? g.V : (m + 1) * S;
      two_link_kernel<<<dim3((unsigned)((3LL * ms + 127) / 128), 12), 128, 0, st>>>(g, GaugeC64{U}, F, t0, m, ms);
      pair_products_kernel<<<(unsigned)((24LL * m * S + 127) / 128), 128, 0, st>>>(g, F, W, t0, m, ms, full);
      note_launches(2);
    }
    cudaFreeAsync(F, st);
  }
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? 0 : cuda_fail(e);
}

}  // namespace swc
