// CG iterations of the mixed modes on small lattices: one cooperative launch
// runs many iterations of every running system.
//
// On a lattice that a few hundred warps hold, an iteration is latency: the
// launches of its kernels, three reductions finished by a last block each, and
// one thread's chain of hops (8^4, one staggered Wilson system: 13 + 14 + 3 us
// of kernels and 15 us between them; 6x10x12x14 Wilson 12 + 13 + 3 and 16).
// Here a few lanes of a warp share a site, each holding the gauge matrices of
// its share of the hops in registers for the whole launch, and an iteration is
// three phases of all blocks with a barrier after each:
//   t = (D+m) p, |t|^2  |  r -= alpha (D+m)^+ t, |r|^2  |  x += alpha p, p = r + beta p
// (even-odd operator: the odd-site pass of each stencil is a phase of its own).
// Every block adds up all tile sums itself, in the same order, and follows the
// systems' states in shared memory, so no block waits for another's scalar.
//
// Wilson: 2 lanes a site (16 sites a warp): half 0 holds the 4 forward links,
// half 1 the 4 adjoint backward links (72 registers); after the exchange half 0
// has spins 0, 1 and half 1 spins 2, 3.  Staggered Wilson: 4 lanes a site (8
// sites a warp): lane q holds the hops +-q and the corners +-s_2q, +-s_(2q+1)
// (108 registers) and applies them to a pair of systems; it ends with 3 of the
// pair's 12 real numbers.  Signs and phases are folded into the matrices; the
// corners' coefficient r/16 is applied to their sum, before the hops are added
// (folded into the FP32 matrices and accumulated last it made the operator's
// error 1.7 times that of the kernels of larger lattices).
//
// Used for lattices whose warps are all resident at once, at most 12 an SM
// (168 registers a thread; up to 8 warps and with a group of blocks for every
// system 255, all hops' loads under way at once); the blocks of a group of
// systems wait on one another only, and the launch is cooperative, so they are
// resident together.
// A wait gives up after SW_PARAM_WAIT_POLLS polls: the launch ends, and the
// group's systems end without a result (ST_GAVE_UP, SW_ERR_TIMEOUT to the caller).
//
// An iteration of one system takes 12-14 us, of which the hops are 4, the FP64
// sums and divisions 3-4 and the fences and inboxes 5.  Measured against the
// kernels of larger lattices on whole chunks: one system to 1e-10, 8^4 staggered
// Wilson 2.87 -> 1.0 ms, 6x10x12x14 Wilson 5.40 -> 2.2; 12 systems gain 1.04-2.2;
// 48 are near parity (their FP64 updates run alone here), Wilson to 1e-8: 8^4 13.4
// / 13.2 ms, 6x10x12x14 26.5 / 26.5, 12^4 41.9 / 43.5, 12^3x16 54.3 / 53.2.
//
// The tiles of the reductions depend on the volume only, so a system's
// results are the same alone and in any batch.
#pragma once
#include <algorithm>

#include "cg_kernels.cuh"
#include "epochs.h"
#include "internal.h"

namespace swc {

constexpr int kSmallThreads = 384;  // largest block: 12 warps of 168 registers
constexpr int kSmallWide = 256;     // largest block of the 255-register form
// Smallest block: fewer warps a block make more blocks that each follow every
// system of their group (8^4, 48 Wilson systems: 18.7 ms with 2 warps, 16.4
// with 4, 15.8 with 6, 15.4 with 12), more of them leave one system's sites to
// few SMs (4^3x8: 1.79, 1.77, 1.79, 2.15 ms).  At least 32 sites a block, for the
// room of the inboxes.
constexpr int kSmallWarps = 6;
constexpr int kSmallShare = 64;     // systems a group of blocks holds
constexpr double kSmallFetch = 1 << 27;  // bytes of the running systems' vectors from which they are fetched ahead
constexpr int kSmallIters = 512;    // iterations a launch at most
static_assert(5 * kSmallIters < BarrierEpochs::kLaunch, "epochs of a launch (even-odd: 5 an iteration)");

// Units (systems, or pairs of them) that run, in order: list[0] = their
// number, list[1 + i] = (unit << 2) | mask of the unit's systems; systems in
// ST_READY are set RUNNING first.  Also clears the groups' "gave up" words.
// One block.
static __global__ void __launch_bounds__(256) build_list(int nsys, SysState* S, int* list, unsigned* bad, int groups,
                                                         int per) {
  __shared__ int wcnt[8];
  const int units = (nsys + per - 1) / per, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < groups; i += blockDim.x) bad[i] = 0u;
  int base = 0;
  for (int u0 = 0; u0 < units; u0 += 256) {
    const int u = u0 + threadIdx.x;
    int mask = 0;
    if (u < units)
      for (int s = 0; s < per; ++s) {
        const int sys = u * per + s;
        if (sys >= nsys) break;
        if (S[sys].status == ST_READY) S[sys].status = ST_RUNNING;
        if (S[sys].status == ST_RUNNING) mask |= 1 << s;
      }
    const unsigned b = __ballot_sync(0xffffffffu, mask != 0);
    if (lane == 0) wcnt[w] = __popc(b);
    __syncthreads();
    int at = base, tot = 0;
    for (int k = 0; k < 8; ++k) {
      if (k < w) at += wcnt[k];
      tot += wcnt[k];
    }
    if (mask) list[1 + at + __popc(b & ((1u << lane) - 1u))] = (u << 2) | mask;
    base += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) list[0] = base;
}

struct SmallArgs {
  const int* list;
  SysState* S;
  RedBuf rb;
  BatchParams bp;
  int nsys;
  unsigned long long* slots;  // [2][boxes][tiles][tiles][2] each block's inbox: tagged halves of the tile sums
  int boxes;                  // nsys, or kSmallShare a group where that is less
  unsigned* flags;            // [groups][tiles][tiles] each block's inbox: barrier epochs
  unsigned* bad;              // [groups] "gave up"
  unsigned epoch;             // above every epoch of the launches before
  int window, windows;        // this launch's part of the list
  int polls;                  // polls after which a wait gives up
  int iters;                  // iterations at most
  int fetch;                  // the vectors of the running systems exceed L2: prefetch the next system's
};

// ---------------------------------------------------------------- the group's state and barriers
struct SmallShared {
  SysState st[kSmallShare];
  int sys[kSmallShare];  // -1: no system
  int on[kSmallShare];   // still running
  float alpha[kSmallShare], beta[kSmallShare], mass[kSmallShare];
  double wsum[kSmallShare][kSmallThreads / 32];
  int ok;  // no wait has given up
};

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v, unsigned long long w) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(v), "l"(w) : "memory");
}
__device__ __forceinline__ void ld_relaxed(const unsigned long long* p, unsigned long long& v, unsigned long long& w) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v), "=l"(w) : "l"(p) : "memory");
}
__device__ __forceinline__ unsigned ld_relaxed(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// one more poll in vain: whether to give up
__device__ __forceinline__ bool give_up(const SmallArgs& a, SmallShared& s, int& n) {
  if (++n <= a.polls && ((n & 255) || !ld_relaxed(a.bad + blockIdx.y))) return false;
  atomicExch(a.bad + blockIdx.y, 1u);
  s.ok = 0;
  return true;
}

constexpr int kPolls = 5;  // tiles a lane polls at once (160 a warp)

// All blocks of the group (blockIdx.y) have reached `epoch`, and their stores
// before it are visible; false: gave up.
__device__ __forceinline__ bool group_barrier(const SmallArgs& a, SmallShared& s, unsigned& epoch) {
  ++epoch;
  __syncthreads();
  if (threadIdx.x < 32) {
    const int nt = gridDim.x;
    unsigned* f = a.flags + (size_t)blockIdx.y * nt * nt;
    fence_gpu();
    for (int i = threadIdx.x; i < nt; i += 32)
      asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(f + (size_t)i * nt + blockIdx.x), "r"(epoch) : "memory");
    f += (size_t)blockIdx.x * nt;
    int n = 0;
    for (int i0 = threadIdx.x; i0 < nt; i0 += 32 * kPolls) {
      for (;;) {
        unsigned v[kPolls];
#pragma unroll
        for (int k = 0; k < kPolls; ++k) v[k] = i0 + 32 * k < nt ? ld_relaxed(f + i0 + 32 * k) : epoch;
        bool all = true;
#pragma unroll
        for (int k = 0; k < kPolls; ++k) all &= (int)(v[k] - epoch) >= 0;
        if (all || give_up(a, s, n)) break;
      }
    }
    __syncwarp();
    fence_gpu();
  }
  __syncthreads();
  return s.ok != 0;
}

// A barrier that carries the phase's sums: each block posts its sum of every
// running system (two 64-bit words, each half of the double tagged with the
// epoch) into every block's inbox, waits for all tiles' words in its own and
// adds them in the same order -- one trip through L2 where a counter, its polls
// and the reading of the sums take three, and no line that all blocks poll
// (126 blocks polling one array of words held its writers up by 6 us).  Then
// each block moves its copy of the states on (block 0 records the
// coefficients).  The slots of a phase are written again only after every block
// has passed a later barrier.
// The slots of system t of the group: by its number in the batch, or by the
// group's t where the batch takes several launches (whose words the epochs tell apart).
__device__ __forceinline__ size_t box(const SmallArgs& a, const SmallShared& s, int t) {
  return a.boxes < a.nsys ? blockIdx.y * kSmallShare + t : s.sys[t];
}
template <int PHASE>
__device__ __forceinline__ bool exchange(const SmallArgs& a, SmallShared& s, int share, unsigned& epoch) {
  ++epoch;
  __syncthreads();
  const int nw = blockDim.x >> 5, lane = threadIdx.x & 31, nt = gridDim.x;
  const unsigned long long tag = (unsigned long long)epoch << 32;
  unsigned long long* slots = a.slots + (size_t)(PHASE - 1) * a.boxes * nt * nt * 2;
  // The block's stores, before any of its words: by every warp that posts, before
  // its first word, whichever of its systems that is of.  (After the sum: the
  // stores drain meanwhile; a fence before it cost 0.25 us an exchange.)
  bool fenced = false;
  for (int t = threadIdx.x >> 5; t < share; t += nw) {
    if (!s.on[t]) continue;
    double v = s.wsum[t][0];
    for (int w = 1; w < nw; ++w) v += s.wsum[t][w];
    if (!fenced) fence_gpu();
    fenced = true;
    const unsigned long long hi = tag | (unsigned)__double2hiint(v), lo = tag | (unsigned)__double2loint(v);
    unsigned long long* w = slots + (box(a, s, t) * nt * nt + blockIdx.x) * 2;
    for (int i = lane; i < nt; i += 32) st_relaxed(w + (size_t)i * nt * 2, hi, lo);
  }
  int n = 0;
  for (int t = threadIdx.x >> 5; t < share; t += nw) {
    if (!s.on[t]) continue;
    const unsigned long long* p = slots + (box(a, s, t) * nt + blockIdx.x) * nt * 2;
    double v = 0.0;
    for (int i0 = lane; i0 < nt; i0 += 32 * kPolls) {
      unsigned long long hi[kPolls], lo[kPolls];
      for (;;) {
#pragma unroll
        for (int k = 0; k < kPolls; ++k) {
          hi[k] = lo[k] = tag;
          if (i0 + 32 * k < nt) ld_relaxed(p + 2 * (i0 + 32 * k), hi[k], lo[k]);
        }
        bool all = true;
#pragma unroll
        for (int k = 0; k < kPolls; ++k) all &= (hi[k] >> 32) == epoch && (lo[k] >> 32) == epoch;
        if (all || give_up(a, s, n)) break;
      }
#pragma unroll
      for (int k = 0; k < kPolls; ++k)
        if (i0 + 32 * k < nt) v += __hiloint2double((int)(unsigned)hi[k], (int)(unsigned)lo[k]);
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) s.wsum[t][0] = v;
  }
  fence_gpu();
  __syncthreads();
  // one thread a system: the divisions of all systems at once (after a wait that
  // gave up, of incomplete sums: not recorded, and the states stay in the block)
  RedBuf rb = a.rb;
  if (blockIdx.x || !s.ok) rb.hist = nullptr;
  for (int t = threadIdx.x; t < share; t += blockDim.x) {
    if (!s.on[t]) continue;
    SysState& st = s.st[t];
    if (PHASE == 1) {
      finish_k1(st, rb, s.sys[t], s.wsum[t][0]);
      s.alpha[t] = (float)st.alpha;
    } else {
      finish_k2(st, rb, s.sys[t], s.wsum[t][0]);
      s.beta[t] = (float)st.beta;
    }
    if (st.status != ST_RUNNING) s.on[t] = 0;
  }
  __syncthreads();
  return s.ok != 0;
}

// The group's part of the list -> shared memory; returns its size (systems).
__device__ __forceinline__ int load_share(const SmallArgs& a, SmallShared& s, int per) {
  // every parts-th unit: neighbours in the batch often stop together (one mass),
  // and a group whose systems stop at different iterations keeps its SMs busy
  const int cnt = a.list[0], parts = a.windows * gridDim.y, part = a.window * gridDim.y + blockIdx.y;
  const int n = part < cnt ? (cnt - part - 1) / parts + 1 : 0;
  for (int t = threadIdx.x; t < n * per; t += blockDim.x) {
    const int e = a.list[1 + part + (t / per) * parts], sys = (e >> 2) * per + t % per;
    const bool run = (e >> (t % per)) & 1;
    s.sys[t] = run ? sys : -1;
    s.on[t] = run;
    s.alpha[t] = s.beta[t] = s.mass[t] = 0.f;
    if (run) {
      s.st[t] = a.S[sys];
      s.mass[t] = (float)s.st[t].mass;
    }
  }
  if (threadIdx.x == 0) s.ok = 1;
  __syncthreads();
  return n * per;
}

// End of an iteration: whether the group goes on (half of its systems have
// stopped, or none is left: a reliable update is due).
__device__ __forceinline__ bool group_goes_on(const SmallShared& s, int share) {
  int on = 0, all = 0;
  for (int t = 0; t < share; ++t) {
    on += s.on[t];
    all += s.sys[t] >= 0;
  }
  return on > 0 && 2 * on > all;
}

// The group's states at the launch's end, by its block 0: what the iterations
// change, and the status where it is still the one the launch found.  A block
// whose wait gave up ends its group's systems, whatever the other blocks make of
// them: block 0 may have passed its last wait before another gave up in its own.
__device__ __forceinline__ void store_states(const SmallArgs& a, const SmallShared& s, int share, bool gave_up) {
  __syncthreads();
  if (!gave_up && blockIdx.x) return;
  for (int t = threadIdx.x; t < share; t += blockDim.x) {
    if (s.sys[t] < 0) continue;
    SysState& g = a.S[s.sys[t]];
    if (gave_up) {
      atomicExch(&g.status, ST_GAVE_UP);
      continue;
    }
    const SysState& l = s.st[t];
    g.rr = l.rr, g.rr_old = l.rr_old, g.pAp = l.pAp, g.alpha = l.alpha, g.beta = l.beta, g.rmax2 = l.rmax2;
    g.iter = l.iter;
    atomicCAS(&g.status, ST_RUNNING, l.status);
  }
}

// The FP64 sum of a warp's FP32 norms (NV lanes a system), lane l with l ^ 1,
// then ^ 2, ^ 4, ...  For up to 8 systems at once 4 lanes a system add NV / 4
// values each (the FP64 pipe takes 64 clocks a warp's instruction: 17 of them
// for 8 systems, or 5 a system by the tree of shuffles, which is therefore
// taken for one or two systems).  Both add in the same order.
template <int NV> struct NormBuf { float v[8][NV + 1]; };
template <int NV>
__device__ __forceinline__ void flush_norms(NormBuf<NV>& b, SmallShared& sh, int slot0, int nslot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncwarp();
  if (nslot <= 2) {
    if (NV == 32 || nslot == 1) {
      for (int s = 0; s < nslot; ++s) {
        double a = (double)b.v[s][lane % NV];
#pragma unroll
        for (int o = 1; o < NV; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) sh.wsum[slot0 + s][warp] = a;
      }
    } else {  // two systems, 16 lanes each
      double a = (double)b.v[lane / NV][lane % NV];
#pragma unroll
      for (int o = 1; o < NV; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane % NV == 0) sh.wsum[slot0 + lane / NV][warp] = a;
    }
  } else {
    const int s = lane >> 2, q = lane & 3;
    double a[NV / 4];
#pragma unroll
    for (int j = 0; j < NV / 4; ++j) a[j] = (double)b.v[s][q * (NV / 4) + j];
#pragma unroll
    for (int o = 1; o < NV / 4; o <<= 1)
#pragma unroll
      for (int j = 0; j < NV / 4; j += 2 * o) a[j] += a[j + o];
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
    if (q == 0 && s < nslot) sh.wsum[slot0 + s][warp] = a[0];
  }
  __syncwarp();
}

// ---------------------------------------------------------------- Wilson
// Spinors of the storages (plain loads: other blocks write them between the
// launch's phases).
template <class V> struct SpinorIO;
template <> struct SpinorIO<VecP32q<12>> {
  // a warp's 16 sites from n0 (12 lines) into L2
  __device__ static __forceinline__ void prefetch(const VecP32q<12>& v, int n0, int lane) {
    if (lane < 12) asm volatile("prefetch.global.L2 [%0];" ::"l"(v.p + pk(n0, 6, 0) + lane * 8));
  }
  struct Raw { float4 q[6]; };
  __device__ static __forceinline__ unsigned offset(int n) { return (unsigned)pk(n, 6, 0); }
  __device__ static __forceinline__ Raw load(const VecP32q<12>& v, unsigned off, int) {
    Raw r;
#pragma unroll
    for (int k = 0; k < 6; ++k) r.q[k] = v.p[off + k * 16];
    return r;
  }
  __device__ static __forceinline__ Sp<float> unpack(const Raw& r) {
    Sp<float> p;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int c0 = 2 * k, c1 = 2 * k + 1;
      p.s[c0 / 3].c[c0 % 3] = {r.q[k].x, r.q[k].y};
      p.s[c1 / 3].c[c1 % 3] = {r.q[k].z, r.q[k].w};
    }
    return p;
  }
  // the 12 real numbers of spins 0, 1 (half 0) or 2, 3 (half 1)
  __device__ static __forceinline__ void load_half(const VecP32q<12>& v, int n, int half, float o[12]) {
    const float4* b = v.p + pk(n, 6, 3 * half);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float4 w = b[k * 16];
      o[4 * k] = w.x, o[4 * k + 1] = w.y, o[4 * k + 2] = w.z, o[4 * k + 3] = w.w;
    }
  }
  __device__ static __forceinline__ void store_half(const VecP32q<12>& v, int n, int half, bool on, const float o[12]) {
    if (!on) return;
    float4* b = v.p + pk(n, 6, 3 * half);
#pragma unroll
    for (int k = 0; k < 3; ++k) b[k * 16] = make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
  }
};
template <> struct SpinorIO<VecP16<12>> {
  struct Raw { uint4 q[3]; float s; };
  __device__ static __forceinline__ unsigned offset(int n) { return (unsigned)pk(n, 3, 0); }
  __device__ static __forceinline__ Raw load(const VecP16<12>& v, unsigned off, int n) {
    Raw r;
#pragma unroll
    for (int k = 0; k < 3; ++k) r.q[k] = reinterpret_cast<const uint4*>(v.p)[off + k * 16];
    r.s = v.scale(n);
    return r;
  }
  __device__ static __forceinline__ Sp<float> unpack(const Raw& r) {
    Sp<float> p;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const unsigned u[4] = {r.q[k].x, r.q[k].y, r.q[k].z, r.q[k].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 4 * k + j;
        p.s[c / 3].c[c % 3] = r.s * half2_of(u[j]);
      }
    }
    return p;
  }
  __device__ static __forceinline__ uint2* pair(const VecP16<12>& v, int n, int c) {  // components c, c + 1 (c even)
    return reinterpret_cast<uint2*>(v.p) + pk(n, 3, c >> 2) * 2 + ((c >> 1) & 1);
  }
  __device__ static __forceinline__ void load_half(const VecP16<12>& v, int n, int half, float o[12]) {
    const float s = v.scale(n);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint2 u = *pair(v, n, 6 * half + 2 * k);
      const cx<float> a0 = s * half2_of(u.x), a1 = s * half2_of(u.y);
      o[4 * k] = a0.re, o[4 * k + 1] = a0.im, o[4 * k + 2] = a1.re, o[4 * k + 3] = a1.im;
    }
  }
  __device__ static __forceinline__ void store_half(const VecP16<12>& v, int n, int half, bool on, const float o[12]) {
    float m = 0.f, inv;
#pragma unroll
    for (int k = 0; k < 12; ++k) m = fmaxf(m, fabsf(o[k]));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    if (!on) return;
    half_scale(m, inv);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const __half2 h0 = __floats2half2_rn(o[4 * k] * inv, o[4 * k + 1] * inv);
      const __half2 h1 = __floats2half2_rn(o[4 * k + 2] * inv, o[4 * k + 3] * inv);
      uint2 u;
      memcpy(&u.x, &h0, 4);
      memcpy(&u.y, &h1, 4);
      *pair(v, n, 6 * half + 2 * k) = u;
    }
    if (half == 0) v.scale(n) = m;
  }
};

// Where the sites and neighbours are: the whole lattice, or the sites of one
// parity with half-index vectors on the links of the whole lattice.
template <class GG> struct FullSites {
  static constexpr bool kEO = false;
  GG g;
  __device__ __forceinline__ int count() const { return g.V; }
  // this lane's neighbours (forward: half 0): sites of the links, vector
  // indices, time boundary sign
  __device__ __forceinline__ void neighbours(int n, int, int half, int li[4], int vi[4], bool* flip) const {
    int x[4];
    coords(g, n, x);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int y = hop(g, n, x, mu, half ? -1 : +1);
      li[mu] = half ? y : n;
      vi[mu] = y;
    }
    *flip = bc_flip(g, x, half ? -1 : +1);
  }
};
// Full index and coordinates of half-lattice site h of parity `par`.
__device__ __forceinline__ int half_site(const Geom& g, int h, int par, int x[4]) {
  coords(g, 2 * h, x);
  const int b = ((x[1] + x[2] + x[3]) & 1) ^ par;  // x0 of site 2h is even
  x[0] += b;
  return 2 * h + b;
}
struct HalfSites {
  static constexpr bool kEO = true;
  Geom g;  // the whole lattice
  __device__ __forceinline__ int count() const { return g.V / 2; }
  __device__ __forceinline__ void neighbours(int h, int par, int half, int li[4], int vi[4], bool* flip) const {
    int x[4];
    const int n = half_site(g, h, par, x);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int y = hop(g, n, x, mu, half ? -1 : +1);
      li[mu] = half ? y : n;
      vi[mu] = y >> 1;
    }
    *flip = bc_flip(g, x, half ? -1 : +1);
  }
};

// scratch: units from a system's vector to its scratch (even-odd operator)
template <int MAXT, bool R1, class Sites, class GA, class VI>
__global__ void __launch_bounds__(MAXT, 1)
    wilson_small(Sites sites, GA U, VI p, VI t, VecP32q<12> r, VecP32q<12> x, size_t scratch, SmallArgs a) {
  using IO = SpinorIO<VI>;
  using RO = SpinorIO<VecP32q<12>>;
  constexpr bool kEO = Sites::kEO;
  __shared__ SmallShared s;
  __shared__ NormBuf<32> nbuf[kSmallThreads / 32];
  const int share = load_share(a, s, 1);
  if (share == 0) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, half = lane >> 4;
  const int V = sites.count();
  const int nn = (blockIdx.x * (blockDim.x >> 5) + warp) * 16 + (lane & 15);
  const bool on = nn < V;
  const int n = on ? nn : V - 1;  // lanes beyond the lattice compute its last site and store nothing
  M3<float> L[4];
  int vi[4];
  unsigned off[4];
  auto load_links = [&](int par) {
    int li[4];
    bool flip;
    sites.neighbours(n, par, half, li, vi, &flip);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      L[mu] = U.link(li[mu], mu);
      if (half) L[mu] = dag(L[mu]);
      off[mu] = IO::offset(vi[mu]);
    }
    if (flip) {
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) L[3].e[i][j] = {-L[3].e[i][j].re, -L[3].e[i][j].im};
    }
  };
  const float rw = (float)a.bp.r;
  // this lane's part of the hops' sum: spins 0, 1 (half 0) or 2, 3 (half 1)
  auto hops = [&](const VI& in, bool dagger, float o[12]) {
    const float sg = (half != 0) == dagger ? 1.f : -1.f;  // (r - sg g_mu): 1 forward, -1 backward, the reverse for the adjoint
    Sp<float> acc;
#pragma unroll
    for (int k = 0; k < 4; ++k) acc.s[k] = zero3<float>();
    constexpr int kAhead = MAXT <= kSmallWide ? 4 : 1;  // hops whose loads are under way: all of them where registers allow
    typename IO::Raw raw[4];
#pragma unroll
    for (int mu = 0; mu < kAhead; ++mu) raw[mu] = IO::load(in, off[mu], vi[mu]);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const Sp<float> q = IO::unpack(raw[mu]);
      if (mu + kAhead < 4) raw[mu + kAhead] = IO::load(in, off[mu + kAhead], vi[mu + kAhead]);
      if constexpr (R1) {
        V3<float> h0, h1;
        wproject(mu, sg, q, h0, h1);
        wreconstruct(mu, sg, mv(L[mu], h0), mv(L[mu], h1), acc);
      } else {
        Sp<float> f;
#pragma unroll
        for (int k = 0; k < 4; ++k) f.s[k] = mv(L[mu], q.s[k]);
        wgeneral(mu, sg, rw, f, acc);
      }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const cx<float> up = acc.s[k / 3].c[k % 3], dn = acc.s[2 + k / 3].c[k % 3];
      o[2 * k] = (half ? dn.re : up.re) + __shfl_xor_sync(0xffffffffu, half ? up.re : dn.re, 16);
      o[2 * k + 1] = (half ? dn.im : up.im) + __shfl_xor_sync(0xffffffffu, half ? up.im : dn.im, 16);
    }
  };
  auto aside = [&](VI v) {
    v.p += scratch;
    return v;
  };
  // The system after k whose lines are to be fetched ahead (-1: none).  A system's
  // turn in a phase is latency, of which its own and its neighbours' first loads
  // from memory are the most where the batch's vectors exceed L2; each block
  // fetches its own sites.  FP32 spinors from kSmallFetch bytes of p, t, r and x, a
  // solve to 1e-8 of 48 systems, without / with: 6x10x12x14 27.2 / 26.6 ms, 12^4
  // 46.1 / 43.7, 12^3x16 56.7 / 53.3; below, 8^4 13.2 / 13.5, 12^3x16 with 12
  // systems 15.75 / 15.79.  FP16 storage (half the bytes) and the even-odd
  // operator (its scratch is read, too) gain less than they lose: 36.2 / 37.8 and
  // 61.6 / 62.5.  (The wide form holds a system a block: it has no next one.)
  constexpr bool kFetch = MAXT > kSmallWide && !kEO && std::is_same<VI, VecP32q<12>>::value;
  const int n0 = nn - (lane & 15);
  auto next = [&](int k) {
    return kFetch && a.fetch && k + 1 < share && n0 < V && s.on[k + 1] ? s.sys[k + 1] : -1;
  };
  unsigned epoch = a.epoch;
  // even-odd: u = D_oe v of every running system into v's scratch
  auto odd_pass = [&](const VI& v, bool dagger) {
    load_links(1);
    for (int k = 0; k < share; ++k) {
      if (!s.on[k]) continue;
      const VI w = sys_view(v, s.sys[k], a.bp.vstride);
      float o[12];
      hops(w, dagger, o);
#pragma unroll
      for (int c = 0; c < 12; ++c) o[c] *= -0.5f;
      IO::store_half(aside(w), n, half, on, o);
    }
    if (!group_barrier(a, s, epoch)) return false;
    load_links(0);
    return true;
  };
  if constexpr (!kEO) load_links(0);
  bool ok = true;
  for (int it = 0; it < a.iters; ++it) {
    if constexpr (kEO)
      if (!(ok = odd_pass(p, false))) break;
#pragma unroll 1
    for (int k = 0; k < share; ++k) {
      if (s.on[k]) {
        const VI w = sys_view(p, s.sys[k], a.bp.vstride);
        float o[12], own[12];
        if constexpr (kFetch)
          if (const int f = next(k); f >= 0) IO::prefetch(sys_view(p, f, a.bp.vstride), n0, lane);
        IO::load_half(w, n, half, own);
        hops(kEO ? aside(w) : w, false, o);
        const float M = 4.f * rw + s.mass[k], c = kEO ? 0.5f / M : -0.5f;
        float s2 = 0.f;
#pragma unroll
        for (int i = 0; i < 12; ++i) {
          o[i] = fmaf(M, own[i], c * o[i]);
          s2 = fmaf(o[i], o[i], s2);
        }
        IO::store_half(sys_view(t, s.sys[k], a.bp.vstride), n, half, on, o);
        nbuf[warp].v[k & 7][lane] = on ? s2 : 0.f;
      }
      if ((k & 7) == 7 || k == share - 1) flush_norms<32>(nbuf[warp], s, k & ~7, (k & 7) + 1);
    }
    if (!(ok = exchange<1>(a, s, share, epoch))) break;
    if constexpr (kEO)
      if (!(ok = odd_pass(t, true))) break;
#pragma unroll 1
    for (int k = 0; k < share; ++k) {
      if (s.on[k]) {
        const VI w = sys_view(t, s.sys[k], a.bp.vstride);
        const VecP32q<12> rs = sys_view(r, s.sys[k], a.bp.sstride);
        float o[12], own[12], rv[12];
        if constexpr (kFetch)
          if (const int f = next(k); f >= 0) {
            IO::prefetch(sys_view(t, f, a.bp.vstride), n0, lane);
            RO::prefetch(sys_view(r, f, a.bp.sstride), n0, lane);
          }
        RO::load_half(rs, n, half, rv);
        IO::load_half(w, n, half, own);
        hops(kEO ? aside(w) : w, true, o);
        const float M = 4.f * rw + s.mass[k], c = kEO ? 0.5f / M : -0.5f, al = s.alpha[k];
        float s2 = 0.f;
#pragma unroll
        for (int i = 0; i < 12; ++i) {
          o[i] = fmaf(-al, fmaf(M, own[i], c * o[i]), rv[i]);
          s2 = fmaf(o[i], o[i], s2);
        }
        RO::store_half(rs, n, half, on, o);
        nbuf[warp].v[k & 7][lane] = on ? s2 : 0.f;
      }
      if ((k & 7) == 7 || k == share - 1) flush_norms<32>(nbuf[warp], s, k & ~7, (k & 7) + 1);
    }
    if (!(ok = exchange<2>(a, s, share, epoch))) break;
    const bool more = group_goes_on(s, share);
#pragma unroll 1
    for (int k = 0; k < share; ++k) {
      if (!s.on[k]) continue;  // (a stopped system's x is brought up to date by its reliable update)
      const VI w = sys_view(p, s.sys[k], a.bp.vstride);
      const VecP32q<12> xs = sys_view(x, s.sys[k], a.bp.sstride);
      float pv[12], xv[12], rv[12];
      if constexpr (kFetch)
        if (const int f = next(k); f >= 0) {
          IO::prefetch(sys_view(p, f, a.bp.vstride), n0, lane);
          RO::prefetch(sys_view(x, f, a.bp.sstride), n0, lane);
          RO::prefetch(sys_view(r, f, a.bp.sstride), n0, lane);
        }
      IO::load_half(w, n, half, pv);
      RO::load_half(xs, n, half, xv);
      RO::load_half(sys_view(r, s.sys[k], a.bp.sstride), n, half, rv);
      const float al = s.alpha[k], be = s.beta[k];
#pragma unroll
      for (int i = 0; i < 12; ++i) {
        xv[i] = fmaf(al, pv[i], xv[i]);
        pv[i] = fmaf(be, pv[i], rv[i]);
      }
      RO::store_half(xs, n, half, on, xv);
      IO::store_half(w, n, half, on, pv);
    }
    if (!more) break;
    if (!(ok = group_barrier(a, s, epoch))) break;
  }
  store_states(a, s, share, !ok);
}

// ---------------------------------------------------------------- staggered Wilson
// A pair's colour vectors at a site.
template <class V> struct PairIO;
template <> struct PairIO<VecP32x2<3>> {
  struct Raw { float4 c[3]; };
  struct View { float4* b; };
  __device__ static __forceinline__ View view(const VecP32x2<3>& v, int s0, int, size_t stride) {
    return {v.p + (size_t)s0 * stride};  // s0 even
  }
  __device__ static __forceinline__ unsigned offset(int n) { return (unsigned)pk(n, 3, 0); }
  __device__ static __forceinline__ Raw load(const View& v, unsigned off) {
    Raw r;
#pragma unroll
    for (int c = 0; c < 3; ++c) r.c[c] = v.b[off + c * 16];
    return r;
  }
  __device__ static __forceinline__ void unpack(const Raw& r, V3<float> v[2]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      v[0].c[c] = {r.c[c].x, r.c[c].z};
      v[1].c[c] = {r.c[c].y, r.c[c].w};
    }
  }
  // the real (part 0) or imaginary (part 1) parts of system s of the pair at site n
  __device__ static __forceinline__ void load_part(const View& v, int n, int s, int part, float o[3]) {
    const float* f = reinterpret_cast<const float*>(v.b + pk(n, 3, 0)) + part * 2 + s;
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c] = f[c * 64];
  }
  __device__ static __forceinline__ void store_part(const View& v, int n, int s, int part, bool on, const float o[3]) {
    if (!on) return;
    float* f = reinterpret_cast<float*>(v.b + pk(n, 3, 0)) + part * 2 + s;
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c * 64] = o[c];
  }
};
template <> struct PairIO<VecP16<3>> {
  struct Raw { uint4 s[2]; };
  struct View { uint4* b[2]; };
  // a pair of which one system runs reads that one twice (the other may be beyond the batch)
  __device__ static __forceinline__ View view(const VecP16<3>& v, int s0, int mask, size_t stride) {
    uint4* b = reinterpret_cast<uint4*>(v.p);
    const size_t u = stride / 4;  // 16-byte units of a system
    return {{b + (size_t)(s0 + ((mask & 1) ? 0 : 1)) * u, b + (size_t)(s0 + ((mask & 2) ? 1 : 0)) * u}};
  }
  __device__ static __forceinline__ unsigned offset(int n) { return (unsigned)n; }
  __device__ static __forceinline__ Raw load(const View& v, unsigned off) { return {{v.b[0][off], v.b[1][off]}}; }
  __device__ static __forceinline__ void unpack(const Raw& r, V3<float> v[2]) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const unsigned u[3] = {r.s[s].x, r.s[s].y, r.s[s].z};
      const float sc = __uint_as_float(r.s[s].w);
#pragma unroll
      for (int c = 0; c < 3; ++c) v[s].c[c] = sc * half2_of(u[c]);
    }
  }
  __device__ static __forceinline__ void load_part(const View& v, int n, int s, int part, float o[3]) {
    const uint4 w = v.b[s][n];
    const unsigned u[3] = {w.x, w.y, w.z};
    const float sc = __uint_as_float(w.w);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const cx<float> z = half2_of(u[c]);
      o[c] = sc * (part ? z.im : z.re);
    }
  }
  __device__ static __forceinline__ void store_part(const View& v, int n, int s, int part, bool on, const float o[3]) {
    float m = fmaxf(fmaxf(fabsf(o[0]), fabsf(o[1])), fabsf(o[2])), im[3], inv;
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 8));
#pragma unroll
    for (int c = 0; c < 3; ++c) im[c] = __shfl_xor_sync(0xffffffffu, o[c], 8);
    if (!on || part) return;
    half_scale(m, inv);
    unsigned u[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const __half2 h = __floats2half2_rn(o[c] * inv, im[c] * inv);
      memcpy(&u[c], &h, 4);
    }
    v.b[s][n] = make_uint4(u[0], u[1], u[2], __float_as_uint(m));
  }
};

__device__ __forceinline__ M3<float> scaled(float c, const M3<float>& A) {
  M3<float> B;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) B.e[i][j] = {c * A.e[i][j].re, c * A.e[i][j].im};
  return B;
}

template <int MAXT, class GG, class GA, class TA, class VI>
__global__ void __launch_bounds__(MAXT, 1)
    sw_small(GG g, GA U, TA W, VI p, VI t, VecP32<3> r, VecP32<3> x, SmallArgs a) {
  using IO = PairIO<VI>;
  __shared__ SmallShared s;
  __shared__ NormBuf<16> nbuf[kSmallThreads / 32];
  const int share = load_share(a, s, 2);
  if (share == 0) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane >> 3, sl = lane & 7;
  const int nn = (blockIdx.x * (blockDim.x >> 5) + warp) * 8 + sl;
  const bool on = nn < g.V;
  const int n = on ? nn : g.V - 1;
  const float rw = (float)a.bp.r;
  M3<float> M[6];  // the hops' two matrices (their sign turns for the adjoint), then the corners'
  float hs;        // the corners' coefficient
  unsigned off[6];
  {
    int y[4], df[4], db[4];
    coords(g, n, y);
    hop_deltas(g, n, y, df, db);
    const bool ff = bc_flip(g, y, +1), fb = bc_flip(g, y, -1);
    const int par = (q > 0 ? y[0] : 0) + (q > 1 ? y[1] : 0) + (q > 2 ? y[2] : 0);
    const float eta = (par & 1) ? -0.5f : 0.5f;  // eta_q / 2
    const int dfq = q == 0 ? df[0] : q == 1 ? df[1] : q == 2 ? df[2] : df[3];
    const int dbq = q == 0 ? db[0] : q == 1 ? db[1] : q == 2 ? db[2] : db[3];
    M[0] = scaled(q == 3 && ff ? -eta : eta, U.link(n, q));
    M[1] = scaled(q == 3 && fb ? eta : -eta, dag(U.link(n + dbq, q)));
    off[0] = IO::offset(n + dfq);
    off[1] = IO::offset(n + dbq);
    hs = (eps_eta5_neg(y) ? rw : -rw) * 0.0625f;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int k = 2 * q + j;
      int of, ob;
      corner_offsets(k, df, db, of, ob);
      M[2 + 2 * j] = scaled(ff ? -1.f : 1.f, W.mat(n, k));
      M[3 + 2 * j] = scaled(fb ? -1.f : 1.f, dag(W.mat(n + ob, k)));
      off[2 + 2 * j] = IO::offset(n + of);
      off[3 + 2 * j] = IO::offset(n + ob);
    }
  }
  const int ls = q >> 1, part = q & 1;  // what this lane ends with: system ls of the pair, real or imaginary parts
  // this lane's 3 numbers of sum of the hops and corners
  auto hops = [&](const typename IO::View& in, float o[3]) {
    V3<float> acc[2] = {zero3<float>(), zero3<float>()};
    typename IO::Raw raw[6];
#pragma unroll
    for (int h = 0; h < 6; ++h) raw[h] = IO::load(in, off[h]);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int h = k < 4 ? k + 2 : k - 4;
      if (k == 4) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          acc[0].c[c] = hs * acc[0].c[c];
          acc[1].c[c] = hs * acc[1].c[c];
        }
      }
      V3<float> v[2];
      IO::unpack(raw[h], v);
      mv_acc(acc[0], M[h], v[0]);
      mv_acc(acc[1], M[h], v[1]);
    }
    float kr[3], ki[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const cx<float> a0 = acc[0].c[c], a1 = acc[1].c[c];
      kr[c] = (ls ? a1.re : a0.re) + __shfl_xor_sync(0xffffffffu, ls ? a0.re : a1.re, 16);
      ki[c] = (ls ? a1.im : a0.im) + __shfl_xor_sync(0xffffffffu, ls ? a0.im : a1.im, 16);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c] = (part ? ki[c] : kr[c]) + __shfl_xor_sync(0xffffffffu, part ? kr[c] : ki[c], 8);
  };
  auto adjoint = [&]() {  // the hops change sign between D and D^+
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        M[0].e[i][j] = {-M[0].e[i][j].re, -M[0].e[i][j].im};
        M[1].e[i][j] = {-M[1].e[i][j].re, -M[1].e[i][j].im};
      }
  };
  auto first = [&](int k) { return (s.sys[k] >= 0 ? s.sys[k] : s.sys[k + 1] - 1); };  // the pair's first system
  auto rpart = [&](const VecP32<3>& v, int s0) {
    return reinterpret_cast<float*>(v.p + (size_t)(s0 + ls) * a.bp.sstride + pk(n, 3, 0)) + part;
  };
  unsigned epoch = a.epoch;
  bool ok = true;
  for (int it = 0; it < a.iters; ++it) {
#pragma unroll 1
    for (int k = 0; k < share; k += 2) {
      const int mask = s.on[k] | (s.on[k + 1] << 1);
      if (mask) {
        const int s0 = first(k);
        const typename IO::View vp = IO::view(p, s0, mask, a.bp.vstride);
        float own[3], o[3];
        IO::load_part(vp, n, ls, part, own);
        hops(vp, o);
        const float d = rw + s.mass[k + ls];
#pragma unroll
        for (int c = 0; c < 3; ++c) o[c] = fmaf(d, own[c], o[c]);
        IO::store_part(IO::view(t, s0, 3, a.bp.vstride), n, ls, part, on && ((mask >> ls) & 1), o);
        nbuf[warp].v[(k & 7) + ls][part * 8 + sl] = on ? fmaf(o[0], o[0], fmaf(o[1], o[1], o[2] * o[2])) : 0.f;
      }
      if ((k & 7) == 6 || k == share - 2) flush_norms<16>(nbuf[warp], s, k & ~7, (k & 7) + 2);
    }
    if (!(ok = exchange<1>(a, s, share, epoch))) break;
    adjoint();
#pragma unroll 1
    for (int k = 0; k < share; k += 2) {
      const int mask = s.on[k] | (s.on[k + 1] << 1);
      if (mask) {
        const int s0 = first(k);
        const typename IO::View vt = IO::view(t, s0, mask, a.bp.vstride);
        const bool st = (mask >> ls) & 1;
        float own[3], o[3], rv[3] = {0.f, 0.f, 0.f};
        float* rp = rpart(r, s0);
        if (st) {
#pragma unroll
          for (int c = 0; c < 3; ++c) rv[c] = rp[c * 32];
        }
        IO::load_part(vt, n, ls, part, own);
        hops(vt, o);
        const float d = rw + s.mass[k + ls], al = s.alpha[k + ls];
#pragma unroll
        for (int c = 0; c < 3; ++c) o[c] = fmaf(-al, fmaf(d, own[c], o[c]), rv[c]);
        if (st && on) {
#pragma unroll
          for (int c = 0; c < 3; ++c) rp[c * 32] = o[c];
        }
        nbuf[warp].v[(k & 7) + ls][part * 8 + sl] = on ? fmaf(o[0], o[0], fmaf(o[1], o[1], o[2] * o[2])) : 0.f;
      }
      if ((k & 7) == 6 || k == share - 2) flush_norms<16>(nbuf[warp], s, k & ~7, (k & 7) + 2);
    }
    adjoint();
    if (!(ok = exchange<2>(a, s, share, epoch))) break;
    const bool more = group_goes_on(s, share);
#pragma unroll 1
    for (int k = 0; k < share; k += 2) {
      const int mask = s.on[k] | (s.on[k + 1] << 1);
      if (!mask) continue;
      const int s0 = first(k);
      const typename IO::View vp = IO::view(p, s0, mask, a.bp.vstride);
      const bool st = (mask >> ls) & 1;
      float pv[3];
      IO::load_part(vp, n, ls, part, pv);
      if (st) {
        float *xp = rpart(x, s0), *rp = rpart(r, s0);
        const float al = s.alpha[k + ls], be = s.beta[k + ls];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float xv = fmaf(al, pv[c], xp[c * 32]);
          pv[c] = fmaf(be, pv[c], rp[c * 32]);
          if (on) xp[c * 32] = xv;
        }
      }
      IO::store_part(IO::view(p, s0, 3, a.bp.vstride), n, ls, part, on && st, pv);
    }
    if (!more) break;
    if (!(ok = group_barrier(a, s, epoch))) break;
  }
  store_states(a, s, share, !ok);
}

// ---------------------------------------------------------------- launches
// warps that hold the sites; 0: the operator has no small form
template <class Op> struct small_traits { static constexpr int kSites = 0, kPer = 1; };
template <typename G, typename Wt, template <int> class VA> struct small_traits<SWOp<float, G, Wt, VA>> {
  static constexpr int kSites = 8, kPer = 2;
};
template <typename G, template <int> class VA, bool R1, bool LEAN> struct small_traits<WOp<float, G, VA, R1, LEAN>> {
  static constexpr int kSites = 16, kPer = 1;
};

struct SmallPlan {
  int nt = 0, tiles = 0, groups = 1, windows = 1;
  bool wide = false;
};

// Whether a lattice of V sites (of the operator's vectors) takes the small
// form, and its blocks: as few warps a block as spread the lattice over every
// SM.  By the volume only.
inline bool small_tiles(int V, int sites_per_warp, SmallPlan* p) {
  const int sms = sm_count();
  const long long warps = (V + sites_per_warp - 1) / sites_per_warp;
  if (warps > (long long)sms * (kSmallThreads / 32)) return false;
  int per = (int)((warps + sms - 1) / sms);
  per = std::max(per, kSmallWarps);
  p->nt = 32 * per;
  p->tiles = (int)((warps + per - 1) / per);
  return true;
}

// Scratch of a batch of nsys systems of NC components on V sites: the inboxes'
// 64-bit words, and the ints of the list, the "gave up" words and the barrier
// epochs (0: the lattice does not take the small form).  Bounded by the groups
// resident at once (at most two blocks an SM), so that the workspace of a large
// batch grows by little (8^4 staggered Wilson, 600 systems: 46 MB on 480).
constexpr int small_sites(int NC) { return NC == 3 ? 8 : 16; }  // a warp holds
inline int small_groups(int tiles) { return std::max(1, 2 * sm_count() / tiles); }
inline int small_boxes(int tiles, int nsys) { return std::min(nsys, small_groups(tiles) * kSmallShare); }
inline size_t small_slots(int V, int NC, int nsys) {
  SmallPlan p;
  if (!small_tiles(V, small_sites(NC), &p)) return 0;
  return (size_t)4 * p.tiles * p.tiles * small_boxes(p.tiles, nsys);
}
inline size_t small_words(int V, int NC, int nsys) {
  SmallPlan p;
  if (!small_tiles(V, small_sites(NC), &p)) return 0;
  return 1 + 2 * (size_t)nsys + (size_t)p.tiles * p.tiles * std::min(nsys, small_groups(p.tiles));
}

// Refused (an error returned, nothing launched) where the grid cannot be
// resident, for instance beside a limit on the SMs the process may use.
template <class... Args>
cudaError_t launch_cooperative(const void* kernel, const SmallPlan& p, cudaStream_t st, Args... args) {
  void* v[] = {(void*)&args...};
  return cudaLaunchCooperativeKernel(kernel, dim3(p.tiles, p.groups), dim3(p.nt), v, 0, st);
}

// the kernel of an operator (wide: the 255-register form), and its launch
template <typename G, typename Wt, template <int> class VA>
const void* small_kernel(const SWOp<float, G, Wt, VA>&, bool wide) {
  return wide ? (const void*)sw_small<kSmallWide, GeomBlk, G, Wt, VA<3>>
              : (const void*)sw_small<kSmallThreads, GeomBlk, G, Wt, VA<3>>;
}
template <typename G, typename Wt, template <int> class VA>
cudaError_t launch_small(const SWOp<float, G, Wt, VA>& op, const GeomBlk& g, VA<3> p, VA<3> t, VecP32<3> r, VecP32<3> x,
                         const SmallArgs& a, const SmallPlan& pl, cudaStream_t st) {
  return launch_cooperative(small_kernel(op, pl.wide), pl, st, g, op.U, op.W, p, t, r, x, a);
}
template <bool R1, class Sites, class GA, class VI> const void* wilson_small_kernel(bool wide) {
  return wide ? (const void*)wilson_small<kSmallWide, R1, Sites, GA, VI>
              : (const void*)wilson_small<kSmallThreads, R1, Sites, GA, VI>;
}
template <typename G, template <int> class VA, bool R1, bool LEAN>
const void* small_kernel(const WOp<float, G, VA, R1, LEAN>&, bool wide) {
  return wilson_small_kernel<R1, FullSites<GeomBlk>, G, VA<12>>(wide);
}
template <typename G, template <int> class VA, bool R1, bool LEAN>
cudaError_t launch_small(const WOp<float, G, VA, R1, LEAN>& op, const GeomBlk& g, VA<12> p, VA<12> t, VecP32q<12> r,
                         VecP32q<12> x, const SmallArgs& a, const SmallPlan& pl, cudaStream_t st) {
  return launch_cooperative(small_kernel(op, pl.wide), pl, st, FullSites<GeomBlk>{g}, op.U, p, t, r, x, size_t(0), a);
}

}  // namespace swc
