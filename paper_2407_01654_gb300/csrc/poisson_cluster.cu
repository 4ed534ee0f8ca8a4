// The whole potential loop of one solve (Algorithm 1 step 3) on one thread-block cluster,
// for lattices whose potential populations fit the shared memory of at most 16 SMs.
//
// On a small lattice a sub-iteration of the tiled loop (poisson_resident.cu) is a few
// hundred instructions per thread between a grid barrier through L2, an export of the
// tile's perimeter to L2 and its import by the neighbours: about 3.5 us whatever the size.
// Here every exchange stays in the cluster: post-collision populations are pushed to the
// node they stream to, in the own CTA's shared memory or in a neighbour's (distributed
// shared memory), and a sub-iteration ends in a CTA barrier and, where there are neighbours,
// with the arrival of their rows, counted on an mbarrier.
//
// Decomposition: CTA r of C owns the rows [r rows, (r + 1) rows) of the lattice, so x stays
// inside a CTA and only a CTA's first and last row push to another one.  A thread owns NPT
// nodes, t + s T for s < NPT, as packed pairs (the arithmetic of the other loops, bit for
// bit).  Three copies of the eight incoming populations rotate: phase p
//   reads state p from copy p mod 3 and forms varphi^p and the thread's part of the stopping
//   sums of sub-iteration p;
//   collides and pushes state p + 1 into copy (p + 1) mod 3: into this CTA's shared memory,
//   or by st.async into the neighbour's, which counts the bytes on an mbarrier there;
//   meets its own CTA at a barrier.
// Meanwhile one more warp, which owns no nodes, adds up the CTA's sums of sub-iteration p - 1,
// sends them to every CTA's table (st.async again), waits for theirs and applies the rule; the
// barrier hands its verdict to the others.  (With every warp sending its own sums and deciding
// for itself the rule cost 0.4 to 0.5 us of a sub-iteration, as much as the rest of it.)
// A phase starts once the neighbours' rows are counted in.  There is no cluster-wide barrier:
// its release waits for every outstanding remote store (a memory barrier, 38 % of a phase when
// this loop used barrier.cluster: 1.44 us per sub-iteration at 128 x 128), while a counted
// store needs none.  CTAs drift by at most one phase (a neighbour needs our rows, and the rule
// every CTA's sums), so two row barriers, two table slots and, because all take the same
// decision before they go on, three copies are enough; state p - 1 stays in its copy until the
// rule has judged it.  With two copies (lattices that leave
// no room for three) the rule is applied before the push.  A fixed count needs no rule: only
// its last phase, which finds the final state in its registers, forms sums.
//
// A population that would cross a wall returns to its own node by the anti-bounce-back rule,
// written by the node itself.  Sums are FP32 throughout in a fixed order; every CTA adds the
// same table in the same order and takes the same decision.  The order is not the tiled
// loop's, whose sums can differ from these in the last bits; where that could matter, with
// num within 2e-5 of tol^2 den (both orders are far closer than that to the exact sums: at
// most 25 roundings of 6e-8), the sums are formed again in the tiled loop's own order
// (tiled_sums), so both loops stop at the same sub-iteration.
// The waits are bounded (2 s): one that runs out sets Ctl::bar_error and the kernel returns.
#include <type_traits>

#include "ehd_internal.cuh"

namespace ehd {

namespace {

constexpr int MAX_CLUSTER = 16;

__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
// The address, in the cluster's shared window, of CTA `rank`'s copy of a shared variable.
__device__ __forceinline__ unsigned map_rank(unsigned a, unsigned rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// Stores at a shared address plus a compile-time byte offset: in this CTA, or in any CTA of
// the cluster (slower; only the rows that border another CTA take it).
template <int OFF>
__device__ __forceinline__ void st_own(unsigned a, float v) {
  asm volatile("st.shared.f32 [%0 + %1], %2;" ::"r"(a), "n"(OFF), "f"(v) : "memory");
}
// The same into another CTA's shared memory, its bytes counted on that CTA's mbarrier.
template <int OFF>
__device__ __forceinline__ void st_async(unsigned a, float v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0 + %1], %2, [%3];" ::
                   "r"(a), "n"(OFF), "f"(v), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async2(unsigned a, float x, float y, unsigned bar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(a),
      "f"(x), "f"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
// The one arrival of a phase, which announces the bytes the phase waits for.
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0u;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
constexpr unsigned long long WAIT_LIMIT_NS = 2000000000ull;  // 2 s
// Waits until the barrier's phase of this parity is complete; false when the limit ran out.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_try(bar, parity))
    if (global_ns() - t0 > WAIT_LIMIT_NS) return false;
  return true;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// __syncthreads_or for a place that not every warp of the CTA comes through: the hardware joins a
// barrier's arrivals wherever in the code they come from.
__device__ __forceinline__ bool cta_or(bool v) {
  unsigned r;
  __syncwarp();
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, 0, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((unsigned)v)
      : "memory");
  return r != 0u;
}

// Warp sums of x and y in five shuffles: after the first, the low half of the warp carries x
// and the high half y.  The same tree (lanes 16, 8, 4, 2, 1 apart) as two butterflies, so the
// same bits; the low lanes return x's sum, the high lanes y's.
__device__ __forceinline__ float warp_sum2(float x, float y, int lane) {
  const bool hi = lane >= 16;
  float v = (hi ? y : x) + __shfl_xor_sync(0xffffffffu, hi ? x : y, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Compile-time shape: CAP nodes per CTA at most, NPT per thread.
template <int CAP, int NPT>
struct ClusterShape {
  static_assert(NPT % 2 == 0 && CAP % (32 * NPT) == 0, "whole warps of packed pairs");
  static constexpr int THREADS = CAP / NPT;
  static constexpr int WARPS = THREADS / 32;
  static constexpr int LAUNCH = THREADS + 32;  // and the warp that keeps the sums
  static constexpr int COPIES = CAP <= 2048 ? 3 : 2;
  static constexpr bool KEEP = NPT <= 2 || THREADS <= 384;  // push addresses kept in registers
  static constexpr int COPY = 8 * CAP;  // floats of one copy
  static constexpr size_t SMEM = sizeof(float) * (size_t)COPIES * COPY;
};

template <int V>
using Const = std::integral_constant<int, V>;
template <class F>
__device__ __forceinline__ void each_direction(F f) {
  f(Const<1>{}), f(Const<2>{}), f(Const<3>{}), f(Const<4>{});
  f(Const<5>{}), f(Const<6>{}), f(Const<7>{}), f(Const<8>{});
}

}  // namespace

template <int CAP, int NPT, bool CONV>
__global__ void __launch_bounds__(ClusterShape<CAP, NPT>::LAUNCH, 1)
    k_poisson_cluster(KParams k, int rows, ResidentGeom rg, float* __restrict__ hbuf,
                      const float2* __restrict__ aq, float2* __restrict__ scratch, Ctl* ctl) {
  using S = ClusterShape<CAP, NPT>;
  constexpr int NP = NPT / 2;
  constexpr int T = S::THREADS;
  __shared__ __align__(8) unsigned long long s_rows[2], s_sums[2];  // mbarriers
  __shared__ __align__(8) float2 s_table[2][MAX_CLUSTER];  // every CTA's sums, in turn
  __shared__ float2 s_warp[2][S::WARPS];                   // this CTA's warps' sums, in turn
  __shared__ int s_verdict;
  extern __shared__ __align__(16) float smc[];  // [COPIES][8][CAP]

  const int nx = k.nx, ny = k.ny;
  const size_t N = (size_t)k.N;
  const int C = (int)gridDim.x, rank = (int)blockIdx.x;  // one cluster: its rank is the block
  const int row0 = rank * rows;
  const int th = min(rows, ny - row0);
  const int nloc = th * nx;
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool keeper = warp == S::WARPS;  // the warp that keeps the sums
  const int parity = __ldg(&ctl->parity);
  float* __restrict__ hsrc = hbuf + (size_t)parity * NH * N;
  const int g0 = row0 * nx;  // my first node

  // every load of the thread's nodes is issued before any is used (a node past the CTA's
  // rows loads node 0 and takes no further part)
  float2 h[NP][8], a[NP], qs[NP];
  bool valid[NPT];
#pragma unroll
  for (int s = 0; s < NPT; ++s) {
    valid[s] = !keeper && tid + s * T < nloc;
    const size_t g = EHD_IDX(k, g0 + (valid[s] ? tid + s * T : 0), N);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float v = hsrc[i * N + g];
      if (s & 1)
        h[s >> 1][i].y = v;
      else
        h[s >> 1][i].x = v;
    }
    const float2 c = aq[g];
    if (s & 1) {
      a[s >> 1].y = c.x;
      qs[s >> 1].y = c.y;
    } else {
      a[s >> 1].x = c.x;
      qs[s >> 1].x = c.y;
    }
  }
  const float qshift = k.neutralize ? __ldg(&ctl->mean_q) : 0.0f;
  const float vw_b = __ldg(&ctl->vw_b), vw_t = __ldg(&ctl->vw_t);
  const double tol = ctl->tol;
  // a non-finite phi or q (flagged by the moments pass) stops the loop after one
  // sub-iteration, not converged
  const bool bad_state = __ldg(&ctl->nonfinite) != 0;
  const int min_iter = bad_state ? 1 : ctl->min_iter, max_iter = bad_state ? 1 : ctl->max_iter,
            fixed = bad_state ? 0 : ctl->fixed_iter;
  const float om = k.omega_h;
  const float tol2 = (float)(tol * tol);
  const bool tol_ok = tol2 > 1e-25f && tol2 < 1e25f;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    float2 q = __fadd2_rn(qs[j], f2(-qshift));
    if (CONV) q = __fmul2_rn(q, f2(k.inv_chi));
    qs[j] = __fmul2_rn(f2(0.125f), q);
  }

  // Where a node's populations go.  Nodes whose eight neighbours lie in this CTA's rows, away
  // from the lattice's x edges, push at fixed offsets; the others' row bits say that a push
  // leaves for the neighbouring CTA (FAR_LO, FAR_HI) or returns to the node from a wall
  // (WALL_LO, WALL_HI) to slot opp(i).  A node past the CTA's rows pushes to its own unused
  // cell.  Where the register budget allows it, a node's eight addresses are kept
  // (KEEP); elsewhere an edge node's are formed at each push from its x.
  constexpr unsigned FAR_LO = 1u << 16, FAR_HI = 2u << 16, WALL_LO = 4u << 16, WALL_HI = 8u << 16,
                     BOT = 16u << 16, TOP = 32u << 16, EDGE = 64u << 16;
  const unsigned self = smem_addr(smc);
  const int below = rank == 0 ? C - 1 : rank - 1, above = rank + 1 == C ? 0 : rank + 1;
  unsigned lo_bar = 0u, hi_bar = 0u, row_bytes = 0u;  // the neighbours' row barriers; bytes in
  unsigned lo_row = self + 4u * (unsigned)((th - 1) * nx), hi_row = self;  // rows beyond mine
  if (C > 1) {
    const int th_below = min(rows, ny - below * rows);
    lo_row = map_rank(self, (unsigned)below) + 4u * (unsigned)((th_below - 1) * nx);
    hi_row = map_rank(self, (unsigned)above);
    lo_bar = map_rank(smem_addr(s_rows), (unsigned)below);
    hi_bar = map_rank(smem_addr(s_rows), (unsigned)above);
    row_bytes = 12u * (unsigned)nx * ((k.walls && row0 == 0 ? 0u : 1u) +
                                      (k.walls && row0 + th == ny ? 0u : 1u));
    // diagnostics: an expired barrier waits for bytes that nobody sends
    if (ctl->bar_count == EXPIRED_BARRIER) row_bytes += 4u;
  }
  // shared byte address (copy 0) that direction i of node l, described by w, is pushed to
  auto target = [&](int i, int l, unsigned w) -> unsigned {
    const unsigned own = self + 4u * (unsigned)l;
    if (cy(i) > 0 ? (w & WALL_HI) : (cy(i) < 0 ? (w & WALL_LO) : 0u))
      return own + 4u * (unsigned)((opp(i) - 1) * CAP);
    const int x = (int)(w & 0xffffu);
    const int xx = cx(i) > 0 ? (x + 1 == nx ? 0 : x + 1) : (cx(i) < 0 ? (x == 0 ? nx - 1 : x - 1) : x);
    const unsigned mid = own - 4u * (unsigned)x;
    const unsigned row = cy(i) > 0 ? ((w & TOP) ? hi_row : mid + 4u * (unsigned)nx)
                                   : (cy(i) < 0 ? ((w & BOT) ? lo_row : mid - 4u * (unsigned)nx) : mid);
    return row + 4u * (unsigned)((i - 1) * CAP + xx);
  };
  unsigned info[NPT];  // x and the row bits
  unsigned dst[S::KEEP ? NPT : 1][8];
#pragma unroll
  for (int s = 0; s < NPT; ++s) {
    const int l = tid + s * T;
    info[s] = 0u;
    if (valid[s]) {
      const int y = l / nx, x = l - y * nx;
      unsigned w = (unsigned)x;
      if (y == 0) w |= BOT | (k.walls && row0 == 0 ? WALL_LO : (C > 1 ? FAR_LO : 0u));
      if (y == th - 1) w |= TOP | (k.walls && row0 + th == ny ? WALL_HI : (C > 1 ? FAR_HI : 0u));
      if (y == 0 || y == th - 1 || x == 0 || x == nx - 1) w |= EDGE;
      info[s] = w;
      if constexpr (S::KEEP) {
#pragma unroll
        for (int i = 1; i < 9; ++i) dst[s][i - 1] = target(i, l, w);
      }
    } else if constexpr (S::KEEP) {
#pragma unroll
      for (int i = 1; i < 9; ++i) dst[s][i - 1] = self + 4u * (unsigned)(l + (i - 1) * CAP);
    }
  }
  float *own0 = smc + tid, *up0 = own0 + nx, *dn0 = own0 - nx;
  // where the CTA's sums go: lane c writes CTA c's table
  const unsigned to = (unsigned)(lane < C ? lane : 0);
  const unsigned my_table = map_rank(smem_addr(s_table), to) + 8u * (unsigned)rank;
  const unsigned sums_bar = map_rank(smem_addr(s_sums), to);
  const unsigned my_rows = smem_addr(s_rows), my_sums = smem_addr(s_sums);
  if (tid < 2 * MAX_CLUSTER) s_table[0][tid] = make_float2(0.0f, 0.0f);  // past C: zero
  // no remote store before every CTA of the cluster has started and set up its barriers
  if (C > 1) {
    if (tid == 0) {
      for (int j = 0; j < 2; ++j) {
        mbar_init(my_rows + 8u * j);
        mbar_init(my_sums + 8u * j);
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }

  float2 vold[NP];          // varphi of the state in the registers
  float2 v1[NP], v2[NP];    // and of the two states before it
  float rel = 0.0f;
  int conv = 0, it = 0;
  bool fail = false;  // a wait of this thread ran out

  // The parity of the sums' barrier at phase p: under the rule slots take turns from phase 1
  // on; a fixed count uses one of them, once.
  auto sums_parity = [&](int p) { return fixed > 0 ? 0u : (unsigned)((p - 1) >> 1) & 1u; };
  auto meet = [&]() {  // every thread of the cluster, global memory included
    if (C > 1) {
      __syncwarp();
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  };
  // The potential of the state after sub-iteration st, and its change from potential v as the
  // one-step tiled loop forms it: from the rounded new potential in odd sub-iterations (its own
  // layout), with one rounding in even ones.
  auto change = [&](int st, const float2 (&hn)[8], float2 v, float2& vnew) -> float2 {
    const float2 hsum = h_sum8x2(hn);
    // (scalar products: a packed one may be contracted with the addition)
    vnew = make_float2(h_varphi(hsum.x), h_varphi(hsum.y));
    return (st & 1) ? __fadd2_rn(vnew, neg2(v)) : __ffma2_rn(hsum, f2(9.0f / 5.0f), neg2(v));
  };
  // The stopping sums of sub-iteration st, whose state is in h and which began from potential
  // v, in the order of the one-step tiled loop: per thread of a 64 x TY tile the nodes of one
  // column TY / 4 rows apart, then lanes, warps and tiles.  Every node leaves its change and
  // its old potential in scratch; the cluster's warps share out the tiles' warps.
  // A CTA that had given up took part in the first meeting on its way out and is gone: nothing
  // may be sent to it any more.
  auto tiled_sums = [&](int st, float& sa, float& sb, const float2 (&v)[NP]) {
    float2 d[NP], vn;
#pragma unroll
    for (int j = 0; j < NP; ++j) d[j] = change(st, h[j], v[j], vn);
#pragma unroll
    for (int s = 0; s < NPT; ++s) {
      if (valid[s])
        scratch[g0 + tid + s * T] = (s & 1) ? make_float2(d[s >> 1].y, v[s >> 1].y)
                                            : make_float2(d[s >> 1].x, v[s >> 1].x);
    }
    meet();
    const int nw = rg.TY / 2, step = rg.TY / 4, tiles = rg.ntx * rg.nty;
    float2* wsum = scratch + N;
    for (int u = keeper ? tiles * nw : rank * S::WARPS + warp; u < tiles * nw; u += C * S::WARPS) {
      const int t = u / nw, w = u - t * nw;
      const int x = (t % rg.ntx) * 64 + (w & 1) * 32 + lane, y0 = (t / rg.ntx) * rg.TY;
      float num = 0.0f, den = 0.0f;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int y = y0 + (w >> 1) + s * step;
        if (x < nx && y < ny) {
          const float2 e = __ldcg(scratch + (size_t)y * nx + x);
          num = __fmaf_rn(e.x, e.x, num);
          den = __fmaf_rn(e.y, e.y, den);
        }
      }
      const float part = warp_sum2(num, den, lane);
      const float other = __shfl_xor_sync(0xffffffffu, part, 16);
      if (lane == 0) __stcg(wsum + u, make_float2(part, other));
    }
    meet();
    float a = 0.0f, b = 0.0f;
    for (int t = 0; t < tiles; ++t) {
      const float2 e = lane < nw ? __ldcg(wsum + t * nw + lane) : make_float2(0.0f, 0.0f);
      const float part = warp_sum2(e.x, e.y, lane);
      const float other = __shfl_xor_sync(0xffffffffu, part, 16);
      if (lane == (t & 31)) {
        a += lane < 16 ? part : other;
        b += lane < 16 ? other : part;
      }
    }
    const float part = warp_sum2(a, b, lane);
    const float other = __shfl_xor_sync(0xffffffffu, part, 16);
    sa = lane < 16 ? part : other;
    sb = lane < 16 ? other : part;
    meet();  // scratch may be written again
    if (C > 1 && __ldcg(&ctl->redo) != 0) fail = true;
  };
  // The keeper adds up the CTA's sums of sub-iteration st (after the CTA barrier that followed
  // them) and sends them to every CTA.
  auto send_sums = [&](int st) {
    if (C == 1) return;
    const float2 v = lane < S::WARPS ? s_warp[st & 1][lane] : make_float2(0.0f, 0.0f);
    const float part = warp_sum2(v.x, v.y, lane);
    const float other = __shfl_xor_sync(0xffffffffu, part, 16);
    if (lane == 0) mbar_expect(my_sums + 8u * (unsigned)(st & 1), 8u * (unsigned)C);
    if (lane < C && !fail)
      st_async2(my_table + 8u * MAX_CLUSTER * (unsigned)(st & 1), lane < 16 ? part : other,
                lane < 16 ? other : part, sums_bar + 8u * (unsigned)(st & 1));
  };
  // The sums of sub-iteration st over the lattice, from the CTAs' (with one CTA, its warps').
  auto all_sums = [&](int st, float& sa, float& sb) {
    const float2* e = C > 1 ? s_table[st & 1] : s_warp[st & 1];
    const int n = C > 1 ? C : S::WARPS;
    if (C > 1 && !mbar_wait(my_sums + 8u * (unsigned)(st & 1), sums_parity(st))) fail = true;
    float part = 0.0f;  // the low lanes add num, the high lanes den
    for (int j = lane & 15; j < n; j += 16) part += reinterpret_cast<const float*>(e + j)[lane >> 4];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const float other = __shfl_xor_sync(0xffffffffu, part, 16);
    sa = lane < 16 ? part : other;
    sb = lane < 16 ? other : part;
  };
  auto ratio = [&](float n, float d) {
    return n == 0.0f && d == 0.0f ? 0.0f : (d == 0.0f ? __int_as_float(0x7f800000) : sqrtf(n / d));
  };
  // The stopping rule for sub-iteration st from its sums: GO_ON, STOP (it, rel and conv set) or
  // UNSURE, which wants the sums in the tiled loop's order (sure = true takes them as such).
  enum { GO_ON = 0, STOP = 1, UNSURE = 2 };
  auto decide = [&](int st, float sa, float sb, bool sure) -> int {
    if (fixed > 0) {
      conv = 1;
    } else {
      const bool plain = !sure && tol_ok && sb > 1e-25f && sb < 1e25f;
      if (plain && sa > 1.00002f * tol2 * sb) {
        conv = 0;
      } else if (plain && sa < 0.99998f * tol2 * sb) {
        conv = st >= min_iter;
      } else if (st < min_iter && st < max_iter) {
        conv = 0;  // whatever the sums say
      } else if (!sure && sb != 0.0f) {  // all zero is zero in any order
        return UNSURE;
      } else {
        conv = (st >= min_iter) && ((double)ratio(sa, sb) < tol);
      }
      if (!conv && st < max_iter) return GO_ON;
    }
    rel = ratio(sa, sb);
    it = st;
    return STOP;
  };
  auto load_state = [&](auto copy) {
    constexpr int at = decltype(copy)::value * S::COPY;
    if (keeper) return;  // owns no nodes: its cells would lie past the copies
#pragma unroll
    for (int j = 0; j < NP; ++j)
#pragma unroll
      for (int i = 0; i < 8; ++i)
        h[j][i] = make_float2(smc[at + i * CAP + tid + (2 * j) * T],
                              smc[at + i * CAP + tid + (2 * j + 1) * T]);
  };
  // The push of phase p, into the given copy.
  auto collide_push = [&](int p, auto copy) {
    constexpr int at = decltype(copy)::value * S::COPY * 4;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      float2 hs[8];
      if constexpr (CONV) {
        h_star_conv8x2(h[j], a[j], vold[j], qs[j], hs);
      } else {
        float2 m1x, m1y;
        h_moment1x2(h[j], m1x, m1y);
        h_star8x2(h[j], om, vold[j], a[j], m1x, m1y, qs[j], hs);
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int s = 2 * j + c;
        // the address and the store of one direction; FAR rows carry their barrier
        auto put = [&](auto dir, unsigned a, unsigned w) {
          constexpr int i = decltype(dir)::value;
          const unsigned bar = 8u * (unsigned)(p & 1);
          float x = c ? hs[i - 1].y : hs[i - 1].x;
          if constexpr (cy(i) > 0) {
            if (w & WALL_HI) x = h_wall(i, x, vw_t);
            if (w & FAR_HI) {
              st_async<at>(a, x, hi_bar + bar);
              return;
            }
          } else if constexpr (cy(i) < 0) {
            if (w & WALL_LO) x = h_wall(i, x, vw_b);
            if (w & FAR_LO) {
              st_async<at>(a, x, lo_bar + bar);
              return;
            }
          }
          st_own<at>(a, x);
        };
        unsigned w = info[s];
        if constexpr (S::KEEP) {
          if (w & (WALL_LO | WALL_HI | FAR_LO | FAR_HI)) {
            each_direction([&](auto dir) { put(dir, dst[s][decltype(dir)::value - 1], w); });
          } else {
            each_direction([&](auto dir) { put(dir, dst[s][decltype(dir)::value - 1], 0u); });
          }
        } else {
          if (w & EDGE) {
            // opaque to the compiler, which would otherwise form every edge address before the
            // loop and spill them
            asm volatile("" : "+r"(w));
            const unsigned own = self + 4u * (unsigned)(tid + s * T), x = w & 0xffffu;
            const unsigned e = x + 1u == (unsigned)nx ? 4u - 4u * (unsigned)nx : 4u;
            const unsigned wst = x == 0u ? 4u * (unsigned)nx - 4u : 0u - 4u;
            auto row = [&](auto d0, auto de, auto dw, unsigned base, unsigned flags) {
              put(d0, base + 4u * (unsigned)((decltype(d0)::value - 1) * CAP), flags);
              put(de, base + e + 4u * (unsigned)((decltype(de)::value - 1) * CAP), flags);
              put(dw, base + wst + 4u * (unsigned)((decltype(dw)::value - 1) * CAP), flags);
            };
            auto back = [&](auto dir) {
              constexpr int i = decltype(dir)::value;
              put(dir, own + 4u * (unsigned)((opp(i) - 1) * CAP), w);
            };
            put(Const<1>{}, own + e, 0u);
            put(Const<3>{}, own + wst + 8u * CAP, 0u);
            if (w & WALL_HI)
              back(Const<2>{}), back(Const<5>{}), back(Const<6>{});
            else if (w & FAR_HI)
              row(Const<2>{}, Const<5>{}, Const<6>{}, hi_row + 4u * x, FAR_HI);
            else
              row(Const<2>{}, Const<5>{}, Const<6>{},
                  (w & TOP) ? hi_row + 4u * x : own + 4u * (unsigned)nx, 0u);
            if (w & WALL_LO)
              back(Const<4>{}), back(Const<8>{}), back(Const<7>{});
            else if (w & FAR_LO)
              row(Const<4>{}, Const<8>{}, Const<7>{}, lo_row + 4u * x, FAR_LO);
            else
              row(Const<4>{}, Const<8>{}, Const<7>{},
                  (w & BOT) ? lo_row + 4u * x : own - 4u * (unsigned)nx, 0u);
          } else if (valid[s]) {
#pragma unroll
            for (int i = 1; i < 9; ++i) {
              float* base = cy(i) > 0 ? up0 : (cy(i) < 0 ? dn0 : own0);
              base[decltype(copy)::value * S::COPY + (i - 1) * CAP + cx(i) + s * T] =
                  c ? hs[i - 1].y : hs[i - 1].x;
            }
          }
        }
      }
    }
  };
  // Phase p (p >= 1), reading state p from copy RD and pushing state p + 1 into copy WR; OLD
  // holds state p - 1.  0: go on; 1: the loop is over, with the final state in h; 2: a wait
  // ran out.
  auto phase = [&](int p, auto RD, auto WR, auto OLD) -> int {
    const bool last = fixed > 0 && p == fixed;
    const bool rule = fixed == 0 && p > 1;
    int verdict = GO_ON;
    bool pushed = !last;
    float sa, sb;
    if (keeper) {
      // what this phase's neighbours will send
      if (C > 1 && lane == 0 && !last) mbar_expect(my_rows + 8u * (unsigned)(p & 1), row_bytes);
      if (rule) send_sums(p - 1);
    } else {
      // the neighbours' rows of state p, pushed in their phase p - 1
      if (C > 1 && !mbar_wait(my_rows + 8u * (unsigned)((p - 1) & 1), (unsigned)((p - 1) >> 1) & 1u))
        fail = true;
      load_state(RD);
    }
    if (S::COPIES == 2 && rule) {
      // no copy to spare: every warp decides before the push
      all_sums(p - 1, sa, sb);
      verdict = decide(p - 1, sa, sb, false);
      if (verdict == UNSURE) {
        // a wait that ran out may have left another warp with another verdict: it is at the
        // barriers at the end of the phase, and these are the same two
        if (cta_or(fail)) {
          cta_or(fail);
          return 2;
        }
        load_state(OLD);
        tiled_sums(p - 1, sa, sb, v1);
        verdict = decide(p - 1, sa, sb, true);
        load_state(RD);
      }
      pushed = verdict == GO_ON;
    }
    if (!keeper) {
      float num = 0.0f, den = 0.0f;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        float2 vnew;
        const float2 d = change(p, h[j], vold[j], vnew);
        if (S::COPIES == 3) v2[j] = v1[j];
        v1[j] = vold[j];
        if (valid[2 * j]) {
          num = __fmaf_rn(d.x, d.x, num);
          den = __fmaf_rn(vold[j].x, vold[j].x, den);
        }
        if (valid[2 * j + 1]) {
          num = __fmaf_rn(d.y, d.y, num);
          den = __fmaf_rn(vold[j].y, vold[j].y, den);
        }
        vold[j] = vnew;
      }
      if (pushed && !fail) collide_push(p, WR);
      if (fixed == 0 || last) {
        const float part = warp_sum2(num, den, lane);
        const float other = __shfl_xor_sync(0xffffffffu, part, 16);
        if (lane == 0) s_warp[p & 1][warp] = make_float2(part, other);
      }
    } else if (S::COPIES == 3 && rule) {
      all_sums(p - 1, sa, sb);
      verdict = decide(p - 1, sa, sb, false);
      if (verdict != GO_ON && lane == 0) s_verdict = verdict;
    }
    if (__syncthreads_or(fail || verdict != GO_ON)) {
      if (__syncthreads_or(fail)) return 2;
      if (S::COPIES == 3) {
        verdict = s_verdict;
        if (verdict == UNSURE) {
          load_state(OLD);
          tiled_sums(p - 1, sa, sb, v2);
          verdict = decide(p - 1, sa, sb, true);
          if (verdict == GO_ON) return 0;
        }
      }
      if (!keeper) {
        load_state(OLD);
        // what the neighbours sent before they took the same decision must have arrived before
        // this CTA leaves
        if (C > 1 && pushed && !mbar_wait(my_rows + 8u * (unsigned)(p & 1), (unsigned)(p >> 1) & 1u))
          fail = true;
      }
      return __syncthreads_or(fail) ? 2 : 1;
    }
    if (last) {  // the fixed count's state is in the registers
      if (keeper) {
        send_sums(p);
        all_sums(p, sa, sb);
        decide(p, sa, sb, false);
      }
      return __syncthreads_or(fail) ? 2 : 1;
    }
    return 0;
  };

  // phase 0: the state is in the registers
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    v1[j] = v2[j] = vold[j] = h_varphi2(h_sum8x2(h[j]));
  }
  if (C > 1 && keeper && lane == 0) mbar_expect(my_rows, row_bytes);
  if (!keeper) collide_push(0, Const<1>{});
  __syncthreads();
  int end = 0;
  if constexpr (S::COPIES == 3) {
    for (int p = 1;; p += 3) {
      if ((end = phase(p, Const<1>{}, Const<2>{}, Const<0>{}))) break;
      if ((end = phase(p + 1, Const<2>{}, Const<0>{}, Const<1>{}))) break;
      if ((end = phase(p + 2, Const<0>{}, Const<1>{}, Const<2>{}))) break;
    }
  } else {
    for (int p = 1;; p += 2) {
      if ((end = phase(p, Const<1>{}, Const<0>{}, Const<0>{}))) break;
      if ((end = phase(p + 1, Const<0>{}, Const<1>{}, Const<1>{}))) break;
    }
  }
  if (end == 2) {
    if (tid == 0) {
      atomicOr(&ctl->bar_error, 1);
      atomicOr(&ctl->redo, 1);  // tells a CTA that meets this one in tiled_sums
    }
    // every CTA's waits run out, or it meets this one: none leaves before the others have
    // stopped pushing to it
    if (C > 1) {
      cluster_arrive();
      cluster_wait();
    }
    return;
  }

  // the registers hold the final state: write it back in place
#pragma unroll
  for (int s = 0; s < NPT; ++s) {
    if (!valid[s]) continue;
    const size_t g = EHD_IDX(k, g0 + tid + s * T, N);
#pragma unroll
    for (int i = 0; i < 8; ++i) hsrc[i * N + g] = (s & 1) ? h[s >> 1][i].y : h[s >> 1][i].x;
  }
  if (rank == 0 && keeper && lane == 0) {
    ctl->iter = it;
    ctl->rel = (double)rel;
    ctl->converged = conv;
    ctl->done = 1;
  }
}

namespace {

struct ClusterKernel {
  int cap, threads;
  size_t smem;
  const void* f[2];  // the paper's scheme, the conventional one
};
template <int CAP, int NPT>
ClusterKernel cluster_kernel_of() {
  using S = ClusterShape<CAP, NPT>;
  return {CAP, S::LAUNCH, S::SMEM,
          {(const void*)k_poisson_cluster<CAP, NPT, false>,
           (const void*)k_poisson_cluster<CAP, NPT, true>}};
}
const ClusterKernel* cluster_kernels(int* n) {
  static const ClusterKernel all[] = {
      cluster_kernel_of<256, 2>(),  cluster_kernel_of<512, 2>(),  cluster_kernel_of<768, 2>(),
      cluster_kernel_of<1024, 2>(), cluster_kernel_of<1408, 4>(), cluster_kernel_of<1920, 4>(),
      cluster_kernel_of<2432, 4>(), cluster_kernel_of<2880, 6>()};
  *n = (int)(sizeof(all) / sizeof(all[0]));
  return all;
}
const ClusterKernel* cluster_kernel(int cap) {
  int n;
  const ClusterKernel* all = cluster_kernels(&n);
  for (int j = 0; j < n; ++j)
    if (all[j].cap == cap) return &all[j];
  return nullptr;
}

}  // namespace

// Nodes from which a lattice is spread over more than one CTA, and nodes a CTA should at
// least get then.
#ifndef EHD_CLUSTER_ONE
#define EHD_CLUSTER_ONE 512
#endif
#ifndef EHD_CLUSTER_MIN
#define EHD_CLUSTER_MIN 256
#endif

bool cluster_geometry(const KParams& kp, ClusterGeom* g, int max_cluster) {
  *g = ClusterGeom{};
  if (kp.slab) return false;
  const long long N = (long long)kp.nx * kp.ny;
  if (max_cluster > MAX_CLUSTER) max_cluster = MAX_CLUSTER;
  int want = 1;
  if (N > EHD_CLUSTER_ONE) {
    want = (int)((N + EHD_CLUSTER_MIN - 1) / EHD_CLUSTER_MIN < max_cluster
                     ? (N + EHD_CLUSTER_MIN - 1) / EHD_CLUSTER_MIN
                     : max_cluster);
  }
  if (want > kp.ny) want = kp.ny;
  const int rows = (kp.ny + want - 1) / want;
  const long long nodes = (long long)rows * kp.nx;
  int n;
  const ClusterKernel* all = cluster_kernels(&n);
  for (int j = 0; j < n; ++j)
    if (nodes <= all[j].cap) {
      g->size = (kp.ny + rows - 1) / rows;
      g->rows = rows;
      g->cap = all[j].cap;
      return true;
    }
  return false;
}

static void cluster_config(const ClusterKernel& ck, const ClusterGeom& g, cudaStream_t st,
                           cudaLaunchAttribute* attr, cudaLaunchConfig_t* cfg) {
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)g.size;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3((unsigned)g.size);
  cfg->blockDim = dim3((unsigned)ck.threads);
  cfg->dynamicSmemBytes = ck.smem;
  cfg->stream = st;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
}

bool cluster_usable(const KParams& kp, const ClusterGeom& g) {
  const ClusterKernel* ck = g.size > 0 ? cluster_kernel(g.cap) : nullptr;
  if (!ck) return false;
  const void* f = ck->f[kp.scheme == 1];
  int clusters = 0;
  cudaLaunchAttribute attr;
  cudaLaunchConfig_t cfg;
  cluster_config(*ck, g, nullptr, &attr, &cfg);
  const bool ok =
      cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ck->smem) ==
          cudaSuccess &&
      (g.size <= 8 ||
       cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) &&
      cudaOccupancyMaxActiveClusters(&clusters, f, &cfg) == cudaSuccess && clusters >= 1;
  cudaGetLastError();
  return ok;
}

// One pair per node and per warp of the tiled loop, in the upper half of the partial sums (the
// moments pass's partials, which the coupled pass still reads, are at most N / 256 at the
// start of the lower half).
static float2* cluster_scratch(const Buffers& b) {
  static_assert(MAX_CLUSTER * 2880 + 256 * 32 <= MAX_PARTIALS, "nodes and warps of all tiles");
  return reinterpret_cast<float2*>(b.partials + MAX_PARTIALS / 2);
}

cudaError_t launch_poisson_cluster(const KParams& kp, const ResidentGeom& rg, const Buffers& b,
                                   cudaStream_t st) {
  const ClusterGeom& g = rg.cluster;
  const ClusterKernel* ck = cluster_kernel(g.cap);
  if (!ck) return cudaErrorInvalidValue;
  KParams k = kp;
  int rows = g.rows;
  ResidentGeom tiles = rg;
  float* h = b.h;
  const float2* aq = b.aq;
  float2* scratch = cluster_scratch(b);
  Ctl* ctl = b.ctl;
  void* args[] = {&k, &rows, &tiles, &h, &aq, &scratch, &ctl};
  cudaLaunchAttribute attr;
  cudaLaunchConfig_t cfg;
  cluster_config(*ck, g, st, &attr, &cfg);
  return cudaLaunchKernelExC(&cfg, ck->f[kp.scheme == 1], args);
}

cudaError_t add_poisson_cluster_node(cudaGraph_t graph, const cudaGraphNode_t* deps, size_t nd,
                                     cudaGraphNode_t* out, const KParams& kp,
                                     const ResidentGeom& rg, const Buffers& b) {
  const ClusterGeom& g = rg.cluster;
  const ClusterKernel* ck = cluster_kernel(g.cap);
  if (!ck) return cudaErrorInvalidValue;
  KParams k = kp;
  int rows = g.rows;
  ResidentGeom tiles = rg;
  float* h = b.h;
  const float2* aq = b.aq;
  float2* scratch = cluster_scratch(b);
  Ctl* ctl = b.ctl;
  void* args[] = {&k, &rows, &tiles, &h, &aq, &scratch, &ctl};
  cudaKernelNodeParams p = {};
  p.func = const_cast<void*>(ck->f[kp.scheme == 1]);
  p.gridDim = dim3((unsigned)g.size);
  p.blockDim = dim3((unsigned)ck->threads);
  p.sharedMemBytes = (unsigned)ck->smem;
  p.kernelParams = args;
  cudaError_t e = cudaGraphAddKernelNode(out, graph, deps, nd, &p);
  if (e != cudaSuccess) return e;
  cudaKernelNodeAttrValue v = {};
  v.clusterDim.x = (unsigned)g.size;
  v.clusterDim.y = 1;
  v.clusterDim.z = 1;
  return cudaGraphKernelNodeSetAttribute(*out, cudaLaunchAttributeClusterDimension, &v);
}

}  // namespace ehd
