// Several sub-iterations of the potential LBE (Eq. weq53) per launch, for lattices beyond the
// chip's storage, whose loop streams through device memory.
//
// One sub-iteration per launch (poisson.cu) reads and writes every population once per
// sub-iteration and spends most of a launch waiting for its loads: 61 us at 1024 x 2048, a third
// of the copy rate.  Here a CTA loads a 64 x 32 tile and a ring n nodes wide, advances the tile
// n <= MULTI_D sub-iterations in shared memory and writes it once; the ring is advanced along,
// one layer less at each sub-iteration.  The populations live in place: sub-iterations alternate
// between reading direction i from the node's own cell and leaving the post-collision
// population in slot opp(i) of it, and reading direction i from slot opp(i) of the cell behind
// (x - c_i) and leaving it in slot i of the cell ahead (x + c_i).  Either way a node writes
// exactly the eight places it read, so one copy (32 bytes a node) and one CTA barrier per
// sub-iteration are enough.  At a wall the population from beyond is the anti-bounce-back of
// the node's own opposite one, kept in the node's own cell.
//
// Per node the arithmetic is the other loops', bit for bit.  The stopping sums are formed as the
// one-step kernel forms them (each thread owns the column and the alternate rows of a 64 x 16
// block that a thread of it owns; FP32 in a warp, FP64 beyond), so a decision differs only
// where FP64 sums in another order do.  The last CTA applies the rule to the n sub-iterations in
// order.  When it stops the loop before the n-th, the state in the other copy of h, from which
// this launch began, is advanced again by that many: one more launch per solve at most.  So that
// settled solves need none, a launch aims at the count that the solves before took (multi_aim):
// with launches of five whatever the count a step took 371, 390, 408, 425 and 325 us at K = 1 ... 5
// and 1024 x 2048, with these it takes 242, 265, 288, 300 and 325, with one sub-iteration a
// launch 237, 296, 355, 414 and 473.
//
// A fixed count needs no decision, so the order of its sums (a statistic) is free and with it
// the tile height: two CTAs fit an SM, and tiles as tall as the lattice's whole waves of
// 2 x 152 need (multi_rows) leave no nearly empty last wave: five sub-iterations at 977 x 811
// take 58.9 us with 592 tiles of 22 rows against 66.1 with 416 of 32, at 1024 x 2048 118.6 with
// 1184 of 28 rows against 120.9 with 1024 of 32.
#include "ehd_internal.cuh"

namespace ehd {

namespace {

constexpr int MTX = 64, MTY = 32, MT = 256;
constexpr int MNODE = MTX * MTY / MT;  // tile nodes per thread: 8, as the one-step kernel's

template <int D>
struct Multi {
  static constexpr int RX = MTX + 2 * D, RY = MTY + 2 * D;
  static constexpr int PLANE = RX * RY;
  static constexpr int RING = (PLANE - MTX * MTY + MT - 1) / MT;  // ring nodes per thread
  static constexpr int PAIRS = (RING + 1) / 2;
  static constexpr size_t SMEM = sizeof(float) * 8 * (size_t)PLANE;
};

constexpr unsigned W_BOT = 1u << 16, W_TOP = 2u << 16, W_NONE = 4u << 16;  // above a frame index

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(__cvta_generic_to_global(src))
               : "memory");
}

// Sub-iterations the next launch may make: what is left of a fixed count in equal launches, or
// under the rule as many as it may.
__host__ __device__ inline int multi_steps(int d, int fixed, int max_iter, int iter) {
  const int left = (fixed > 0 ? fixed : max_iter) - iter;
  if (left <= d) return left;
  if (fixed <= 0) return d;
  const int launches = (left + d - 1) / d;
  return (left + launches - 1) / launches;
}
// Under the rule, after `iter` sub-iterations: equal launches up to the count that the solves before
// took (`guess`, 0: not known), so that the launch that ends the solve mostly ends where the
// rule does; past it one, two, four and then all that a launch may make.
__device__ inline int multi_aim(int d, int guess, int iter) {
  if (guess <= 0) return d;
  const int past = iter - guess;
  const int aim = past < 0 ? -past : (past + 1 < d ? past + 1 : d);
  if (aim <= d) return aim;
  const int launches = (aim + d - 1) / d;
  return (aim + launches - 1) / launches;
}

// Keeps the aim of the next launch after k sub-iterations of a solve under the rule.
// A launch too many repeats a whole one, a launch too short costs one more of a single
// sub-iteration, a third of that: the guess falls at once, and rises when eight solves in a row
// went past it (counts of 4 and 5 in turn at 900 x 900: 184 us a step with the last count as the
// guess, 177 with launches of five, 177 so).
// (Out of line: in line it moved the loops above it, 63.7 us a solve at 977 x 811 against 62.8.)
__device__ __noinline__ void keep_aim(Ctl* ctl, int d, int k, int done) {
  int guess = ctl->guess;
  if (done) {
    const int above = guess > 0 && k > guess ? ctl->above + 1 : 0;
    if (k < guess || guess <= 0 || above >= 8) ctl->guess = guess = k;
    ctl->above = above >= 8 ? 0 : above;
  }
  ctl->aim = multi_aim(d, guess, done ? 0 : k);
}

}  // namespace

template <int D, bool CONV>
__global__ void __launch_bounds__(MT, 2)
    k_poisson_multi(KParams k, int th, float* __restrict__ hbuf, const float2* __restrict__ aq,
                    double2* __restrict__ partials, Ctl* ctl, cudaGraphConditionalHandle cond,
                    int use_cond) {
  using M = Multi<D>;
  constexpr int RX = M::RX, PLANE = M::PLANE;
  extern __shared__ float sm[];  // [8][RY][RX]
  __shared__ float2 s_w[D][MT / 32];
  __shared__ int s_last;

  // control words, written only by a launch's last CTA after every CTA has read them
  if (__ldg(&ctl->done)) return;
  const int parity = __ldg(&ctl->parity);
  const float qshift = k.neutralize ? __ldg(&ctl->mean_q) : 0.0f;
  const float vw_b = __ldg(&ctl->vw_b), vw_t = __ldg(&ctl->vw_t);
  // a non-finite phi or q (flagged by the moments pass) stops the loop after one
  // sub-iteration, not converged
  const bool bad_state = __ldg(&ctl->nonfinite) != 0;
  const int fixed = bad_state ? 0 : __ldg(&ctl->fixed_iter),
            max_iter = bad_state ? 1 : __ldg(&ctl->max_iter);
  const int iter = __ldg(&ctl->iter), redo = __ldg(&ctl->redo), aim = __ldg(&ctl->aim);
  int n = redo > 0 ? redo : multi_steps(D, fixed, max_iter, iter);
  if (fixed <= 0 && redo == 0 && aim > 0 && aim < n) n = aim;
  const int nx = k.nx, ny = k.ny;
  const size_t N = (size_t)k.N;
  const float* __restrict__ src = hbuf + (size_t)parity * NH * N;
  float* __restrict__ dst = hbuf + (size_t)(parity ^ 1) * NH * N;
  const int x0 = blockIdx.x * MTX, y0 = blockIdx.y * th;  // a 64 x th tile, th <= MTY
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float om = k.omega_h;

  // Loads node (x, y) of the frame (tile coordinates) and describes it: its frame index and
  // wall bits.  Beyond an edge in x, or in y without walls, the lattice wraps; beyond a wall
  // there is no node.
  auto fetch = [&](int x, int y, float& a, float& qs) -> unsigned {
    int gy = y0 + y;
    if (gy < 0 || gy >= ny) {
      if (k.walls) {
        a = qs = 0.0f;
        return W_NONE;
      }
      gy = wrap(gy, ny);
    }
    int gx = x0 + x;
    if (gx < 0 || gx >= nx) gx = wrap(gx, nx);
    const unsigned f = (unsigned)((y + D) * RX + x + D);
    const size_t g = EHD_IDX(k, (size_t)gy * nx + gx, N);
#pragma unroll
    for (int i = 0; i < 8; ++i) cp_async4(sm + i * PLANE + f, src + i * N + g);
    const float2 c = __ldg(aq + g);
    a = c.x;
    float q = __fsub_rn(c.y, qshift);
    if (CONV) q = __fmul_rn(q, k.inv_chi);
    qs = __fmul_rn(0.125f, q);
    return f | (k.walls && gy == 0 ? W_BOT : 0u) | (k.walls && gy == ny - 1 ? W_TOP : 0u);
  };

  // my tile nodes, in column lx: of a full tile the rows ly + 2 j of a 16-row block (the
  // one-step kernel's sums); of a lower one pairs of rows, dealt in turn to the four rows of
  // threads, so that all have alike much to do
  const bool full = th == MTY;
  const int lx = tid & 63, ly = (tid >> 7) * 16 + ((tid >> 6) & 1);
  auto row_of = [&](int j) {
    return full ? ly + 2 * j : 2 * ((tid >> 6) + 4 * (j >> 1)) + (j & 1);
  };
  unsigned tf[MNODE];
  float2 ta[MNODE / 2], tq[MNODE / 2];
#pragma unroll
  for (int j = 0; j < MNODE; ++j) {
    float a = 0.0f, q = 0.0f;
    tf[j] = row_of(j) < th ? fetch(lx, row_of(j), a, q) : W_NONE;
    if (j & 1) {
      ta[j >> 1].y = a;
      tq[j >> 1].y = q;
    } else {
      ta[j >> 1].x = a;
      tq[j >> 1].x = q;
    }
  }
  // my nodes of the ring, n wide: n rows below, n above (each 64 + 2 n long), then n columns on
  // either side; the layer (1 next to the tile) above the wall bits
  unsigned rf[2 * M::PAIRS];
  float2 ra[M::PAIRS], rq[M::PAIRS];
  {
    const int wide = MTX + 2 * n, rows = 2 * n * wide, ring = rows + 2 * n * th;
#pragma unroll
    for (int m = 0; m < 2 * M::PAIRS; ++m) {
      const int r = tid + m * MT;
      float a = 0.0f, q = 0.0f;
      unsigned w = W_NONE;
      if (r < ring) {
        int x, y;
        if (r < rows) {
          const int row = r / wide;
          x = r - row * wide - n;
          y = row < n ? row - n : th + row - n;
        } else {
          const int c = (r - rows) / th;
          y = (r - rows) - c * th;
          x = c < n ? c - n : MTX + c - n;
        }
        const int dx = x < 0 ? -x : (x >= MTX ? x - MTX + 1 : 0);
        const int dy = y < 0 ? -y : (y >= th ? y - th + 1 : 0);
        w = fetch(x, y, a, q) | ((unsigned)(dx > dy ? dx : dy) << 20);
      }
      rf[m] = w;
      if (m & 1) {
        ra[m >> 1].y = a;
        rq[m >> 1].y = q;
      } else {
        ra[m >> 1].x = a;
        rq[m >> 1].x = q;
      }
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  // The state of the node at w: direction i from its own cell (sw false) or from slot opp(i) of
  // the cell behind it, at a wall from its own.
  auto read1 = [&](unsigned w, int i, bool sw) -> float {
    const int f = (int)(w & 0xffffu);
    if (!sw) return sm[(i - 1) * PLANE + f];
    if (cy(i) > 0 && (w & W_BOT)) return h_wall(i, sm[(i - 1) * PLANE + f], vw_b);
    if (cy(i) < 0 && (w & W_TOP)) return h_wall(i, sm[(i - 1) * PLANE + f], vw_t);
    return sm[(opp(i) - 1) * PLANE + f - cy(i) * RX - cx(i)];
  };
  // The post-collision population i of the node at w, to where this node read direction opp(i).
  auto write1 = [&](unsigned w, int i, bool sw, float v) {
    const int f = (int)(w & 0xffffu);
    if (!sw)
      sm[(opp(i) - 1) * PLANE + f] = v;
    else if (cy(i) < 0 && (w & W_BOT))
      sm[(opp(i) - 1) * PLANE + f] = h_wall(opp(i), v, vw_b);
    else if (cy(i) > 0 && (w & W_TOP))
      sm[(opp(i) - 1) * PLANE + f] = h_wall(opp(i), v, vw_t);
    else
      sm[(i - 1) * PLANE + f + cy(i) * RX + cx(i)] = v;
  };
  auto read_pair = [&](unsigned w0, unsigned w1, bool sw, float2 (&h)[8]) {
#pragma unroll
    for (int i = 1; i < 9; ++i) h[i - 1] = make_float2(read1(w0, i, sw), read1(w1, i, sw));
  };
  auto collide_pair = [&](unsigned w0, unsigned w1, bool sw, const float2 (&h)[8], float2 varphi,
                          float2 a, float2 qs) {
    float2 hs[8];
    if constexpr (CONV) {
      h_star_conv8x2(h, a, varphi, qs, hs);
    } else {
      float2 m1x, m1y;
      h_moment1x2(h, m1x, m1y);
      h_star8x2(h, om, varphi, a, m1x, m1y, qs, hs);
    }
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      if (!(w0 & W_NONE)) write1(w0, i, sw, hs[i - 1].x);
      if (!(w1 & W_NONE)) write1(w1, i, sw, hs[i - 1].y);
    }
  };

  const bool rule = fixed <= 0 && redo == 0;
  const bool last_sums = fixed > 0 && redo == 0 && iter + n >= fixed;
  float2 vold[MNODE / 2];
  // sums of sub-iteration u (its new potential v2 of each pair), in the thread's node order
  auto add_sums = [&](int j, float2 v, float& num, float& den) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int y = row_of(2 * j + c);
      if (x0 + lx < nx && y < th && y0 + y < ny)
        h_change(c ? v.y : v.x, c ? vold[j].y : vold[j].x, num, den);
    }
  };
  auto keep_sums = [&](int u, float num, float den) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      num += __shfl_xor_sync(0xffffffffu, num, o);
      den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    if (lane == 0) s_w[u - 1][warp] = make_float2(num, den);
  };
  // A CTA away from the walls (mask: only the frame index of a tile node counts) runs code
  // without a wall in it: the walled form is several times as long, more than the instruction
  // cache close to the issue slots holds.
  const bool near_wall = k.walls && (y0 - n <= 0 || y0 + th + n >= ny);
  auto sub_iteration = [&](int u, bool sw, unsigned mask) {
    float num = 0.0f, den = 0.0f;
#pragma unroll
    for (int j = 0; j < MNODE / 2; ++j) {
      float2 h[8];
      const unsigned t0 = tf[2 * j] & mask, t1 = tf[2 * j + 1] & mask;
      if ((t0 & W_NONE) && (t1 & W_NONE)) continue;
      read_pair(t0, t1, sw, h);
      const float2 hsum = h_sum8x2(h);
      // (scalar products: a packed one may be contracted with the subtraction of its old value)
      const float2 v = make_float2(h_varphi(hsum.x), h_varphi(hsum.y));
      if (rule && u > 0) add_sums(j, v, num, den);
      vold[j] = v;
      collide_pair(t0, t1, sw, h, v, ta[j], tq[j]);
    }
    if (rule && u > 0) keep_sums(u, num, den);
    const int most = n - u;  // layers still needed
#pragma unroll
    for (int m = 0; m < M::PAIRS; ++m) {
      unsigned w0 = rf[2 * m], w1 = rf[2 * m + 1];
      if ((int)(w0 >> 20) > most) w0 = W_NONE;
      if ((int)(w1 >> 20) > most) w1 = W_NONE;
      if ((w0 & W_NONE) && (w1 & W_NONE)) continue;
      float2 h[8];
      // a missing partner reads the frame's first cells and writes nothing
      w0 &= mask | W_NONE;
      w1 &= mask | W_NONE;
      read_pair(w0, w1, sw, h);
      collide_pair(w0, w1, sw, h, h_varphi2(h_sum8x2(h)), ra[m], rq[m]);
    }
    __syncthreads();
  };
  auto sub_iterations = [&](unsigned mask) {
    for (int u = 0; u < n; u += 2) {
      sub_iteration(u, false, mask);
      if (u + 1 < n) sub_iteration(u + 1, true, mask);
    }
  };
  if (near_wall)
    sub_iterations(0xfffffu);
  else
    sub_iterations(0xffffu | W_NONE);

  // the new state of the tile, to the other copy of h
  {
    float num = 0.0f, den = 0.0f;
    auto finish = [&](bool sw, unsigned mask) {
#pragma unroll
      for (int j = 0; j < MNODE / 2; ++j) {
        float2 h[8];
        read_pair(tf[2 * j] & mask, tf[2 * j + 1] & mask, sw, h);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int y = row_of(2 * j + c), gy = y0 + y;
          if (x0 + lx >= nx || y >= th || gy >= ny) continue;
          const size_t g = EHD_IDX(k, (size_t)gy * nx + x0 + lx, N);
#pragma unroll
          for (int i = 0; i < 8; ++i) dst[i * N + g] = c ? h[i].y : h[i].x;
        }
        if (rule || last_sums) {
          const float2 hsum = h_sum8x2(h);
          add_sums(j, make_float2(h_varphi(hsum.x), h_varphi(hsum.y)), num, den);
        }
      }
    };
    if (!(n & 1))
      finish(false, 0xffffu);  // the own cells: no wall to ask for
    else if (near_wall)
      finish(true, 0xfffffu);
    else
      finish(true, 0xffffu);
    if (rule || last_sums) keep_sums(n, num, den);
  }
  __syncthreads();

  // FP64 partial sums of this tile, one pair per judged sub-iteration
  const int nblocks = (int)(gridDim.x * gridDim.y);
  const int bid = (int)(blockIdx.y * gridDim.x + blockIdx.x);
  const int first = rule ? 1 : n;  // the first judged sub-iteration
  const bool judged = rule || last_sums;
  if (judged && tid >= first - 1 && tid < n) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < MT / 32; ++w) {
      a += (double)s_w[tid][w].x;
      b += (double)s_w[tid][w].y;
    }
    partials[(size_t)(tid - first + 1) * nblocks + bid] = make_double2(a, b);
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(&ctl->ticket_p, 1u) == (unsigned)nblocks - 1u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();

  // the launch's last CTA: the rule, sub-iteration by sub-iteration
  __shared__ double s_red[MT][2];
  int done = 0, conv = 0, stop = n;
  double rel = 0.0;
  if (redo > 0) {
    done = 1;
  } else if (!judged) {
    done = 0;
  } else {
    for (int u = first; u <= n && !done; ++u) {
      double a = 0.0, b = 0.0;
      for (int j = tid; j < nblocks; j += MT) {
        const double2 v = __ldcg(partials + (size_t)(u - first) * nblocks + j);
        a += v.x;
        b += v.y;
      }
      s_red[tid][0] = a;
      s_red[tid][1] = b;
      __syncthreads();
      for (int o = MT / 2; o > 0; o >>= 1) {
        if (tid < o) {
          s_red[tid][0] += s_red[tid + o][0];
          s_red[tid][1] += s_red[tid + o][1];
        }
        __syncthreads();
      }
      const double nm = s_red[0][0], dn = s_red[0][1];
      __syncthreads();
      if (nm == 0.0 && dn == 0.0)
        rel = 0.0;
      else if (dn == 0.0)
        rel = __longlong_as_double(0x7ff0000000000000ll);  // +inf
      else
        rel = sqrt(nm / dn);
      const int it = iter + u;
      if (fixed > 0) {
        done = it >= fixed;
        conv = 1;
      } else {
        conv = (it >= (bad_state ? 1 : ctl->min_iter)) && (rel < ctl->tol);
        done = conv || it >= max_iter;
      }
      stop = u;
    }
  }
  if (tid != 0) return;
  ctl->plaunch += 1;
  ctl->ticket_p = 0u;
  if (redo > 0) {
    // the iteration count and the rule's outcome stand since the launch before
    ctl->redo = 0;
    ctl->parity = parity ^ 1;
    ctl->done = 1;
  } else {
    ctl->iter = iter + stop;
    if (judged) {
      ctl->rel = rel;
      ctl->converged = conv;
    }
    if (fixed <= 0 && !bad_state) keep_aim(ctl, D, iter + stop, done);
    if (done && stop < n) {
      ctl->redo = stop;  // the next launch repeats this one's first sub-iterations
      done = 0;
    } else {
      ctl->parity = parity ^ 1;
      ctl->done = done;
    }
  }
  __threadfence();
  // inside a step graph: the while node repeats this kernel until the loop is done
  if (use_cond) cudaGraphSetConditional(cond, (redo > 0 || done) ? 0u : 1u);
}

namespace {

#ifndef EHD_MULTI_D
#define EHD_MULTI_D 5
#endif
constexpr int MULTI_D = EHD_MULTI_D;
constexpr long long MULTI_WAVE = 304;  // CTAs on the chip at once: two on each of 152 SMs

dim3 multi_grid(const KParams& kp, int th) {
  return dim3((kp.nx + MTX - 1) / MTX, (kp.ny + th - 1) / th);
}
// The tile height for a fixed count: the one whose waves of resident CTAs take least, a CTA's
// time going with its tile and half the ring.  Under the rule full tiles, whose sums are the
// one-step kernel's.
int multi_rows(const KParams& kp, int fixed) {
  if (fixed <= 0) return MTY;
  const int depth = fixed < EHD_MULTI_D ? fixed : EHD_MULTI_D;
  int best = MTY;
  long long best_cost = -1;
  for (int th = MTY; th >= MTY / 2; th -= 2) {  // whole pairs of rows; full tiles where equal
    const dim3 g = multi_grid(kp, th);
    const long long waves = ((long long)g.x * g.y + MULTI_WAVE - 1) / MULTI_WAVE;
    const long long cost = waves * (th + depth);
    if (best_cost < 0 || cost < best_cost) {
      best = th;
      best_cost = cost;
    }
  }
  return best;
}
int multi_blocks(const KParams& kp) {
  const dim3 g = multi_grid(kp, MTY);
  return (int)(g.x * g.y);
}
const void* multi_kernel(const KParams& kp) {
  return kp.scheme == 1 ? (const void*)k_poisson_multi<MULTI_D, true>
                        : (const void*)k_poisson_multi<MULTI_D, false>;
}

}  // namespace

// Lattices that stream several sub-iterations per launch: those beyond the chip's storage, as
// long as the partial sums of every sub-iteration of a launch have room (a fixed count's lower
// tiles, little more than twice as many, keep only one sub-iteration's).
bool multi_ok(const KParams& kp) {
  return !kp.slab && (long long)kp.nx * kp.ny > MULTI_MIN_NODES &&
         (long long)multi_blocks(kp) * MULTI_D <= MAX_PARTIALS;
}
// Whether the moments pass before the loop may leave its per-CTA partials to the coupled pass:
// they keep the front of the array, the loop's sums its end (the moments pass at 1024 x 2048 went
// from 49.3 to 37.8 us without the tickets and the last CTA's reduction).
bool multi_defers(const KParams& kp) {
  return multi_ok(kp) &&
         moments4_blocks(kp) + (long long)multi_blocks(kp) * MULTI_D <= MAX_PARTIALS;
}
cudaError_t multi_prepare(const KParams& kp) {
  return cudaFuncSetAttribute(multi_kernel(kp), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)Multi<MULTI_D>::SMEM);
}
int multi_launches(int fixed) { return (fixed + MULTI_D - 1) / MULTI_D; }
int multi_depth() { return MULTI_D; }

cudaError_t launch_poisson_multi(const KParams& kp, const Buffers& b, int fixed, cudaStream_t st) {
  KParams k = kp;
  int th = multi_rows(kp, fixed);
  float* h = b.h;
  const float2* aq = b.aq;
  double2* partials = b.partials + (MAX_PARTIALS - multi_blocks(kp) * MULTI_D);
  Ctl* ctl = b.ctl;
  cudaGraphConditionalHandle cond = 0;
  int use = 0;
  void* args[] = {&k, &th, &h, &aq, &partials, &ctl, &cond, &use};
  return cudaLaunchKernel(multi_kernel(kp), multi_grid(kp, th), dim3(MT), args,
                          Multi<MULTI_D>::SMEM, st);
}

// With a null `cond` the node leaves no condition (a fixed count's launches in a row).
cudaError_t add_poisson_multi_node(cudaGraph_t g, const cudaGraphNode_t* deps, size_t nd,
                                   cudaGraphNode_t* out, const KParams& kp, const Buffers& b,
                                   int fixed, const cudaGraphConditionalHandle* handle) {
  KParams k = kp;
  int th = multi_rows(kp, fixed);
  float* h = b.h;
  const float2* aq = b.aq;
  double2* partials = b.partials + (MAX_PARTIALS - multi_blocks(kp) * MULTI_D);
  Ctl* ctl = b.ctl;
  cudaGraphConditionalHandle cond = handle ? *handle : 0;
  int use = handle ? 1 : 0;
  void* args[] = {&k, &th, &h, &aq, &partials, &ctl, &cond, &use};
  cudaKernelNodeParams p = {};
  p.func = const_cast<void*>(multi_kernel(kp));
  p.gridDim = multi_grid(kp, th);
  p.blockDim = dim3(MT);
  p.sharedMemBytes = (unsigned)Multi<MULTI_D>::SMEM;
  p.kernelParams = args;
  return cudaGraphAddKernelNode(out, g, deps, nd, &p);
}

}  // namespace ehd
