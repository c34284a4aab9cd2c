// dw_loop.cuh -- the CG iterations of small lattices in one kernel.
//
// On a lattice that fills the GPU for a few microseconds an iteration of the
// even-odd CG is a chain of latencies: six kernels and three finishing kernels
// of 2.5 to 8 us each, most of it launch, first loads and drain (8^4: 60 us per
// iteration for 0.2 us worth of bytes).  Here one cooperative launch iterates
// until some column wants a reliable update (or none is left): the phases are
// separated by a grid barrier, every block sums the partials and forms the CG
// scalars itself, and the column states live in shared memory.  Links stay in
// L1 where they fit; spinors are re-read after each barrier.
//
// The arithmetic is that of the separate kernels with blocks of 32 sites
// (k_hop or k_hop_split, k_update_r, k_update_p, k_finish with 256 threads), in
// the same order, so the host-stepped loop gives bitwise the same results.
#pragma once

#include "dw_exec.cuh"

namespace dw {

constexpr int kLoopThreads = 512;
constexpr int kLoopCols = 16;       // most columns (system, right-hand side)
constexpr int kLoopPartials = 2048; // most 32-site tiles of one column: k_finish sums those with 256 threads

// All blocks of the (cooperative) launch meet: a block adds itself to the count
// (release) and polls it (acquire) until every block of this round has, one trip
// to L2 and back after the last arrival.  `round` is the count at which this
// barrier opens; the count runs on through a solve's launches (Flags::bar_base).
// Every wait is bounded: about a second of polls, then the barrier reports
// failure to its whole block, which leaves; the blocks that wait for it run out
// in turn.
__device__ __forceinline__ bool grid_barrier(Flags* f, unsigned& round) {
  __shared__ int ok_;
  __syncthreads();
  if (gridDim.x == 1) return true;
  round += gridDim.x;
  if (threadIdx.x == 0) {
    int ok = 1, polls = 0;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&f->bar_count) : "memory");
    for (;;) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&f->bar_count) : "memory");
      if ((int)(v - round) >= 0) break;
      if (++polls > (1 << 21)) {
        f->bar_error = 1;
        ok = 0;
        break;
      }
    }
    ok_ = ok;
  }
  __syncthreads();
  return ok_ != 0;
}

// Sums the partials of every column and leaves the totals in sum[]: columns
// two at a time, 256 threads each, in k_finish's order.
__device__ __forceinline__ void column_sums(const Batch& B, const RedArgs& ra, int ncols, int buf, double* sum) {
  __shared__ DF wpart[2][8];
  const int half = threadIdx.x >> 8, t = threadIdx.x & 255, lane = t & 31, warp = t >> 5;
  for (int c0 = 0; c0 < ncols; c0 += 2) {
    const int c = c0 + half;
    DF v = df_make(0.f, 0.f);
    if (c < ncols) {
      const int nrhs = B.sd[0].nrhs, si = c / nrhs, r = c - si * nrhs;
      const SysDesc& S = B.sd[si];
      v = partial_share(ra.partial + S.part0 + (size_t)(buf * nrhs + r) * S.tpp, S.tpp, t, 256);
    }
    v = warp_sum_lane0(v);
    if (lane == 0) wpart[half][warp] = v;
    __syncthreads();
    if (warp == 0) {
      v = lane < 8 ? wpart[half][lane] : df_make(0.f, 0.f);
      v = warp_sum_lane0(v, 4);
      if (lane == 0 && c < ncols) sum[c] = (double)v;
    }
    __syncthreads();
  }
}

// The sites of one work item (a 32-site tile of one right-hand side).
struct LoopItem {
  int si, r, tile, s;
  bool valid;
};
__device__ __forceinline__ LoopItem loop_item(const Batch& B, const ColState* cs, int i, int n) {
  LoopItem t;
  t.valid = false;
  if (i < n) {
    const int nrhs = B.sd[0].nrhs;
    const int b = nrhs == 1 ? i : i / nrhs;
    t.r = i - b * nrhs;
    t.si = block_system(B, b);
    const SysDesc& S = B.sd[t.si];
    t.tile = b - S.tile0;
    t.s = t.tile * 32 + (threadIdx.x & 31);
    t.valid = cs[S.col0 + t.r].active != 0;  // the same for the whole warp
  }
  return t;
}

// One parity hop over all items: out(par) = H in(1 - par), or with xpay
// out = x + C_MK2 H in and the partials of |out|^2 into buffer buf.
template <int L, bool C12, bool SPLIT, bool DAG>
__device__ __forceinline__ void loop_hop(const Batch& B, const RedArgs& ra, const ColState* cs, float* parts, int n, int par,
                                         int in_slot, bool xpay, int out_slot, int x_slot, int buf) {
  using R = typename Spin<L>::R;
  constexpr int SF = DAG ? +1 : -1;
  constexpr int kPer = SPLIT ? kLoopThreads / 128 : kLoopThreads / 32;  // items a block works on at a time
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int mu = warp & 3, group = warp >> 2;
  const InOne<L> in{in_slot};
  for (int i0 = blockIdx.x * kPer; i0 < n; i0 += gridDim.x * kPer) {
    const LoopItem t = loop_item(B, cs, i0 + (SPLIT ? group : warp), n);
    const SysDesc& S = B.sd[t.valid ? t.si : 0];
    const bool ok = t.valid && t.s < S.vh;
    Cx<R> acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = cx((R)0, (R)0);
    typename Spin<L>::Packed xw;  // the xpay operand, on its way during the hop
    if (ok && xpay && (!SPLIT || mu == 0)) xw = Spin<L>::load_packed(slot_ptr(S, x_slot, t.r, par), S.vh, t.s);
    if (ok) {
      const Coord c = coord_of(S, t.s, par);
      const int pin = par ^ 1;
      const char* own = slot_ptr(S, S_LLO, 0, par);
      const char* nbr = slot_ptr(S, S_LLO, 0, pin);
      const long long mu_stride = (long long)Link<L, C12>::kBytes * S.vh;
      if (!SPLIT || mu == 0) hop_mu<0, L, L, C12, SF>(S, in, c, t.s, t.r, pin, own, nbr, mu_stride, acc);
      if (!SPLIT || mu == 1) hop_mu<1, L, L, C12, SF>(S, in, c, t.s, t.r, pin, own, nbr, mu_stride, acc);
      if (!SPLIT || mu == 2) hop_mu<2, L, L, C12, SF>(S, in, c, t.s, t.r, pin, own, nbr, mu_stride, acc);
      if (!SPLIT || mu == 3) hop_mu<3, L, L, C12, SF>(S, in, c, t.s, t.r, pin, own, nbr, mu_stride, acc);
    }
    if constexpr (SPLIT) {
      float* mine = parts + group * (3 * 24 * 32) + lane;
      if (mu != 0) {
#pragma unroll
        for (int k = 0; k < 12; ++k) {
          mine[((mu - 1) * 24 + 2 * k) * 32] = acc[k].re;
          mine[((mu - 1) * 24 + 2 * k + 1) * 32] = acc[k].im;
        }
      }
      __syncthreads();
      if (mu == 0) {
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
          for (int k = 0; k < 12; ++k)
            acc[k] = acc[k] + cx(mine[(m * 24 + 2 * k) * 32], mine[(m * 24 + 2 * k + 1) * 32]);
      }
    }
    if ((!SPLIT || mu == 0) && t.valid) {
      typename RedT<R>::type nrm = red_zero(typename RedT<R>::type());
      if (!xpay) {
        if (ok) EpiOut<L, C_ONE>{out_slot, G_ALL}.write(S, par, t.r, t.s, acc, nrm);
      } else {
        if (ok) {
          const EpiXpay<L, L, C_MK2, true> epi{out_slot, x_slot, G_ALL};
          Cx<R> xv[12];
          Spin<L>::unpack(xw, xv);
          epi.commit(S, par, t.r, t.s, epi.form(S, acc, xv, nrm));
        }
        nrm = warp_sum_lane0(nrm);
        if (lane == 0) ra.partial[S.part0 + (size_t)(buf * S.nrhs + t.r) * S.tpp + t.tile] = to_partial(nrm);
      }
    }
    if constexpr (SPLIT) __syncthreads();  // parts are free again
  }
}

// B: plan with 32 sites and one right-hand side per block, even-odd Wilson
// system.  rel, loop: the conditions of the reliable-update and the while node.
template <int L, int A, bool C12, bool SPLIT>
__global__ void __launch_bounds__(kLoopThreads, 1)
    k_cg_loop(const __grid_constant__ Batch B, RedArgs ra, unsigned long long rel, unsigned long long loop) {
  __shared__ ColState cs[kLoopCols];
  __shared__ double sum[kLoopCols];
  __shared__ float parts[SPLIT ? 4 * 3 * 24 * 32 : 1];
  using R = typename Spin<L>::R;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ncols = B.nsys * B.sd[0].nrhs, n = B.ntot * B.sd[0].nrhs;
  Flags* f = ra.flags;
  if (tid < ncols) cs[tid] = ra.cols[tid];
  bool resume = __ldcg(&f->loops) > 0;  // a reliable update came before: go on at z = D^dag r
  unsigned round = __ldcg(&f->bar_base);
  __syncthreads();
  bool good = true;
  for (;;) {
    int active = 0, rel_wanted = 0;
    for (int c = 0; c < ncols; ++c) {
      active += cs[c].active;
      rel_wanted += cs[c].do_rel;
    }
    if (active == 0 || rel_wanted > 0 || !good) break;
    if (!resume) {
      // w = Dhat p, |w|^2
      loop_hop<L, C12, SPLIT, false>(B, ra, cs, parts, n, 1, S_P, false, S_T, 0, 0);
      if (!(good = grid_barrier(f, round))) break;
      loop_hop<L, C12, SPLIT, false>(B, ra, cs, parts, n, 0, S_T, true, S_W, S_P, 0);
      if (!(good = grid_barrier(f, round))) break;
      column_sums(B, ra, ncols, 0, sum);
      if (tid < ncols && cs[tid].active && !form_alpha(cs[tid], sum[tid])) {
        cs[tid].active = 0;
        cs[tid].status = 7;  // DW_ERR_BREAKDOWN
      }
      __syncthreads();
      // r -= alpha w, |r|^2
      for (int i = blockIdx.x * (kLoopThreads / 32) + warp; i < n; i += gridDim.x * (kLoopThreads / 32)) {
        const LoopItem t = loop_item(B, cs, i, n);
        if (!t.valid) continue;
        const SysDesc& S = B.sd[t.si];
        typename RedT<R>::type nrm = red_zero(typename RedT<R>::type());
        if (t.s < S.vh) {
          const auto w = update_r_site<L>(S, 0, t.r, t.s, cs[S.col0 + t.r], nrm);
          Spin<L>::store_packed(slot_wptr(S, S_R, t.r, 0), S.vh, t.s, w);
        }
        nrm = warp_sum_lane0(nrm);
        if (lane == 0) ra.partial[S.part0 + (size_t)(S.nrhs + t.r) * S.tpp + t.tile] = to_partial(nrm);
      }
      if (blockIdx.x == 0 && tid == 0) f->late = cs[0].deadline_ns != 0ull && globaltimer_ns() > cs[0].deadline_ns;
      if (!(good = grid_barrier(f, round))) break;
      const bool late = __ldcg(&f->late) != 0;
      column_sums(B, ra, ncols, 1, sum);
      if (tid < ncols && cs[tid].active && !count_update(cs[tid], sum[tid], late)) {
        cs[tid].active = 0;
        cs[tid].status = 7;
      }
      __syncthreads();
      rel_wanted = 0;
      for (int c = 0; c < ncols; ++c) rel_wanted += cs[c].do_rel;
      if (rel_wanted > 0) break;
    }
    resume = false;
    // z = Dhat^dag r, beta
    loop_hop<L, C12, SPLIT, true>(B, ra, cs, parts, n, 1, S_R, false, S_T, 0, 0);
    if (!(good = grid_barrier(f, round))) break;
    loop_hop<L, C12, SPLIT, true>(B, ra, cs, parts, n, 0, S_T, true, S_Z, S_R, 0);
    if (!(good = grid_barrier(f, round))) break;
    column_sums(B, ra, ncols, 0, sum);
    if (tid < ncols && cs[tid].active) form_beta(cs[tid], sum[tid]);
    __syncthreads();
    // xl += alpha p, p = z + beta p
    for (int i = blockIdx.x * (kLoopThreads / 32) + warp; i < n; i += gridDim.x * (kLoopThreads / 32)) {
      const LoopItem t = loop_item(B, cs, i, n);
      if (!t.valid) continue;
      const SysDesc& S = B.sd[t.si];
      if (t.s < S.vh) update_p_site<L, A>(S, 0, t.r, t.s, cs[S.col0 + t.r]);
    }
    if (!(good = grid_barrier(f, round))) break;
  }
  // every block holds the same states; the first writes them back
  if (blockIdx.x == 0) {
    if (tid < ncols) ra.cols[tid] = cs[tid];
    if (tid == 0) {
      int active = 0, wanted = 0;
      for (int c = 0; c < ncols; ++c) {
        active += cs[c].active;
        wanted += cs[c].do_rel;
      }
      if (!good) active = wanted = 0;
      f->active = active;
      f->rel_pending = wanted;
      f->loops += 1;
      f->bar_base = round;
      // with a reliable update pending its finishing kernel decides anew
      cudaGraphSetConditional(rel, wanted > 0 ? 1u : 0u);
      cudaGraphSetConditional(loop, active > 0 && f->loops < f->max_loops ? 1u : 0u);
    }
  }
}

}  // namespace dw
