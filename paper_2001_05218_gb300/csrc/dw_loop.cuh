// dw_loop.cuh -- the CG iterations of small lattices in one kernel.
//
// On a lattice that fills the GPU for a few microseconds an iteration of CG (here
// the even-odd one) is a chain of latencies: six kernels and three finishing kernels
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

enum Mode { MODE_EO = 0, MODE_FULL = 1, MODE_NORMAL = 2, MODE_HERM = 3 };

constexpr int kLoopThreads = 512;
constexpr int kLoopCols = 16;       // most columns (system, right-hand side)
constexpr int kLoopPartials = 2048; // most 32-site tiles of one column: k_finish sums those with 256 threads

// All blocks of the (cooperative) launch meet: a block adds itself to the count
// (release) and polls it (acquire) until every block of this round has, one trip
// to L2 and back after the last arrival.  `round` is the count at which this
// barrier opens; the count runs on through a solve's launches (Flags::bar_base).
// Every wait is bounded: about a second of polls, then the barrier reports
// failure to its whole block, which leaves; the blocks that wait for it run out
// in turn, and the host solves again with the separate kernels.
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

// Sums the partials of every column (ntiles per system: PARS parities) and leaves
// the totals in sum[]: columns two at a time, 256 threads each, in k_finish's order.
template <int PARS>
__device__ __forceinline__ void column_sums(const Batch& B, const RedArgs& ra, int ncols, int buf, double* sum) {
  __shared__ DF wpart[2][8];
  const int half = threadIdx.x >> 8, t = threadIdx.x & 255, lane = t & 31, warp = t >> 5;
  for (int c0 = 0; c0 < ncols; c0 += 2) {
    const int c = c0 + half;
    DF v = df_make(0.f, 0.f);
    if (c < ncols) {
      const int nrhs = B.sd[0].nrhs, si = c / nrhs, r = c - si * nrhs;
      const SysDesc& S = B.sd[si];
      const int ntiles = PARS * S.tpp;
      v = partial_share(ra.partial + (size_t)PARS * S.part0 + (size_t)(buf * nrhs + r) * ntiles, ntiles, t, 256);
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

// One work item: a 32-site tile of one parity of one right-hand side (items of
// both parities: the odd ones follow all even ones).
struct LoopItem {
  int si, r, par, tile, s;
  bool valid;
};
template <int PARS>
__device__ __forceinline__ LoopItem loop_item(const Batch& B, const ColState* cs, int i, int n, int par) {
  LoopItem t;
  t.valid = false;
  t.par = par;
  if (i < n) {
    if (PARS == 2) {
      t.par = i >= n / 2;
      i -= t.par * (n / 2);
    }
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
// The partial of item t in buffer buf.
template <int PARS>
__device__ __forceinline__ DF* loop_partial(const RedArgs& ra, const SysDesc& S, const LoopItem& t, int buf) {
  return ra.partial + (size_t)PARS * S.part0 + (size_t)(buf * S.nrhs + t.r) * (PARS * S.tpp) +
         (PARS == 2 ? t.par * S.tpp : 0) + t.tile;
}

// What a hop does with H in: store it, or xpay with |out|^2, Re <x, out> or
// nothing summed into buffer buf.
enum LoopEpi { LE_OUT = 0, LE_NORM, LE_DOT, LE_XPAY };

// One hop over all items: output parity par, or both (PARS = 2).
template <int L, bool C12, bool SPLIT, bool DAG, int OP, int PARS, int COEF>
__device__ __forceinline__ void loop_hop(const Batch& B, const RedArgs& ra, const ColState* cs, float* parts, int n, int par,
                                         int in_slot, int kind, int out_slot, int x_slot, int buf) {
  using R = typename Spin<L>::R;
  constexpr int SF = DAG ? +1 : -1;
  constexpr int kPer = SPLIT ? kLoopThreads / 128 : kLoopThreads / 32;  // items a block works on at a time
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int mu = warp & 3, group = warp >> 2;
  const InOne<L> in{in_slot};
  for (int i0 = blockIdx.x * kPer; i0 < n; i0 += gridDim.x * kPer) {
    const LoopItem t = loop_item<PARS>(B, cs, i0 + (SPLIT ? group : warp), n, par);
    const SysDesc& S = B.sd[t.valid ? t.si : 0];
    const bool ok = t.valid && t.s < S.vh;
    Cx<R> acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = cx((R)0, (R)0);
    typename Spin<L>::Packed xw;  // the xpay operand, on its way during the hop
    if (ok && kind != LE_OUT && (!SPLIT || mu == 0))
      xw = Spin<L>::load_packed(slot_ptr(S, x_slot, t.r, t.par), S.vh, t.s);
    if (ok) {
      const Coord c = coord_of(S, t.s, t.par);
      const int pin = t.par ^ 1;
      const char* own = slot_ptr(S, S_LLO, 0, t.par);
      const char* nbr = slot_ptr(S, S_LLO, 0, pin);
      const long long mu_stride = (long long)Link<L, C12>::kBytes * S.vh;
      if constexpr (OP == OP_LAPLACE) {
        laplace_dirs<L, L, C12>(S, in, c, t.s, t.r, pin, own, nbr, mu_stride, acc);
      } else {
        if (!SPLIT || mu == 0) hop_mu<0, L, L, C12, SF>(S, in, c, t.s, t.r, pin, own, nbr, mu_stride, acc);
        if (!SPLIT || mu == 1) hop_mu<1, L, L, C12, SF>(S, in, c, t.s, t.r, pin, own, nbr, mu_stride, acc);
        if (!SPLIT || mu == 2) hop_mu<2, L, L, C12, SF>(S, in, c, t.s, t.r, pin, own, nbr, mu_stride, acc);
        if (!SPLIT || mu == 3) hop_mu<3, L, L, C12, SF>(S, in, c, t.s, t.r, pin, own, nbr, mu_stride, acc);
      }
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
      if (kind == LE_OUT) {
        if (ok) EpiOut<L, C_ONE>{out_slot, G_ALL}.write(S, t.par, t.r, t.s, acc, nrm);
      } else {
        if (ok) {
          Cx<R> xv[12];
          Spin<L>::unpack(xw, xv);
          if constexpr (OP == OP_LAPLACE) {
            const EpiXpayDot<L, L, COEF> epi{out_slot, x_slot, G_ALL};
            epi.commit(S, t.par, t.r, t.s, epi.form(S, acc, xv, nrm));
          } else {
            const EpiXpay<L, L, COEF, true> epi{out_slot, x_slot, G_ALL};
            epi.commit(S, t.par, t.r, t.s, epi.form(S, acc, xv, nrm));
          }
        }
        if (kind != LE_XPAY) {
          nrm = warp_sum_lane0(nrm);
          if (lane == 0) *loop_partial<PARS>(ra, S, t, buf) = to_partial(nrm);
        }
      }
    }
    if constexpr (SPLIT) __syncthreads();  // parts are free again
  }
}

// B: plan with 32 sites and one right-hand side per block.  rel, loop: the
// conditions of the reliable-update and the while node.  MODE: the solver's
// (even-odd Wilson; the normal equations on both parities; the Laplacian).
template <int L, int A, bool C12, bool SPLIT, int MODE>
__global__ void __launch_bounds__(kLoopThreads, 1)
    k_cg_loop(const __grid_constant__ Batch B, RedArgs ra, unsigned long long rel, unsigned long long loop) {
  constexpr bool kNormal = MODE == MODE_NORMAL, kHerm = MODE == MODE_HERM;
  constexpr int OP = kHerm ? OP_LAPLACE : OP_WILSON, PARS = kNormal ? 2 : 1;
  __shared__ ColState cs[kLoopCols];
  __shared__ double sum[kLoopCols];
  __shared__ float parts[SPLIT ? 4 * 3 * 24 * 32 : 1];
  using R = typename Spin<L>::R;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ncols = B.nsys * B.sd[0].nrhs, n = PARS * B.ntot * B.sd[0].nrhs;
  Flags* f = ra.flags;
  if (tid < ncols) cs[tid] = ra.cols[tid];
  // a reliable update came before: go on at z = D^dag r, or where z = r (its
  // finishing kernel has formed beta) at the update of p
  bool resume = __ldcg(&f->loops) > 0;
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
      if constexpr (kNormal) {
        // t = D p, |t|^2 = p^dag A p; w = D^dag t
        loop_hop<L, C12, SPLIT, false, OP, 2, C_MK>(B, ra, cs, parts, n, 0, S_P, LE_NORM, S_T, S_P, 0);
        if (!(good = grid_barrier(f, round))) break;
        loop_hop<L, C12, SPLIT, true, OP, 2, C_MK>(B, ra, cs, parts, n, 0, S_T, LE_XPAY, S_W, S_T, 0);
      } else {
        // w = Dhat p and |w|^2 (the Laplacian: p^dag w)
        loop_hop<L, C12, SPLIT, false, OP, 1, C_MK2>(B, ra, cs, parts, n, 1, S_P, LE_OUT, S_T, 0, 0);
        if (!(good = grid_barrier(f, round))) break;
        loop_hop<L, C12, SPLIT, false, OP, 1, C_MK2>(B, ra, cs, parts, n, 0, S_T, kHerm ? LE_DOT : LE_NORM, S_W, S_P, 0);
      }
      if (!(good = grid_barrier(f, round))) break;
      column_sums<PARS>(B, ra, ncols, 0, sum);
      if (tid < ncols && cs[tid].active && !form_alpha(cs[tid], sum[tid])) {
        cs[tid].active = 0;
        cs[tid].status = 7;  // DW_ERR_BREAKDOWN
      }
      __syncthreads();
      // r -= alpha w, |r|^2
      for (int i = blockIdx.x * (kLoopThreads / 32) + warp; i < n; i += gridDim.x * (kLoopThreads / 32)) {
        const LoopItem t = loop_item<PARS>(B, cs, i, n, 0);
        if (!t.valid) continue;
        const SysDesc& S = B.sd[t.si];
        typename RedT<R>::type nrm = red_zero(typename RedT<R>::type());
        if (t.s < S.vh) {
          const auto w = update_r_site<L>(S, t.par, t.r, t.s, cs[S.col0 + t.r], nrm);
          Spin<L>::store_packed(slot_wptr(S, S_R, t.r, t.par), S.vh, t.s, w);
        }
        nrm = warp_sum_lane0(nrm);
        if (lane == 0) *loop_partial<PARS>(ra, S, t, 1) = to_partial(nrm);
      }
      if (blockIdx.x == 0 && tid == 0) f->late = cs[0].deadline_ns != 0ull && globaltimer_ns() > cs[0].deadline_ns;
      if (!(good = grid_barrier(f, round))) break;
      const bool late = __ldcg(&f->late) != 0;
      column_sums<PARS>(B, ra, ncols, 1, sum);
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
    if constexpr (!kNormal && !kHerm) {
      // z = Dhat^dag r, beta
      loop_hop<L, C12, SPLIT, true, OP, 1, C_MK2>(B, ra, cs, parts, n, 1, S_R, LE_OUT, S_T, 0, 0);
      if (!(good = grid_barrier(f, round))) break;
      loop_hop<L, C12, SPLIT, true, OP, 1, C_MK2>(B, ra, cs, parts, n, 0, S_T, LE_NORM, S_Z, S_R, 0);
      if (!(good = grid_barrier(f, round))) break;
      column_sums<PARS>(B, ra, ncols, 0, sum);
      if (tid < ncols && cs[tid].active) form_beta(cs[tid], sum[tid]);
      __syncthreads();
    }
    // xl += alpha p, p = z + beta p
    for (int i = blockIdx.x * (kLoopThreads / 32) + warp; i < n; i += gridDim.x * (kLoopThreads / 32)) {
      const LoopItem t = loop_item<PARS>(B, cs, i, n, 0);
      if (!t.valid) continue;
      const SysDesc& S = B.sd[t.si];
      if (t.s < S.vh) update_p_site<L, A>(S, t.par, t.r, t.s, cs[S.col0 + t.r]);
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
