// Whitening of a step (row a5, Eq. marginal_sigma by the push-through identity:
// z = (lambda I + B^T B)^-1 u): the components of the step's system, and the
// components that one stored inverse solves.
//
// A piece is a connected set of local nodes of one block (see pieces.h).  The
// pieces of the selected blocks, joined wherever a pair occurs in several of
// them, are the connected components of the step's system:
//   * a piece none of whose nodes occurs in another selected block is a whole
//     component; when the inverses (lambda I + B^T B)^-1 were built it is
//     solved here, z = A u, refined with the residual u - K z in double-float
//     (one warp per piece);
//   * every other component (a unit: one or more pieces) goes to the conjugate
//     gradients of k_solve.cu, by size class.
// A piece whose refinement does not converge is handed to k_solve.cu as a unit.
// Every sum runs in a fixed order, so the result is reproducible.
#include <cuda_runtime.h>

#include "dfloat.cuh"
#include "kernels.h"
#include "step_util.cuh"

namespace spider {

namespace {

constexpr int kPieceMaxDev = 256;   // largest piece with a stored inverse
constexpr int kCleanWarps = 8;
constexpr int kRounds = 6;          // refinement rounds (the first is the plain solve)
constexpr int kBlkPieces = 4096;    // pieces of a block at most (4096 observations, two nodes each)
constexpr int kPieceRounds = 64;

__device__ __forceinline__ int32_t plab_root(const int32_t* lab, int32_t g) {
  const volatile int32_t* vl = lab;
  int32_t r = g;
  for (int k = 0; k < 1 << 20; ++k) {
    const int32_t n = vl[r];
    if (n == r) return r;
    r = n;
  }
  return r;
}

// exclusive prefix of x over the active lanes of a full warp; *total = sum
__device__ __forceinline__ int warp_exscan(int x, int lane, int* total) {
  int s = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += y;
  }
  *total = __shfl_sync(0xffffffffu, s, 31);
  return s - x;
}

// The components of the step: labels, then the list of clean pieces, the units
// with their piece lists, and the units of every size class.  One cooperative
// launch instead of a chain of small ones (labels, counts, scan, fill, per-unit
// tables): what bounds it is the latency of its grid barriers (two per hooking
// round, two or three rounds, plus three), not the work.
//   labels: every occurrence of a shared pair links its piece to the piece of
//   the pair's owner occurrence; roots are hooked below smaller roots
//   (atomicMin) and labels compressed until a round changes nothing, so they
//   end as the smallest piece id of each component.
//   lists: positions come from atomic cursors (one atomic per warp); no result
//   depends on the order inside a list.
__global__ void __launch_bounds__(512) k_components(StepView v, int64_t n_b, int use_inv, int multi_grid) {
  __shared__ int any;
  __shared__ int32_t s_rows[kBlkPieces];
  __shared__ uint8_t s_multi[kBlkPieces];
  if (aborted_cta(v)) return;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  int32_t* flags = v.wfast + kWSlots;          // one flag per round
  if (blockIdx.x == 0) {
    for (int i = tid; i < kPieceRounds; i += nt) flags[i] = 0;
    for (int i = tid; i < multi_grid; i += nt) v.msync[i] = v.msync[kMaxGrid + i] = make_int4(0, 0, 0, 0);
  }
  for (int64_t sb = blockIdx.x; sb < n_b; sb += gridDim.x) {
    const int32_t b = v.sel[sb];
    const int32_t g0 = v.blk_piece_off[b], np = v.blk_piece_off[b + 1] - g0;
    const int32_t q0 = v.blk_node_off[b], q1 = v.blk_node_off[b + 1];
    __syncthreads();
    for (int i = tid; i < np; i += nt) {
      s_rows[i] = 0;
      s_multi[i] = 0;
    }
    __syncthreads();
    for (int32_t q = q0 + tid; q < q1; q += nt) {
      const int p = v.node_piece[q];
      if (v.owner_q[q] == q) atomicAdd(&s_rows[p], 1);
      if (v.multi[q]) s_multi[p] = 1;          // every writer stores 1
    }
    __syncthreads();
    for (int i = tid; i < np; i += nt) {
      const int32_t g = g0 + i;
      v.plab[g] = g;
      v.prow[g] = s_rows[i];
      v.pmulti[g] = s_multi[i];
      v.pcount[g] = 0;
      v.urows[g] = 0;
    }
  }
  if (!grid_barrier(v.counters, v.prm->wait_ns)) return;
  int round = 0;
  for (; round < kPieceRounds; ++round) {
    if (tid == 0) any = 0;
    __syncthreads();
    int changed = 0;
    for (int64_t sb = blockIdx.x; sb < n_b; sb += gridDim.x) {
      const int32_t b = v.sel[sb];
      const int32_t q0 = v.blk_node_off[b], q1 = v.blk_node_off[b + 1];
      for (int32_t q = q0 + tid; q < q1; q += nt) {
        if (!v.multi[q]) continue;
        const int32_t qo = v.owner_q[q];
        if (qo == q) continue;
        const int32_t bo = v.owner_b[q];
        const int32_t ga = plab_root(v.plab, v.blk_piece_off[b] + v.node_piece[q]);
        const int32_t gb = plab_root(v.plab, v.blk_piece_off[bo] + v.node_piece[qo]);
        if (ga == gb) continue;
        const int32_t lo = ga < gb ? ga : gb, hi = ga < gb ? gb : ga;
        if (atomicMin(&v.plab[hi], lo) > lo) changed = 1;
      }
    }
    if (changed) any = 1;
    __syncthreads();
    if (tid == 0 && any) flags[round] = 1;
    if (!grid_barrier(v.counters, v.prm->wait_ns)) return;
    if (((volatile int32_t*)flags)[round] == 0) break;
    for (int64_t sb = blockIdx.x; sb < n_b; sb += gridDim.x) {
      const int32_t b = v.sel[sb];
      for (int32_t g = v.blk_piece_off[b] + tid; g < v.blk_piece_off[b + 1]; g += nt)
        v.plab[g] = plab_root(v.plab, g);
    }
    if (!grid_barrier(v.counters, v.prm->wait_ns)) return;
  }
  if (round == kPieceRounds) {
    if (blockIdx.x == 0 && tid == 0) set_error(v.counters, SPIDER_E_TIMEOUT);
    return;
  }
  // pieces and rows (unique pairs) of every component, at its root piece
  for (int64_t sb = blockIdx.x; sb < n_b; sb += gridDim.x) {
    const int32_t b = v.sel[sb];
    for (int32_t g = v.blk_piece_off[b] + tid; g < v.blk_piece_off[b + 1]; g += nt) {
      const int32_t r = v.plab[g];
      atomicAdd(&v.pcount[r], 1);
      atomicAdd(&v.urows[r], v.prow[g]);
    }
  }
  if (!grid_barrier(v.counters, v.prm->wait_ns)) return;
  // unit ids, piece-list ranges and size classes of the roots; the clean list
  for (int64_t sb = blockIdx.x; sb < n_b; sb += gridDim.x) {
    const int32_t b = v.sel[sb];
    const int32_t g1 = v.blk_piece_off[b + 1];
    for (int32_t gb = v.blk_piece_off[b] + (tid & ~31); gb < g1; gb += nt) {
      const int32_t g = gb + lane;
      const bool root = g < g1 && v.plab[g] == g;
      const bool clean = root && use_inv && !v.pmulti[g];
      const bool unit = root && !clean;
      const unsigned mc = __ballot_sync(0xffffffffu, clean), mu = __ballot_sync(0xffffffffu, unit);
      const int rank = __popc((clean ? mc : mu) & ((1u << lane) - 1u));
      int cb = 0, ub = 0, pb = 0, total;
      const int cnt = unit ? v.pcount[g] : 0;
      const int pre = warp_exscan(cnt, lane, &total);
      if (lane == 0) {
        if (mc) cb = atomicAdd(&v.wfast[kWClean], __popc(mc));
        if (mu) {
          ub = atomicAdd(&v.wfast[kWUnits], __popc(mu));
          pb = atomicAdd(&v.wfast[kWPieces], total);
        }
      }
      cb = __shfl_sync(0xffffffffu, cb, 0);
      ub = __shfl_sync(0xffffffffu, ub, 0);
      pb = __shfl_sync(0xffffffffu, pb, 0);
      if (clean) {
        v.clean_list[cb + rank] = g;
        v.clean_blk[cb + rank] = b;
      }
      int cls = -1;
      if (unit) {
        const int32_t u = ub + rank;
        const int rows = v.urows[g];
        v.unit_of[g] = u;
        v.unit_off[u] = pb + pre;
        v.unit_np[u] = cnt;
        v.unit_fill[u] = 0;
        v.unit_rows[u] = rows;
        cls = solve_class(rows, cnt);
        if (cls == kClsMulti)
          v.unit_slot[u] = atomicAdd(&v.wfast[kWRowSlots], (rows + 31) & ~31);
      }
#pragma unroll
      for (int c = 0; c < kClasses; ++c) {
        const unsigned m = __ballot_sync(0xffffffffu, cls == c);
        if (!m) continue;
        int base = 0;
        if (lane == 0) base = atomicAdd(&v.wfast[kWClass0 + c], __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (cls == c) v.cls_list[(int64_t)c * v.cls_cap + base + __popc(m & ((1u << lane) - 1u))] = v.unit_of[g];
      }
    }
  }
  if (!grid_barrier(v.counters, v.prm->wait_ns)) return;
  // the pieces of every unit
  for (int64_t sb = blockIdx.x; sb < n_b; sb += gridDim.x) {
    const int32_t b = v.sel[sb];
    for (int32_t g = v.blk_piece_off[b] + tid; g < v.blk_piece_off[b + 1]; g += nt) {
      if (use_inv && !v.pmulti[g]) continue;
      const int32_t u = v.unit_of[v.plab[g]];
      const int32_t e = v.unit_off[u] + atomicAdd(&v.unit_fill[u], 1);
      v.unit_pieces[e] = g;
      v.unit_pblk[e] = b;
      v.unit_prow[e] = v.prow[g];
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    v.counters[kCntComps] = v.wfast[kWUnits] + v.wfast[kWClean];
    if (v.wfast[kWClass0 + kClsMulti] > 0) v.wfast[kWGeneral] = 1;
  }
}

// ------------------------------------------------------------------ single pieces
// y = A x for one piece held by a warp: A is n x n, symmetric, stored whole, so
// lane i reads A[j][i] over j (consecutive lanes, consecutive words); four
// rows of A in flight per lane.
template <int NS>
__device__ __forceinline__ void warp_matvec(const float* __restrict__ A, int n, const float* x, float* y,
                                            int lane) {
  float acc[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s] = 0.f;
  int j = 0;
  for (; j + 7 < n; j += 8) {
    const float* r0 = A + (size_t)j * n;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i = lane + 32 * s;
      if (i < n) {
        float a[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) a[t] = __ldg(r0 + (size_t)t * n + i);
#pragma unroll
        for (int t = 0; t < 8; ++t) acc[s] = fmaf(a[t], x[j + t], acc[s]);
      }
    }
  }
  for (; j < n; ++j) {
    const float xj = x[j];
    const float* row = A + (size_t)j * n;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i = lane + 32 * s;
      if (i < n) acc[s] = fmaf(__ldg(row + i), xj, acc[s]);
    }
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const int i = lane + 32 * s;
    if (i < n) y[i] = acc[s];
  }
}

__device__ __forceinline__ void warp_matvec_n(const float* A, int n, const float* x, float* y, int lane) {
  if (n <= 32) warp_matvec<1>(A, n, x, y, lane);
  else if (n <= 64) warp_matvec<2>(A, n, x, y, lane);
  else if (n <= 128) warp_matvec<4>(A, n, x, y, lane);
  else warp_matvec<8>(A, n, x, y, lane);
}

// sum over member m's edges of w_e (z_i - z_other) in double-float; zi is the
// member's own value, zoth(j) the value of the member at position j
template <typename ZF>
__device__ __forceinline__ df32 member_bz(const StepView& v, int32_t m, df32 zi, ZF zoth) {
  df32 acc = {0.f, 0.f};
#pragma unroll 4
  for (int32_t t = v.mem_rp[m], t1 = v.mem_rp[m + 1]; t < t1; ++t) {
    const float sw = v.edge_sw[t];
    const df32 zo = zoth((int)v.edge_pos[t]);
    acc = df_add(acc, df_mul(df_two_prod(sw, sw), df_add(zi, df32{-zo.hi, -zo.lo})));
  }
  return acc;
}

struct CleanWarp {
  float uh[kPieceMaxDev], ul[kPieceMaxDev];
  float zh[kPieceMaxDev], zl[kPieceMaxDev];
  float r[kPieceMaxDev], dz[kPieceMaxDev];
};

// Persistent warps over the step's single pieces (one piece at a time each).
__global__ void __launch_bounds__(kCleanWarps * 32) k_whiten_clean(StepView v, float tol) {
  __shared__ CleanWarp sw_[kCleanWarps];
  if (aborted_cta(v)) return;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  CleanWarp& S = sw_[w];
  const float lam = v.lam;
  const int32_t nclean = v.wfast[kWClean];
  int max_rounds = 0;
  for (;;) {
    int32_t c = 0;
    if (lane == 0) c = atomicAdd(&v.wfast[kWCursorC], 1);
    c = __shfl_sync(0xffffffffu, c, 0);
    if (c >= nclean) break;
    const int32_t g = v.clean_list[c];
    const int32_t q0 = v.blk_node_off[v.clean_blk[c]];
    const int32_t m0 = v.piece_node_off[g];
    const int n = v.piece_node_off[g + 1] - m0;
    const float* A = v.piece_inv + v.piece_inv_off[g];
    float uu = 0.f;
    for (int i = lane; i < n; i += 32) {
      const int32_t u = v.loc2u[q0 + v.piece_nodes[m0 + i]];
      S.uh[i] = v.rhs[u];
      S.ul[i] = v.rhs_lo[u];
      S.zh[i] = 0.f;
      S.zl[i] = 0.f;
      uu = fmaf(S.uh[i], S.uh[i], uu);
    }
    uu = warp_sum(uu);
    __syncwarp();
    int round = 0;
    bool done = false;
    for (; round < kRounds; ++round) {
      float rr = 0.f;
      for (int i = lane; i < n; i += 32) {
        float r;
        if (round == 0) {
          r = S.uh[i] + S.ul[i];
        } else {
          const df32 zi = {S.zh[i], S.zl[i]};
          const df32 bz = member_bz(v, m0 + i, zi, [&](int j) { return df32{S.zh[j], S.zl[j]}; });
          df32 rd = df_add(df32{S.uh[i], S.ul[i]}, df_mul_f(zi, -lam));
          rd = df_add(rd, df32{-bz.hi, -bz.lo});
          r = rd.hi;
        }
        S.r[i] = r;
        rr = fmaf(r, r, rr);
      }
      rr = warp_sum(rr);
      __syncwarp();
      if (rr <= tol * tol * uu) {
        done = true;
        break;
      }
      warp_matvec_n(A, n, S.r, S.dz, lane);
      __syncwarp();
      for (int i = lane; i < n; i += 32) {
        const df32 z = df_add_f(df32{S.zh[i], S.zl[i]}, S.dz[i]);
        S.zh[i] = z.hi;
        S.zl[i] = z.lo;
      }
      __syncwarp();
    }
    if (!done) {
      // a unit of its own for the conjugate gradients (the late class)
      if (lane == 0) {
        const int32_t u = atomicAdd(&v.wfast[kWUnits], 1), e = atomicAdd(&v.wfast[kWPieces], 1);
        v.unit_off[u] = e;
        v.unit_np[u] = 1;
        v.unit_rows[u] = n;
        v.unit_pieces[e] = g;
        v.unit_pblk[e] = v.clean_blk[c];
        v.unit_prow[e] = n;
        v.cls_list[(int64_t)kClsLate * v.cls_cap + atomicAdd(&v.wfast[kWClass0 + kClsLate], 1)] = u;
        v.wfast[kWGeneral] = 1;
      }
      __syncwarp();
      continue;
    }
    if (round > max_rounds) max_rounds = round;
    for (int i = lane; i < n; i += 32) {
      const int32_t u = v.loc2u[q0 + v.piece_nodes[m0 + i]];
      v.z[u] = S.zh[i];
      v.z_lo[u] = S.zl[i];
    }
    __syncwarp();
  }
  if (lane == 0 && max_rounds > 0) atomicMax(&v.counters[kCntCompIters], max_rounds);
}

}  // namespace

int piece_max_nodes() { return kPieceMaxDev; }

int whiten_clean_grid(int num_sms) {
  int a = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_whiten_clean, kCleanWarps * 32, 0) != cudaSuccess ||
      a < 1)
    return 0;
  return num_sms * a;
}

int components_grid(int num_sms) {
  int a = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_components, 512, 0) != cudaSuccess || a < 1) return 0;
  return num_sms * (a < 2 ? a : 2);
}

// The whitening solve of a step.  The component classes and the clean pieces
// run side by side on the branch streams; the multi-CTA class, the longest
// when there is one, is launched on st itself.
cudaError_t launch_whiten(const StepView& v, int64_t n_b, const WhitenPlan& w, int max_it, float tol,
                          cudaStream_t st, const Branches* br, const cudaEvent_t* ev) {
  if (!v.whiten) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(v.wfast, 0, kWSlots * sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  {
    StepView vv = v;
    int64_t nb = n_b;
    int inv = w.use_inv, mg = w.multi_grid;
    // a CTA per block; at least two, at most what is resident at once
    int64_t grid = n_b < 2 ? 2 : n_b;
    if (grid > w.cc_grid) grid = w.cc_grid;
    void* args[] = {&vv, &nb, &inv, &mg};
    e = cudaLaunchCooperativeKernel((const void*)k_components, dim3((unsigned)grid), dim3(512), args, 0, st);
    if (e != cudaSuccess) return e;
  }
  if (ev && (e = cudaEventRecord(ev[0], st)) != cudaSuccess) return e;
  const bool clean_side = w.use_inv && w.clean_share > 0 && br;
  if (br) {
    if ((e = cudaEventRecord(br->fork, st)) != cudaSuccess) return e;
    for (int i = 0; i < kBranches; ++i)
      if ((e = cudaStreamWaitEvent(br->s[i], br->fork, 0)) != cudaSuccess) return e;
  }
  auto lane = [&](int i) { return br ? br->s[i] : st; };
  // Classes that no component of this catalog can be of are not launched (on the
  // 200-event catalog three of five: 4 us each to find their lists empty).
  auto reached = [&](int cls) { return w.top_class >= cls; };
  if (reached(kClsMulti) && (e = launch_solve_multi(v, max_it, tol, w.multi_grid, st)) != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[2], st)) != cudaSuccess) return e;
  // The two classes whose CTAs take a whole SM first, the stored inverses' warps after
  // them: ahead of them, those warps kept the CTAs waiting for room (1M-event BF16 step:
  // 2.79 ms, 2.76 in this order; after the 8-warp class 2.84, and the one-warp class
  // before the 8-warp one costs the 200-event chain 6 %).
  const int cta_classes[3] = {kClsCta, kClsMid, kClsSmall};
  for (int i = 0; i < 3; ++i) {
    if (i == 2 && clean_side) {
      const int g = w.clean_grid * w.clean_share / 4;
      k_whiten_clean<<<g > 0 ? g : 1, kCleanWarps * 32, 0, lane(4)>>>(v, tol);
    }
    if (reached(cta_classes[i]) &&
        (e = launch_solve_class(v, cta_classes[i], max_it, tol, w.num_sms * w.cta_mult, lane(i))) != cudaSuccess)
      return e;
  }
  if ((e = launch_solve_class(v, kClsWarp, max_it, tol, w.num_sms * w.warp_mult, lane(3))) != cudaSuccess) return e;
  if (br)
    for (int i = 0; i < 4; ++i) {
      if ((e = cudaEventRecord(br->join[i], br->s[i])) != cudaSuccess) return e;
      if ((e = cudaStreamWaitEvent(st, br->join[i], 0)) != cudaSuccess) return e;
    }
  if (ev && (e = cudaEventRecord(ev[1], st)) != cudaSuccess) return e;
  if (br) {
    if ((e = cudaEventRecord(br->join[4], br->s[4])) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(st, br->join[4], 0)) != cudaSuccess) return e;
  }
  if (w.use_inv) {
    if (!clean_side) k_whiten_clean<<<w.clean_grid, kCleanWarps * 32, 0, st>>>(v, tol);
    if (ev && (e = cudaEventRecord(ev[3], st)) != cudaSuccess) return e;
    if ((e = launch_solve_class(v, kClsLate, max_it, tol, w.num_sms, st)) != cudaSuccess) return e;
  } else if (ev && (e = cudaEventRecord(ev[3], st)) != cudaSuccess) {
    return e;
  }
  return cudaGetLastError();
}

}  // namespace spider
