// Conjugate gradients on the components of the step's whitening system (row a5,
// (lambda I + B^T B) z = B^T r, Eq. marginal_sigma): every component that no
// single stored inverse covers, one component to one warp, one CTA or several
// CTAs by its size (the lists come from k_components).
//
// Each component iterates with its own scalars: the largest of a full-batch
// catalog (4000 nodes, lambda / degree ~ 1e-3) needs ~80 iterations alone,
// where one iteration over all components at once needs ~250 (the union of
// their spectra).  Jacobi-preconditioned CG in FP32; when the recurrence's
// residual has fallen by 1e-3, or to the target, the correction is added to z
// in double-float and the residual replaced by u - A z evaluated in
// double-float, keeping the search direction (no restart: ~10-25 % fewer
// iterations than restarting).
//
// Rows are the component's unique pairs: the owner occurrences of its pieces in
// ascending piece id and member order, so their order, and with it every sum,
// does not depend on how lists were filled.  A row belongs to one lane; the
// entries of the 32 rows of a slice are stored step by step (the t-th entries
// of all rows side by side), so a warp's loads are contiguous.  One thread per
// row over row-contiguous entries touched 32 cache lines per load and was
// bound by the load unit (48 us per iteration over 110 k rows and 4 M entries).
//
// Measured and left out: clusters of two and four CTAs that write their y into
// each other's shared memory.  A component of 700 rows took 3100 cycles an
// iteration on two CTAs, 3400 on one, and clusters, which wait for whole SMs at once, started
// after every smaller class: steps with many components lost 5-30 %.
#include <cuda_runtime.h>

#include "dfloat.cuh"
#include "kernels.h"
#include "pool.h"
#include "step_util.cuh"

namespace spider {

namespace {

constexpr float kReplace = 1e-6f;    // (1e-3)^2: residual drop between replacements
// Squared share of the caller's tolerance that the iteration aims at.  The
// gradient sums q = (u - B z) / sigma^2 with cancellation and amplifies what is
// left of |u - A z| by up to degree / lambda, a few hundred: stopping at the
// tolerance itself (1e-7) leaves 4e-6 in a minibatch gradient, a hundredth of it
// 1e-7.
constexpr float kAim = 1e-4f;
constexpr int kMaxReplace = 8;       // replacements at most
constexpr int kMultiThreads = 512;   // threads per CTA of the multi-CTA class

// Where the entries of a slice are.  Steps [0, ss) sit in shared memory from sb
// on, 32 words a step (rows shorter than `steps` padded with zero weights, so
// the loop needs no predicate); the other steps in the pool in global memory from
// pool_first(gb) on: padded the same way (gb >= 0), or with the t-th entries
// of the rows that have one side by side (slices of very uneven rows, where
// padding would more than double the entries).  ss and steps are multiples of 4.
struct Slice {
  int sb, ss, gb, len, steps;
};
struct EntrySmem {
  float* sw;
  uint16_t* col;
};

// entries of a row: its edges over all selected occurrences of the pair, from
// the owner (local node q, member m) on
__device__ __forceinline__ int row_len(const StepView& v, int32_t q, int32_t m) {
  int len = v.mem_rp[m + 1] - v.mem_rp[m];
  for (q = v.next_q[q]; q >= 0; q = v.next_q[q]) {
    m = v.node_mem[q];
    len += v.mem_rp[m + 1] - v.mem_rp[m];
  }
  return len;
}

__device__ __forceinline__ int slice_steps(int len) { return ((int)__reduce_max_sync(0xffffffffu, len) + 3) & ~3; }

// Writes the entries (sqrt w, column) of a slice of 32 rows held by a full warp
// (lane = row of `len` entries, 0 where there is none), its first ss steps to
// shared memory and the others to a range taken from the pool.  A row's entries
// run over its occurrences in block order, then in observation order.
template <int kFill>
__device__ __forceinline__ Slice fill_slice(const StepView& v, int lane, int len, int steps, int row, int32_t q,
                                            int32_t m, EntrySmem es, int sb, int ss) {
  const unsigned lt = (1u << lane) - 1u;
  int32_t e = 0, e1 = 0, pm0 = 0;
  if (len > 0) {
    e = v.mem_rp[m];
    e1 = v.mem_rp[m + 1];
    pm0 = m - v.node_ppos[q];
  }
  Slice s{sb, ss, 0, len, steps};
  const int rest = __reduce_add_sync(0xffffffffu, len > ss ? len - ss : 0);
  const bool padded = pool_padded(steps - ss, rest);
  if (steps > ss) {
    int g = 0;
    if (lane == 0) g = atomicAdd(&v.wfast[kWEntries], pool_grains(steps - ss, rest));
    g = __shfl_sync(0xffffffffu, g, 0);
    s.gb = padded ? g : ~g;
  }
  float2* const ent = v.ent + pool_first(s.gb);
  int at = 0;                            // entries written, not padded
  // kFill entries at a time: three dependent trips to L2 each (8 instead of 4 saves a
  // tenth of a component's time); steps is a multiple of 4
  for (int j = 0; j < steps; j += kFill) {
    int32_t pos[kFill], ei[kFill], pm[kFill];
#pragma unroll
    for (int i = 0; i < kFill; ++i) {
      if (j + i < ss) {
        pos[i] = sb + 32 * (j + i) + lane;
      } else if (padded) {
        pos[i] = 32 * (j - ss + i) + lane;
      } else {
        const unsigned mask = __ballot_sync(0xffffffffu, j + i < len);
        pos[i] = at + __popc(mask & lt);
        at += __popc(mask);
      }
      ei[i] = 0;
      pm[i] = 0;
      if (j + i < len) {
        while (e == e1) {              // the next selected occurrence
          q = v.next_q[q];
          m = v.node_mem[q];
          e = v.mem_rp[m];
          e1 = v.mem_rp[m + 1];
          pm0 = m - v.node_ppos[q];
        }
        ei[i] = e++;
        pm[i] = pm0;
      }
    }
    float sw[kFill];
    int32_t col[kFill];
#pragma unroll
    for (int i = 0; i < kFill; ++i) {
      sw[i] = 0.f;
      col[i] = -1;
      if (j + i < len) {
        sw[i] = v.edge_sw[ei[i]];
        col[i] = pm[i] + v.edge_pos[ei[i]];
      }
    }
#pragma unroll
    for (int i = 0; i < kFill; ++i) col[i] = col[i] >= 0 ? v.mrow[col[i]] : row;
#pragma unroll
    for (int i = 0; i < kFill; ++i) {
      if (j + i >= steps) break;
      if (j + i < ss) {
        es.sw[pos[i]] = sw[i];
        es.col[pos[i]] = (uint16_t)col[i];
      } else if (padded || j + i < len) {
        ent[pos[i]] = make_float2(sw[i], __int_as_float(col[i]));
      }
    }
  }
  return s;
}

// The first K steps of a slice in registers: weights w = sw^2, columns in pairs.
template <int K>
struct Held {
  float w[K > 0 ? K : 1];
  uint32_t c[K > 0 ? K / 2 : 1];
};

template <int K>
__device__ __forceinline__ void hold(Held<K>& h, EntrySmem es, const Slice& sl, int lane) {
  const float* ws = es.sw + sl.sb + lane;
  const uint16_t* cs = es.col + sl.sb + lane;
#pragma unroll
  for (int j = 0; j < K; j += 2) {
    const bool in = j < sl.ss;
    const float a = in ? ws[32 * j] : 0.f, b = in ? ws[32 * j + 32] : 0.f;
    h.w[j] = a * a;
    h.w[j + 1] = b * b;
    h.c[j / 2] = in ? (uint32_t)cs[32 * j] | ((uint32_t)cs[32 * j + 32] << 16) : 0u;
  }
}

// sum over the row's entries of w (y_row - y_col), w = sw^2
template <int K>
__device__ __forceinline__ float slice_mul(const float2* ent, EntrySmem es, const Slice& sl, const Held<K>& h, int lane,
                                           float yr, const float* y) {
  float s = 0.f;
#pragma unroll
  for (int j = 0; j < K; j += 4) {
    if (j < sl.ss) {
      float t[4];
#pragma unroll
      for (int i = 0; i < 4; i += 2) {
        t[i] = y[h.c[(j + i) / 2] & 0xFFFFu];
        t[i + 1] = y[h.c[(j + i) / 2] >> 16];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) s = fmaf(h.w[j + i], yr - t[i], s);
    }
  }
  if (sl.steps <= K && sl.ss == sl.steps) return s;
  {
    const float* ws = es.sw + sl.sb + lane + 32 * K;
    const uint16_t* cs = es.col + sl.sb + lane + 32 * K;
#pragma unroll 2
    for (int j = K; j < sl.ss; j += 4, ws += 4 * 32, cs += 4 * 32) {
      float w[4];
      int c[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        w[i] = ws[32 * i];
        c[i] = cs[32 * i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) s = fmaf(w[i] * w[i], yr - y[c[i]], s);
    }
  }
  if (sl.steps == sl.ss) return s;
  ent += pool_first(sl.gb);
  if (sl.gb >= 0) {
    const float2* p = ent + lane;
    for (int j = sl.ss; j < sl.steps; j += 8, p += 8 * 32) {
      float2 x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = j + i < sl.steps ? p[32 * i] : make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 8; ++i) s = fmaf(x[i].x * x[i].x, yr - y[__float_as_int(x[i].y)], s);
    }
    return s;
  }
  const unsigned lt = (1u << lane) - 1u;
  int at = 0;
  for (int j = sl.ss; j < sl.steps; j += 4) {
    float2 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned mask = __ballot_sync(0xffffffffu, j + i < sl.len);
      if (j + i < sl.len) x[i] = ent[at + __popc(mask & lt)];
      at += __popc(mask);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (j + i < sl.len) s = fmaf(x[i].x * x[i].x, yr - y[__float_as_int(x[i].y)], s);
  }
  return s;
}

// the same in double-float; even and odd steps in two sums, so that one chain of
// additions does not bound it
__device__ __forceinline__ df32 slice_mul_df(const float2* ent, EntrySmem es, const Slice& sl, int lane, df32 zr,
                                             const float* zh, const float* zl) {
  df32 acc[2] = {{0.f, 0.f}, {0.f, 0.f}};
  auto term = [&](float w, int c) {
    return df_mul(df_two_prod(w, w), df_add(zr, df32{-zh[c], -zl[c]}));
  };
  const float* ws = es.sw + sl.sb + lane;
  const uint16_t* cs = es.col + sl.sb + lane;
  for (int j = 0; j < sl.ss; j += 4, ws += 4 * 32, cs += 4 * 32) {
    df32 t[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) t[i] = term(ws[32 * i], cs[32 * i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i & 1] = df_add(acc[i & 1], t[i]);
  }
  if (sl.steps == sl.ss) return df_add(acc[0], acc[1]);
  const unsigned lt = (1u << lane) - 1u;
  ent += pool_first(sl.gb);
  int at = sl.gb >= 0 ? lane : 0;
  for (int j = sl.ss; j < sl.steps; j += 4) {
    float2 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int k = at;
      if (sl.gb >= 0) {
        at += 32;
      } else {
        const unsigned mask = __ballot_sync(0xffffffffu, j + i < sl.len);
        k = at + __popc(mask & lt);
        at += __popc(mask);
      }
      x[i] = make_float2(0.f, 0.f);
      if (j + i < sl.len) x[i] = ent[k];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (j + i < sl.len) acc[i & 1] = df_add(acc[i & 1], term(x[i].x, __float_as_int(x[i].y)));
  }
  return df_add(acc[0], acc[1]);
}

// Power of two that a component's right-hand side is multiplied by (in place: k_resid
// writes it anew every step) and its solution divided by, from bb = |u|^2: one unless
// bb lies far out.  alpha and beta come from an
// approximate division, good to 2 ulp for divisors in [2^-126, 2^126] and zero above: a
// component of residuals near 1e18 never left z = 0.  (Its last bits steer the iteration
// only, the residual is replaced in double-float: gradients are 1.4e-7 and 2.0e-7 from
// 64 bits and chains 4.1e-11, 2.3e-11 and 9.5e-12, with IEEE quotients just as far, and
// one chain 1.4e-11, with them 2.1e-11; chains and batches would take 1 to 2 % longer,
// and as much with a test of every divisor.)
__device__ __forceinline__ float rhs_scale(float bb) {
  if (bb >= 0x1p-60f && bb <= 0x1p60f) return 1.f;
  const int e = (int)(__float_as_uint(bb) >> 23 & 255u) - 127;
  if (e == 128) return 0x1p-100f;                               // the squares do not fit FP32
  return __uint_as_float((uint32_t)(127 - (e >> 1)) << 23);     // bb scale^2 in [1, 4)
}

// u - lambda z - B^T B z of one row, rounded to FP32
__device__ __forceinline__ float row_residual(const StepView& v, int32_t u, df32 z, df32 bz) {
  df32 rd = df_add(df32{v.rhs[u], v.rhs_lo[u]}, df_mul_f(z, -v.lam));
  rd = df_add(rd, df32{-bz.hi, -bz.lo});
  return rd.hi;
}

__device__ __forceinline__ float2 warp_sum2(float a, float b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  return make_float2(a, b);
}

// ------------------------------------------------------------------ one warp or one CTA
template <int NW>
__device__ __forceinline__ void group_sync() {
  if constexpr (NW == 1) __syncwarp(); else __syncthreads();
}

// Two sums over the group (fixed order), one barrier: warp sums go to one of two
// alternating buffers and every warp adds them up.
template <int NW>
__device__ __forceinline__ float2 group_sum2(float a, float b, float2* part, int& par, int w, int lane) {
  float2 s = warp_sum2(a, b);
  if constexpr (NW == 1) {
    __syncwarp();
    return s;
  } else {
    if (lane == 0) part[par * NW + w] = s;
    __syncthreads();
    // every lane adds eight warps' sums (four at 32 warps, where the reads would
    // take longer than the shuffles), the rest by shuffles
    constexpr int E = NW > 16 ? 4 : 8;
    const float4* q = reinterpret_cast<const float4*>(part + par * NW + (lane & (NW / E - 1)) * E);
    float4 x[E / 2];
#pragma unroll
    for (int i = 0; i < E / 2; ++i) x[i] = q[i];
#pragma unroll
    for (int h = E / 4; h > 0; h >>= 1)
#pragma unroll
      for (int i = 0; i < h; ++i) {
        x[i].x += x[i + h].x;
        x[i].y += x[i + h].y;
        x[i].z += x[i + h].z;
        x[i].w += x[i + h].w;
      }
    s = make_float2(x[0].x + x[0].z, x[0].y + x[0].w);
    par ^= 1;
#pragma unroll
    for (int o = NW / E / 2; o > 0; o >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    return s;
  }
}

// NW warps per component, RPT rows per lane, GROUPS components per CTA, KP
// pieces at most.  Vectors stay in registers but for y and z, which the
// neighbours read from shared memory.
constexpr int kLenBins = 64;

template <int NW, int RPT, int GROUPS, int KP>
struct SolveSmem {
  static constexpr int R = NW * RPT * 32;
  union {
    struct {
      int32_t u[R], m[R], q[R], len[R];     // set-up: unique pair, member, local node, entries
    } row;
    struct {
      float y[R], zh[R], zl[R];
    } vec;
  };
  union {
    struct {
      int32_t pid[KP], pblk[KP], prow[KP], pbase[KP];
    };
    int32_t bin[kLenBins * NW * RPT];       // rows per length and slice
  };
  alignas(16) float2 part[2 * NW];
  int32_t wsum[NW], ssize[NW * RPT];
  int32_t unit;
  float scale;
};

// Exclusive scan of a[0, N) over the group, N / (32 NW) consecutive values per
// thread; ends with the group synchronised.
template <int NW, int N>
__device__ void group_exscan(int32_t* a, int32_t* wsum, int tid, int w, int lane) {
  constexpr int E = N / (32 * NW);
  static_assert(E * 32 * NW == N, "scan shape");
  int x[E], t = 0;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    x[i] = a[tid * E + i];
    t += x[i];
  }
  int s = t;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s += y;
  }
  int before = 0;
  if constexpr (NW > 1) {
    if (lane == 31) wsum[w] = s;
    __syncthreads();
    for (int i = 0; i < w; ++i) before += wsum[i];
  }
  before += s - t;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    a[tid * E + i] = before;
    before += x[i];
  }
  group_sync<NW>();
}

// ENT: matrix entries per component in shared memory (6 bytes each, longest
// slices first).  Through L1 they were evicted by the clean pieces' solver, which
// streams its inverses on the same SMs: 770 cycles per four steps instead of ~100.
// HELD: steps of each slice held in registers besides.  An iteration is bound by
// shared-memory wavefronts, one for the weights, one for the columns and about
// three for the gathered neighbours of a step; those held need the last only.
// With the sums' shorter chain and without IEEE divisions, 170 rows take 75 us instead
// of 104.  24 steps need 127 registers, half the CTAs an SM could hold: no loss for 8
// and 16 warps, where one SM's shared memory is the limit (4 steps and 64 registers for
// 16 warps: 1607 -> 1680 us on the dense 4,000-event chain), but 32 warps keep to 64
// registers (8 steps spill: 213 -> 230 us), and the one-warp class lives on many warps
// (12 steps, 167 registers: batches 3 % slower).
// CTAS: resident CTAs per SM that the register count is held to.
template <int NW, int RPT, int GROUPS, int KP, int ENT, int HELD, int CTAS>
__global__ void __launch_bounds__(NW * 32 * GROUPS, CTAS) k_solve(StepView v, int cls, int max_it, float tol) {
  static_assert(NW == 1 || GROUPS == 1, "a CTA holds one component, or one per warp");
  static_assert(ENT % 128 == 0, "whole groups of four steps");
  using Smem = SolveSmem<NW, RPT, GROUPS, KP>;
  __shared__ Smem smem[GROUPS];
  extern __shared__ __align__(16) uint8_t s_ent[];
  if (aborted_cta(v)) return;
  Smem& S = smem[threadIdx.x / (NW * 32)];
  EntrySmem es;
  es.sw = reinterpret_cast<float*>(s_ent) + (threadIdx.x / (NW * 32)) * ENT;
  es.col = reinterpret_cast<uint16_t*>(s_ent + (size_t)GROUPS * ENT * 4) + (threadIdx.x / (NW * 32)) * ENT;
  const int tid = threadIdx.x % (NW * 32), w = tid >> 5, lane = tid & 31;
  constexpr int NT = NW * 32;
  const unsigned lt = (1u << lane) - 1u;
  const float lam = v.lam;
  const int32_t count = v.wfast[kWClass0 + cls];
  const int32_t* list = v.cls_list + (int64_t)cls * v.cls_cap;
  int most = 0;
  for (;;) {
    group_sync<NW>();
    if (tid == 0) S.unit = atomicAdd(&v.wfast[kWCursor0 + cls], 1);
    group_sync<NW>();
    if (S.unit >= count) break;
    const int32_t unit = list[S.unit];
    const int32_t off = v.unit_off[unit];
    const int np = v.unit_np[unit], rows = v.unit_rows[unit];
    for (int i = tid; i < np; i += NT) {
      S.pid[i] = v.unit_pieces[off + i];
      S.pblk[i] = v.unit_pblk[off + i];
      S.prow[i] = v.unit_prow[off + i];
    }
    group_sync<NW>();
    // first row of each piece: the rows of the pieces with smaller ids
    for (int i = tid; i < np; i += NT) {
      int b = 0;
      const int32_t id = S.pid[i];
      for (int j = 0; j < np; ++j) b += S.pid[j] < id ? S.prow[j] : 0;
      S.pbase[i] = b;
    }
    group_sync<NW>();
    // rows: owner occurrences, member order
    for (int i = w; i < np; i += NW) {
      const int32_t g = S.pid[i];
      const int32_t q0 = v.blk_node_off[S.pblk[i]], pm0 = v.piece_node_off[g], pm1 = v.piece_node_off[g + 1];
      int row0 = S.pbase[i];
      for (int32_t c = pm0; c < pm1; c += 32) {
        const int32_t m = c + lane;
        int32_t q = -1;
        if (m < pm1) q = q0 + v.piece_nodes[m];
        const bool own = m < pm1 && v.owner_q[q] == q;
        const unsigned mask = __ballot_sync(0xffffffffu, own);
        if (own) {
          const int row = row0 + __popc(mask & lt);
          const int32_t u = v.loc2u[q];
          S.row.u[row] = u;
          S.row.m[row] = m;
          S.row.q[row] = q;
        }
        row0 += __popc(mask);
      }
    }
    group_sync<NW>();
    // rows by decreasing length (stable), so that a slice's rows take similar
    // numbers of steps: the lengths of a minibatch run from 1 to 24 around a mean
    // of 6, and in member order every slice ran to its longest
    {
      int32_t u[RPT], m[RPT], q[RPT];
      int len[RPT], bin[RPT], rank[RPT];
      for (int i = tid; i < kLenBins * NW * RPT; i += NT) S.bin[i] = 0;
      group_sync<NW>();
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        const int sl = w + NW * k, row = sl * 32 + lane;
        len[k] = 0;
        if (row < rows) {
          u[k] = S.row.u[row];
          m[k] = S.row.m[row];
          q[k] = S.row.q[row];
          len[k] = row_len(v, q[k], m[k]);
        }
        bin[k] = row < rows ? kLenBins - 1 - (len[k] < kLenBins ? len[k] : kLenBins - 1) : -1;
        const unsigned same = __match_any_sync(0xffffffffu, bin[k]);
        rank[k] = __popc(same & lt);
        if (row < rows && rank[k] == 0) S.bin[bin[k] * (NW * RPT) + sl] = __popc(same);
      }
      group_sync<NW>();
      group_exscan<NW, kLenBins * NW * RPT>(S.bin, S.wsum, tid, w, lane);
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        const int sl = w + NW * k;
        if (sl * 32 + lane >= rows) continue;
        const int row = S.bin[bin[k] * (NW * RPT) + sl] + rank[k];
        S.row.u[row] = u[k];
        S.row.m[row] = m[k];
        S.row.q[row] = q[k];
        S.row.len[row] = len[k];
        v.rowof[u[k]] = row;
        v.mrow[m[k]] = row;
      }
    }
    group_sync<NW>();
    if (np > 1) {
      for (int i = w; i < np; i += NW) {
        const int32_t g = v.unit_pieces[off + i];
        const int32_t q0 = v.blk_node_off[v.unit_pblk[off + i]], pm1 = v.piece_node_off[g + 1];
        for (int32_t m = v.piece_node_off[g] + lane; m < pm1; m += 32) {
          const int32_t q = q0 + v.piece_nodes[m];
          if (v.owner_q[q] != q) v.mrow[m] = v.rowof[v.loc2u[q]];
        }
      }
      group_sync<NW>();
    }
    // entries and vectors: rows of slices w, w + NW, ...
    Slice sl[RPT];
    int32_t u[RPT];
    float r[RPT], yv[RPT], p[RPT], ap[RPT], dz[RPT], di[RPT];
    bool on[RPT];
    float bb = 0.f, rz = 0.f, rr = 0.f;
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const int row = (w + NW * k) * 32 + lane;
      on[k] = row < rows;
      sl[k] = Slice{0, 0, 0, on[k] ? S.row.len[row] : 0, 0};
      sl[k].steps = slice_steps(sl[k].len);
      // what it takes of shared memory, all of it at most (no sum overflows then)
      if (lane == 0) S.ssize[w + NW * k] = 32 * (sl[k].steps < ENT / 32 ? sl[k].steps : ENT / 32);
    }
    group_sync<NW>();
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const int row = (w + NW * k) * 32 + lane;
      u[k] = on[k] ? S.row.u[row] : 0;
      int sb = 0;
      for (int i = 0; i < w + NW * k; ++i) sb += S.ssize[i];
      int ss = sb < ENT ? ((ENT - sb) >> 5) & ~3 : 0;
      ss = ss < sl[k].steps ? ss : sl[k].steps;
      sl[k] = fill_slice<(RPT == 1 && NW < 32) ? 8 : 4>(v, lane, sl[k].len, sl[k].steps, row, on[k] ? S.row.q[row] : 0, on[k] ? S.row.m[row] : 0, es,
                         sb, ss);
    }
    group_sync<NW>();
    Held<HELD> held[RPT];
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const int row = (w + NW * k) * 32 + lane;
      hold<HELD>(held[k], es, sl[k], lane);
      r[k] = yv[k] = p[k] = ap[k] = dz[k] = 0.f;
      di[k] = 0.f;
      if (on[k]) {
        const float h = v.rhs[u[k]];
        r[k] = h + v.rhs_lo[u[k]];
        di[k] = 1.f / v.diag[u[k]];
        yv[k] = r[k] * di[k];
        bb = fmaf(h, h, bb);
        rz = fmaf(r[k], yv[k], rz);
        rr = fmaf(r[k], r[k], rr);
      }
      S.vec.y[row] = yv[k];
      S.vec.zh[row] = 0.f;
      S.vec.zl[row] = 0.f;
    }
    int par = 0, it = 0, rounds = 0;
    bb = group_sum2<NW>(bb, 0.f, S.part, par, w, lane).x;
    const float scale = rhs_scale(bb);
    if (tid == 0) S.scale = scale;
    if (scale != 1.f) {
      rz = rr = 0.f;
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        if (on[k]) {
          v.rhs[u[k]] *= scale;
          v.rhs_lo[u[k]] *= scale;
        }
        r[k] *= scale;
        yv[k] = r[k] * di[k];
        S.vec.y[(w + NW * k) * 32 + lane] = yv[k];
        rz = fmaf(r[k], yv[k], rz);
        rr = fmaf(r[k], r[k], rr);
      }
    }
    float2 s = group_sum2<NW>(rz, rr, S.part, par, w, lane);
    if (scale != 1.f) bb = s.y;
    const float thr = kAim * tol * tol * bb;
    float last = s.y, beta = 0.f;
    rz = s.x;
    while (bb > 0.f && it < max_it) {
      // p = y + beta p, A p = A y + beta A p
      float dot = 0.f;
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        const float ay = fmaf(lam, yv[k], slice_mul<HELD>(v.ent, es, sl[k], held[k], lane, yv[k], S.vec.y));
        p[k] = fmaf(beta, p[k], yv[k]);
        ap[k] = fmaf(beta, ap[k], ay);
        dot = fmaf(p[k], ap[k], dot);
      }
      const float pap = group_sum2<NW>(dot, 0.f, S.part, par, w, lane).x;
      if (!(pap > 0.f)) break;
      const float alpha = __fdividef(rz, pap);
      float rzn = 0.f;
      rr = 0.f;
#pragma unroll
      for (int k = 0; k < RPT; ++k) {
        dz[k] = fmaf(alpha, p[k], dz[k]);
        r[k] = fmaf(-alpha, ap[k], r[k]);
        yv[k] = r[k] * di[k];
        S.vec.y[(w + NW * k) * 32 + lane] = yv[k];
        rzn = fmaf(r[k], yv[k], rzn);
        rr = fmaf(r[k], r[k], rr);
      }
      s = group_sum2<NW>(rzn, rr, S.part, par, w, lane);
      ++it;
      if (s.y <= kReplace * last || s.y <= 0.5f * thr) {
        // z += dz; the residual of z in double-float takes the recurrence's place
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          const int row = (w + NW * k) * 32 + lane;
          const df32 zn = df_add_f(df32{S.vec.zh[row], S.vec.zl[row]}, dz[k]);
          S.vec.zh[row] = zn.hi;
          S.vec.zl[row] = zn.lo;
          dz[k] = 0.f;
        }
        group_sync<NW>();
        rzn = rr = 0.f;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
          const int row = (w + NW * k) * 32 + lane;
          const df32 z = {S.vec.zh[row], S.vec.zl[row]};
          const df32 bz = slice_mul_df(v.ent, es, sl[k], lane, z, S.vec.zh, S.vec.zl);
          r[k] = on[k] ? row_residual(v, u[k], z, bz) : 0.f;
          yv[k] = r[k] * di[k];
          S.vec.y[row] = yv[k];
          rzn = fmaf(r[k], yv[k], rzn);
          rr = fmaf(r[k], r[k], rr);
        }
        s = group_sum2<NW>(rzn, rr, S.part, par, w, lane);
        if (s.y <= thr || ++rounds >= kMaxReplace) break;
        last = s.y;
      }
      beta = __fdividef(s.x, rz);
      rz = s.x;
    }
#pragma unroll
    for (int k = 0; k < RPT; ++k)
      if (on[k]) {
        const int row = (w + NW * k) * 32 + lane;
        const df32 zn = df_add_f(df32{S.vec.zh[row], S.vec.zl[row]}, dz[k]);
        v.z[u[k]] = zn.hi;
        v.z_lo[u[k]] = zn.lo;
        if (S.scale != 1.f) {
          v.z[u[k]] /= S.scale;
          v.z_lo[u[k]] /= S.scale;
        }
      }
    if (it > most) most = it;
  }
  if (tid == 0 && most > 0) atomicMax(&v.counters[kCntCompIters], most);
}

// ------------------------------------------------------------------ several CTAs
// shared memory of a CTA of the multi-CTA class: the entries of the first
// kMultiSteps steps of each warp's rows, and the component's y where it fits
// (after a group barrier y comes from L2 once, not gather by gather)
constexpr int kMultiSteps = 32;
constexpr int kMultiY = 4096;
constexpr int kMultiEnt = kMultiSteps * kMultiThreads;
constexpr size_t kMultiBytes = (size_t)kMultiEnt * 6 + (size_t)kMultiY * 4;
// Pieces sorted together, and pieces a CTA of the group takes at most.  Every piece
// compared with every other, on CTAs counted by rows alone, grew with the square of a
// catalog's blocks: 1,200 rows in 96,000 pieces took 140 ms, now 2.16 (1.13 with the
// same observations in blocks of 64).  Runs leave log2(kRun) bisection steps a piece
// and run; where all pieces fit one, the sort costs what the comparisons did (the
// regional gradient takes 2.20 ms with either).
constexpr int kRun = 4096;
static_assert(kRun * sizeof(uint64_t) <= kMultiBytes && kRun % kMultiThreads == 0, "room for a run's keys");

struct MultiSmem {
  float2 part[kMultiThreads / 32];
  float2 sum;
  float scale;
  int32_t unit, size, ok;
  int32_t scan[33];
};

struct Group {
  int32_t seq;                       // position of the component in the list, from 1
  int32_t call;                      // barriers passed in this component
  int rank, size, cta0;
};

// A word is one 128-bit access: the sums must be those of the barrier number read
// with them, and a vector access (.v4.s32) is four accesses in no stated order.
__device__ __forceinline__ int4 ld_slot(const int4* p) {
  uint64_t a, b;
  asm volatile(
      "{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
      : "=l"(a), "=l"(b)
      : "l"(p)
      : "memory");
  return make_int4((int)a, (int)(a >> 32), (int)b, (int)(b >> 32));
}
__device__ __forceinline__ void st_slot(int4* p, int4 r) {
  const uint64_t a = (uint32_t)r.x | (uint64_t)(uint32_t)r.y << 32, b = (uint32_t)r.z | (uint64_t)(uint32_t)r.w << 32;
  asm volatile(
      "{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
      "l"(a), "l"(b)
      : "memory");
}

// Group-wide barrier with two sums (fixed order).  Each CTA publishes its sums
// and the barrier's number in one 16-byte word of its own, and reads the words
// of its group until they carry that number (or a later one, which a CTA that
// has gone on to its next component may show after the last barrier): one trip
// through L2 instead of a counter's three.  Words alternate between two sets; a
// set is overwritten two barriers later, when every CTA of the group has read
// it.  Bounded like grid_barrier; false when the wait gave up.
__device__ bool multi_sum2(const StepView& v, MultiSmem& S, Group& G, float a, float b, float2* out) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int NW = kMultiThreads / 32;
  float2 s = warp_sum2(a, b);
  if (lane == 0) S.part[w] = s;
  ++G.call;
  __syncthreads();
  if (w == 0) {
    s = lane < NW ? S.part[lane] : make_float2(0.f, 0.f);
    s = warp_sum2(s.x, s.y);
    int4* slots = v.msync + (G.call & 1) * kMaxGrid;
    if (lane == 0) {
      fence_gpu();
      st_slot(slots + blockIdx.x, make_int4(__float_as_int(s.x), __float_as_int(s.y), G.seq, G.call));
    }
    float x = 0.f, y = 0.f;
    bool ok = true;
    const uint64_t limit = v.prm->wait_ns;
    uint64_t t0 = 0;
    for (int i = lane; i < G.size && ok; i += 32) {
      for (uint32_t n = 0;; ++n) {
        const int4 r = ld_slot(slots + G.cta0 + i);
        if (r.z > G.seq || (r.z == G.seq && r.w >= G.call)) {
          x += __int_as_float(r.x);
          y += __int_as_float(r.y);
          break;
        }
        // not on the first spins, where it would cost most barriers another trip to L2
        if (limit == 0 || (n & 255u) == 16) {
          const uint64_t t = gtimer();
          if (t0 == 0) t0 = t;
          if (*((const volatile int32_t*)v.counters + kCntError) != 0) ok = false;
          else if (t - t0 >= limit) {
            set_error(v.counters, SPIDER_E_TIMEOUT);
            ok = false;
          }
          if (!ok) break;
        }
      }
    }
    fence_gpu();
    ok = __all_sync(0xffffffffu, ok);
    s = warp_sum2(x, y);
    if (lane == 0) {
      S.sum = s;
      S.ok = ok ? 1 : 0;
    }
  }
  __syncthreads();
  *out = S.sum;
  return S.ok != 0;
}

__device__ bool multi_sync(const StepView& v, MultiSmem& S, Group& G) {
  float2 t;
  return multi_sum2(v, S, G, 0.f, 0.f, &t);
}

// One run of a component's piece list, n <= kRun pieces: sorted by id in place, with
// the rows before each piece of the run in pbase.  key: kRun words of shared
// memory.  Kept out of line: its registers would spill the iteration's.
__device__ __noinline__ void sort_run(int32_t* pieces, int32_t* pblk, int32_t* prow, int32_t* pbase, int32_t* scan,
                                      uint64_t* key, int n) {
  const int tid = threadIdx.x;
  int n2 = 2;
  while (n2 < n) n2 <<= 1;
  for (int i = tid; i < n2; i += kMultiThreads)
    key[i] = i < n ? (uint64_t)pieces[i] << 32 | (uint32_t)i : ~0ull;
  __syncthreads();
  for (int k = 2; k <= n2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int h = tid; h < n2 / 2; h += kMultiThreads) {
        const int i = ((h & ~(j - 1)) << 1) | (h & (j - 1)), l = i | j;
        const uint64_t p = key[i], q = key[l];
        if ((p > q) == ((i & k) == 0)) {
          key[i] = q;
          key[l] = p;
        }
      }
      __syncthreads();
    }
  constexpr int E = kRun / kMultiThreads;
  int32_t blk[E], rows[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = e * kMultiThreads + tid;
    const int from = i < n ? (int)(uint32_t)key[i] : 0;
    blk[e] = i < n ? pblk[from] : 0;
    rows[e] = i < n ? prow[from] : 0;
  }
  __syncthreads();
  int before = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int i = e * kMultiThreads + tid;
    if (e * kMultiThreads >= n) break;
    int total;
    const int pre = block_exscan(rows[e], scan, &total);
    if (i < n) {
      pieces[i] = (int32_t)(key[i] >> 32);
      pblk[i] = blk[e];
      prow[i] = rows[e];
      pbase[i] = before + pre;
    }
    before += total;
  }
  __syncthreads();
}

// First rows of the pieces k0, k0 + step, ... of a list in sorted runs: the rows
// before a piece in its own run, and from every other run's by bisection.
__device__ __noinline__ void rows_before(const int32_t* pieces, const int32_t* prow, const int32_t* pbase,
                                         int32_t* first, int np, int k0, int step) {
  for (int k = k0; k < np; k += step) {
    const int32_t id = pieces[k];
    int b = pbase[k];
    for (int c = 0; c < np; c += kRun) {
      if (k / kRun == c / kRun) continue;
      int lo = c, hi = np - c < kRun ? np : c + kRun;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (pieces[mid] < id) lo = mid + 1; else hi = mid;
      }
      if (lo > c) b += pbase[lo - 1] + prow[lo - 1];
    }
    first[k] = b;
  }
}

// Components beyond one CTA: a cooperative launch whose CTAs form groups of
// consecutive CTAs, one group per component, sized so that all components run
// at once where they fit (rows per thread grow with the total) and batch after
// batch otherwise.  Every CTA walks the same assignment, so a group's CTAs meet
// in the same order.  Vectors live in memory by row slot (each thread reads
// back its own rows; y and z are read by the group).  What bounds an iteration
// is its two group barriers and the latency of the gathers, ~4 us against the
// ~50 us of one grid-wide iteration over all components.
__global__ void __launch_bounds__(kMultiThreads, 2) k_solve_multi(StepView v, int max_it, float tol) {
  __shared__ MultiSmem S;
  extern __shared__ __align__(16) uint8_t s_dyn[];
  if (aborted_cta(v)) return;
  EntrySmem es;
  es.sw = reinterpret_cast<float*>(s_dyn);
  float* const ys = es.sw + kMultiEnt;
  es.col = reinterpret_cast<uint16_t*>(ys + kMultiY);
  const int32_t nbig = v.wfast[kWClass0 + kClsMulti];
  if (nbig == 0) return;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  constexpr int NW = kMultiThreads / 32;
  const unsigned lt = (1u << lane) - 1u;
  const float lam = v.lam;
  const int32_t* list = v.cls_list + (int64_t)kClsMulti * v.cls_cap;
  // rows per CTA: the total over the grid, in whole rounds of one row per thread
  const int64_t all = v.wfast[kWRowSlots];
  const int64_t per_cta = kMultiThreads * ((all + (int64_t)gridDim.x * kMultiThreads - 1) /
                                           ((int64_t)gridDim.x * kMultiThreads));
  int pos = 0, most = 0;
  for (int32_t i = 0; i < nbig; ++i) {
    __syncthreads();
    if (tid == 0) {
      const int32_t u = list[i];
      int64_t size = ((int64_t)v.unit_rows[u] + per_cta - 1) / per_cta;
      const int runs = (v.unit_np[u] + kRun - 1) / kRun;      // a run of pieces per CTA, too
      size = size < runs ? runs : size;
      S.unit = u;
      S.size = size < 1 ? 1 : (size > gridDim.x ? (int)gridDim.x : (int)size);
    }
    __syncthreads();
    if (pos + S.size > (int)gridDim.x) pos = 0;
    const int cta0 = pos;
    pos += S.size;
    if ((int)blockIdx.x < cta0 || (int)blockIdx.x >= cta0 + S.size) continue;
    const int32_t unit = S.unit;
    Group G;
    G.seq = i + 1;
    G.call = 0;
    G.rank = blockIdx.x - cta0;
    G.size = S.size;
    G.cta0 = cta0;
    const int32_t off = v.unit_off[unit], slot0 = v.unit_slot[unit];
    const int np = v.unit_np[unit], rows = v.unit_rows[unit];
    const int gw = G.rank * NW + w, ngw = G.size * NW;
    const int nsl = (rows + 31) >> 5;
    // first row of each piece: the rows of the pieces with smaller ids
    for (int c = G.rank * kRun; c < np; c += G.size * kRun)
      sort_run(v.unit_pieces + off + c, v.unit_pblk + off + c, v.unit_prow + off + c, v.unit_pbase + off + c, S.scan,
               reinterpret_cast<uint64_t*>(s_dyn), np - c < kRun ? np - c : kRun);
    if (!multi_sync(v, S, G)) return;
    if (np > kRun) {
      rows_before(v.unit_pieces + off, v.unit_prow + off, v.unit_pbase + off, v.unit_first + off, np,
                  G.rank * kMultiThreads + tid, G.size * kMultiThreads);
      if (!multi_sync(v, S, G)) return;
    }
    // rows of the owner occurrences
    for (int k = gw; k < np; k += ngw) {
      const int32_t g = v.unit_pieces[off + k];
      const int32_t q0 = v.blk_node_off[v.unit_pblk[off + k]], pm0 = v.piece_node_off[g], pm1 = v.piece_node_off[g + 1];
      int row0 = (np > kRun ? v.unit_first : v.unit_pbase)[off + k];
      for (int32_t c = pm0; c < pm1; c += 32) {
        const int32_t m = c + lane;
        int32_t q = -1;
        if (m < pm1) q = q0 + v.piece_nodes[m];
        const bool own = m < pm1 && v.owner_q[q] == q;
        const unsigned mask = __ballot_sync(0xffffffffu, own);
        if (own) {
          const int row = row0 + __popc(mask & lt);
          const int32_t u = v.loc2u[q];
          v.rs_u[slot0 + row] = u;
          v.rs_m[slot0 + row] = m;
          v.rs_q[slot0 + row] = q;
          v.rowof[u] = row;
          v.mrow[m] = row;
        }
        row0 += __popc(mask);
      }
    }
    if (!multi_sync(v, S, G)) return;
    for (int k = gw; k < np; k += ngw) {
      const int32_t g = v.unit_pieces[off + k];
      const int32_t q0 = v.blk_node_off[v.unit_pblk[off + k]], pm1 = v.piece_node_off[g + 1];
      for (int32_t m = v.piece_node_off[g] + lane; m < pm1; m += 32) {
        const int32_t q = q0 + v.piece_nodes[m];
        if (v.owner_q[q] != q) v.mrow[m] = v.rowof[v.loc2u[q]];
      }
    }
    if (!multi_sync(v, S, G)) return;
    float* const y = v.rs_y + slot0;
    float* const zh = v.rs_zh + slot0;
    float* const zl = v.rs_zl + slot0;
    const bool y_smem = rows <= kMultiY;
    int used = 0;                        // steps of this warp's shared memory taken
    float bb = 0.f, rz = 0.f, rr = 0.f;
    for (int sl = gw; sl < nsl; sl += ngw) {
      const int row = sl * 32 + lane, t = slot0 + row;
      const bool on = row < rows;
      const int32_t u = on ? v.rs_u[t] : 0;
      const int32_t m = on ? v.rs_m[t] : 0;
      const int32_t q = on ? v.rs_q[t] : 0;
      const int len = on ? row_len(v, q, m) : 0;
      const int steps = slice_steps(len);
      int ss = rows <= 65536 ? kMultiSteps - used : 0;
      ss = ss < steps ? ss : steps;
      const Slice e = fill_slice<4>(v, lane, len, steps, row, q, m, es, (w * kMultiSteps + used) * 32, ss);
      used += ss;
      v.rs_len[t] = len;
      if (lane == 0) v.rs_slice[t >> 5] = make_int4(e.sb, e.ss, e.gb, e.steps);
      float r = 0.f, d = 0.f;
      if (on) {
        const float h = v.rhs[u];
        r = h + v.rhs_lo[u];
        d = 1.f / v.diag[u];
        bb = fmaf(h, h, bb);
      }
      const float yy = r * d;
      v.rs_r[t] = r;
      v.rs_di[t] = d;
      v.rs_p[t] = 0.f;
      v.rs_ap[t] = 0.f;
      v.rs_dz[t] = 0.f;
      y[row] = yy;
      zh[row] = 0.f;
      zl[row] = 0.f;
      rz = fmaf(r, yy, rz);
      rr = fmaf(r, r, rr);
    }
    float2 s;
    if (!multi_sum2(v, S, G, bb, 0.f, &s)) return;
    bb = s.x;
    const float scale = rhs_scale(bb);
    if (tid == 0) S.scale = scale;
    if (scale != 1.f) {
      rz = rr = 0.f;
      for (int sl = gw; sl < nsl; sl += ngw) {
        const int row = sl * 32 + lane, t = slot0 + row;
        if (row < rows) {
          v.rhs[v.rs_u[t]] *= scale;
          v.rhs_lo[v.rs_u[t]] *= scale;
        }
        const float r = scale * v.rs_r[t], yy = r * v.rs_di[t];
        v.rs_r[t] = r;
        y[row] = yy;
        rz = fmaf(r, yy, rz);
        rr = fmaf(r, r, rr);
      }
    }
    if (!multi_sum2(v, S, G, rz, rr, &s)) return;
    if (scale != 1.f) bb = s.y;
    const float thr = kAim * tol * tol * bb;
    float last = s.y, beta = 0.f;
    rz = s.x;
    int it = 0, rounds = 0;
    while (bb > 0.f && it < max_it) {
      float dot = 0.f;
      if (y_smem) {
        // slots start on a slice, so y is 128-byte aligned
        for (int k = tid; k < nsl * 8; k += kMultiThreads)
          reinterpret_cast<float4*>(ys)[k] = reinterpret_cast<const float4*>(y)[k];
        __syncthreads();
      }
      const float* yg = y_smem ? ys : y;
      for (int sl = gw; sl < nsl; sl += ngw) {
        const int row = sl * 32 + lane, t = slot0 + row;
        const int4 e = v.rs_slice[t >> 5];
        const float yr = yg[row];
        const float ay = fmaf(lam, yr, slice_mul<0>(v.ent, es, Slice{e.x, e.y, e.z, v.rs_len[t], e.w}, Held<0>{}, lane, yr, yg));
        const float p = fmaf(beta, v.rs_p[t], yr);
        const float ap = fmaf(beta, v.rs_ap[t], ay);
        v.rs_p[t] = p;
        v.rs_ap[t] = ap;
        dot = fmaf(p, ap, dot);
      }
      if (!multi_sum2(v, S, G, dot, 0.f, &s)) return;
      const float pap = s.x;
      if (!(pap > 0.f)) break;
      const float alpha = __fdividef(rz, pap);
      float rzn = 0.f;
      rr = 0.f;
      for (int sl = gw; sl < nsl; sl += ngw) {
        const int row = sl * 32 + lane, t = slot0 + row;
        v.rs_dz[t] = fmaf(alpha, v.rs_p[t], v.rs_dz[t]);
        const float r = fmaf(-alpha, v.rs_ap[t], v.rs_r[t]);
        const float yy = r * v.rs_di[t];
        v.rs_r[t] = r;
        y[row] = yy;
        rzn = fmaf(r, yy, rzn);
        rr = fmaf(r, r, rr);
      }
      if (!multi_sum2(v, S, G, rzn, rr, &s)) return;
      ++it;
      if (s.y <= kReplace * last || s.y <= 0.5f * thr) {
        for (int sl = gw; sl < nsl; sl += ngw) {
          const int row = sl * 32 + lane, t = slot0 + row;
          const df32 zn = df_add_f(df32{zh[row], zl[row]}, v.rs_dz[t]);
          zh[row] = zn.hi;
          zl[row] = zn.lo;
          v.rs_dz[t] = 0.f;
        }
        if (!multi_sync(v, S, G)) return;
        rzn = rr = 0.f;
        for (int sl = gw; sl < nsl; sl += ngw) {
          const int row = sl * 32 + lane, t = slot0 + row;
          const int4 e = v.rs_slice[t >> 5];
          const df32 z = {zh[row], zl[row]};
          const df32 bz = slice_mul_df(v.ent, es, Slice{e.x, e.y, e.z, v.rs_len[t], e.w}, lane, z, zh, zl);
          const float r = row < rows ? row_residual(v, v.rs_u[t], z, bz) : 0.f;
          const float yy = r * v.rs_di[t];
          v.rs_r[t] = r;
          y[row] = yy;
          rzn = fmaf(r, yy, rzn);
          rr = fmaf(r, r, rr);
        }
        if (!multi_sum2(v, S, G, rzn, rr, &s)) return;
        if (s.y <= thr || ++rounds >= kMaxReplace) break;
        last = s.y;
      }
      beta = __fdividef(s.x, rz);
      rz = s.x;
    }
    for (int sl = gw; sl < nsl; sl += ngw) {
      const int row = sl * 32 + lane, t = slot0 + row;
      if (row >= rows) continue;
      const df32 zn = df_add_f(df32{zh[row], zl[row]}, v.rs_dz[t]);
      const int32_t u = v.rs_u[t];
      v.z[u] = zn.hi;
      v.z_lo[u] = zn.lo;
      if (S.scale != 1.f) {
        v.z[u] /= S.scale;
        v.z_lo[u] /= S.scale;
      }
    }
    // every word is read before the CTA's next group overwrites it
    if (!multi_sync(v, S, G)) return;
    if (it > most) most = it;
  }
  if (tid == 0 && most > 0) atomicMax(&v.counters[kCntIters], most);
}

}  // namespace

// warps, rows per lane, components per CTA, pieces, entries in shared memory, steps in registers
#define SOLVE_WARP 1, 2, 4, kWarpPieces, 1024, 0, 7
#define SOLVE_SMALL 8, 1, 1, kSmallPieces, 5120, 24, 2
#define SOLVE_MID 16, 1, 1, kMidPieces, 12288, 24, 1
#define SOLVE_CTA 32, 1, 1, kCtaPieces, 24576, 4, 1

namespace {

template <int NW, int RPT, int GROUPS, int KP, int ENT, int HELD, int CTAS>
cudaError_t configure_one() {
  return cudaFuncSetAttribute(k_solve<NW, RPT, GROUPS, KP, ENT, HELD, CTAS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              GROUPS * ENT * 6);
}

template <int NW, int RPT, int GROUPS, int KP, int ENT, int HELD, int CTAS>
cudaError_t launch_one(const StepView& v, int cls, int max_it, float tol, int ctas, cudaStream_t st) {
  k_solve<NW, RPT, GROUPS, KP, ENT, HELD, CTAS><<<ctas, NW * 32 * GROUPS, GROUPS * ENT * 6, st>>>(v, cls, max_it, tol);
  return cudaGetLastError();
}

}  // namespace

cudaError_t configure_solve_kernels() {
  cudaError_t e;
  if ((e = configure_one<SOLVE_WARP>())) return e;
  if ((e = configure_one<SOLVE_SMALL>())) return e;
  if ((e = configure_one<SOLVE_MID>())) return e;
  if ((e = configure_one<SOLVE_CTA>())) return e;
  return cudaFuncSetAttribute(k_solve_multi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMultiBytes);
}

int solve_multi_grid(int num_sms) {
  int a = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_solve_multi, kMultiThreads, kMultiBytes) != cudaSuccess ||
      a < 1)
    return 0;
  const int g = num_sms * (a < 2 ? a : 2);
  return g > kMaxGrid ? kMaxGrid : g;
}

// ctas: persistent CTAs of 1024 threads; the smaller classes take more of them
cudaError_t launch_solve_class(const StepView& v, int cls, int max_it, float tol, int ctas, cudaStream_t st) {
  switch (cls) {
    case kClsWarp: return launch_one<SOLVE_WARP>(v, cls, max_it, tol, 4 * ctas, st);
    case kClsSmall: return launch_one<SOLVE_SMALL>(v, cls, max_it, tol, 4 * ctas, st);
    case kClsMid: return launch_one<SOLVE_MID>(v, cls, max_it, tol, 2 * ctas, st);
    default: return launch_one<SOLVE_CTA>(v, cls, max_it, tol, ctas, st);
  }
}

cudaError_t launch_solve_multi(const StepView& v, int max_it, float tol, int grid, cudaStream_t st) {
  StepView vv = v;
  int mi = max_it;
  float tl = tol;
  void* args[] = {&vv, &mi, &tl};
  return cudaLaunchCooperativeKernel((const void*)k_solve_multi, dim3(grid), dim3(kMultiThreads), args, kMultiBytes,
                                     st);
}

}  // namespace spider
