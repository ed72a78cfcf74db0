// Step kernels: minibatch selection, the minibatch pair table, residuals, the
// deterministic scatter of dlogp/dT onto pairs and events, and the fused prior +
// SGLD update (the whitening between them is in k_whiten.cu and k_solve.cu).
//
// Determinism: every reduction runs in a fixed order (per-node half-edge lists
// in observation order, per-pair occurrence lists in block order, per-CTA
// partials summed by index); no floating-point atomics anywhere.
#include <cuda_runtime.h>

#include "dfloat.cuh"
#include "kernels.h"
#include "philox.cuh"
#include "spider.h"
#include "step_util.cuh"

namespace spider {

namespace {

constexpr int kThreads = 256;

// Sum over the selected occurrences of a pair of vals[q], from its owner on (block order).
__device__ __forceinline__ float merge_occ(const StepView& v, int32_t q, const float* vals) {
  float a = 0.f;
  for (; q >= 0; q = v.next_q[q]) a += vals[q];
  return a;
}

// ------------------------------------------------------------------ selection
__global__ void k_select(StepView v, int64_t n_b) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n_b) return;
  const StepParams& pr = *v.prm;
  const int32_t* so = pr.full ? v.sub_sel_full : v.sub_sel_mb;
  int lo = 0, hi = v.n_sub;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (so[mid] <= t) lo = mid; else hi = mid;
  }
  const int s = lo;
  const int64_t i = t - so[s];
  const int64_t nbs = v.sub_blk_off[s + 1] - v.sub_blk_off[s];
  // each sub-problem draws its blocks with its own key
  const uint64_t key = pr.seed ^ (0x9E3779B97F4A7C15ull * (uint64_t)s);
  int64_t b = pr.full ? i : feistel_index(i, nbs, key);
  if (b < 0 || b >= nbs) {
    set_error(v.counters, SPIDER_E_TIMEOUT);
    b = i % nbs;
  }
  b += v.sub_blk_off[s];
  v.sel[t] = (int32_t)b;
  v.blk_stamp[b] = pr.tag;
  const int sz = v.blk_e0[b + 1] - v.blk_e0[b];
  atomicAdd(&v.counters[kCntObs], sz);
  atomicAdd(&v.sub_nsel[s], sz);
}

// owner of each local node = its occurrence in the selected block of lowest id
__global__ void k_owner(StepView v) {
  const int tag = v.prm->tag;
  __shared__ int sm[33];
  const int s = blockIdx.x;
  const int32_t b = v.sel[s];
  const int32_t q0 = v.blk_node_off[b], q1 = v.blk_node_off[b + 1];
  int cnt = 0;
  for (int32_t q = q0 + threadIdx.x; q < q1; q += blockDim.x) {
    const int32_t p = v.node_pair[q];
    int32_t qo = -1, bo = -1, next = -1;
    int c = 0;
    // four incidences at a time: their loads go out together
    for (int32_t t = v.inc_off[p], t1 = v.inc_off[p + 1]; t < t1; t += 4) {
      int32_t bb[4], qq[4];
      bool sel[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        bb[i] = t + i < t1 ? v.inc_b[t + i] : -1;
        qq[i] = t + i < t1 ? v.inc_q[t + i] : -1;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) sel[i] = bb[i] >= 0 && v.blk_stamp[bb[i]] == tag;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (sel[i]) {
          if (qo < 0) {
            qo = qq[i];
            bo = bb[i];
          }
          if (next < 0 && qq[i] > q) next = qq[i];      // occurrences ascend with the blocks
          ++c;
        }
    }
    v.owner_q[q] = qo;
    v.next_q[q] = next;
    if (v.owner_b) v.owner_b[q] = bo;
    v.multi[q] = (uint8_t)(c > 1);
    cnt += (qo == q);
  }
  int tot = block_sum<int>(cnt, sm);
  if (threadIdx.x == 0) v.blk_owner_cnt[s] = tot;
}

__global__ void k_scan_owner(StepView v, int64_t n_b) {
  __shared__ int sm[33];
  int carry = 0;
  for (int64_t c = 0; c < n_b; c += blockDim.x) {
    int64_t s = c + threadIdx.x;
    int val = s < n_b ? v.blk_owner_cnt[s] : 0;
    int total;
    int pre = block_exscan(val, sm, &total);
    if (s < n_b) v.blk_owner_off[s] = carry + pre;
    carry += total;
  }
  if (threadIdx.x == 0) v.counters[kCntPairs] = carry;
}

__global__ void k_assign(StepView v) {
  __shared__ int sm[33];
  const int s = blockIdx.x;
  const int32_t b = v.sel[s];
  const int32_t q0 = v.blk_node_off[b], q1 = v.blk_node_off[b + 1];
  int carry = v.blk_owner_off[s];
  for (int32_t c = q0; c < q1; c += blockDim.x) {
    int32_t q = c + threadIdx.x;
    int own = (q < q1) && (v.owner_q[q] == q);
    int total;
    int pre = block_exscan(own, sm, &total);
    if (own) {
      int u = carry + pre;
      v.loc2u[q] = u;
      v.uniq_pair[u] = v.node_pair[q];
      v.uniq_q[u] = q;
      v.umulti[u] = v.multi[q];
    }
    carry += total;
  }
}

__global__ void k_link(StepView v) {
  const int32_t b = v.sel[blockIdx.x];
  const int32_t q0 = v.blk_node_off[b], q1 = v.blk_node_off[b + 1];
  for (int32_t q = q0 + threadIdx.x; q < q1; q += blockDim.x) {
    int32_t qo = v.owner_q[q];
    if (qo != q) v.loc2u[q] = v.loc2u[qo];
  }
}

// ------------------------------------------------------------------ residuals
// r_n = dt~_n - [(T_i - T_j) + (dt0_i - dt0_j)]  (Eq. 1; dt~ = dt - (t0_i - t0_j) of theta_0)
// and the whitening right-hand side u = B^T r (double-float), diag(lambda + B^T B) per node.
__global__ void k_resid(StepView v) {
  extern __shared__ float smf[];
  const int L_max = v.L_max;
  float* Thi = smf;
  float* Tlo = Thi + L_max;
  float* t0 = Tlo + L_max;
  float* rs = t0 + L_max;
  float* sw = rs + v.B;
  const int s = blockIdx.x;
  const int32_t b = v.sel[s];
  const int32_t q0 = v.blk_node_off[b];
  const int L = v.blk_node_off[b + 1] - q0;
  const int64_t e0 = v.blk_e0[b];
  const int ne = v.blk_e0[b + 1] - v.blk_e0[b];
  for (int l = threadIdx.x; l < L; l += blockDim.x) {
    const int32_t q = q0 + l;
    const float2 t = v.T2[v.loc2u[q]];
    Thi[l] = t.x;
    Tlo[l] = t.y;
    t0[l] = v.dth[v.pair_ev[v.node_pair[q]]].w;
  }
  for (int e = threadIdx.x; e < ne; e += blockDim.x) sw[e] = v.obs_sw[e0 + e];
  __syncthreads();
  for (int e = threadIdx.x; e < ne; e += blockDim.x) {
    const uint32_t lij = v.obs_l[e0 + e];
    const int li = lij & 0xFFFF, lj = lij >> 16;
    const float dhi = Thi[li] - Thi[lj];
    const float dlo = Tlo[li] - Tlo[lj];
    const float dt0 = t0[li] - t0[lj];
    const float r = ((v.obs_dt[e0 + e] - dhi) - dt0) - dlo;
    rs[e] = r;
    v.r_obs[e0 + e] = r;
  }
  __syncthreads();
  if (!v.whiten) return;
  const uint16_t* he = v.blk_he + 2 * e0;
  for (int l = threadIdx.x; l < L; l += blockDim.x) {
    const int32_t q = q0 + l;
    const int h0 = v.node_he[q];
    const int h1 = (l + 1 < L) ? (int)v.node_he[q + 1] : 2 * ne;
    df32 a = {0.f, 0.f};
    float d = 0.f;
    for (int h = h0; h < h1; ++h) {
      const int code = he[h];
      const int e = code >> 1;
      const float w = sw[e];
      a = df_add(a, df_two_prod((code & 1) ? -w : w, rs[e]));
      d += w * w;
    }
    if (!v.multi[q]) {
      const int32_t u = v.loc2u[q];
      v.rhs[u] = a.hi;
      v.rhs_lo[u] = a.lo;
      v.diag[u] = v.lam + d;
    } else {
      v.part_a[q] = a.hi;
      v.part_c[q] = a.lo;
      v.part_b[q] = d;
    }
  }
}

// u = B^T r and the diagonal of the pairs with several selected occurrences
__global__ void k_merge_rhs(StepView v) {
  const int32_t P_u = v.counters[kCntPairs];
  for (int32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < P_u; u += gridDim.x * blockDim.x) {
    if (!v.umulti[u]) continue;
    df32 a = {0.f, 0.f};
    float d = 0.f;
    for (int32_t q = v.uniq_q[u]; q >= 0; q = v.next_q[q]) {
      a = df_add(a, df32{v.part_a[q], v.part_c[q]});
      d += v.part_b[q];
    }
    v.rhs[u] = a.hi;
    v.rhs_lo[u] = a.lo;
    v.diag[u] = v.lam + d;
  }
}

struct BlockRange {
  int32_t q0;
  int L;
  int64_t e0;
  int ne;
};

__device__ __forceinline__ BlockRange block_range(const StepView& v, int64_t s) {
  BlockRange r;
  const int32_t b = v.sel[s];
  r.q0 = v.blk_node_off[b];
  r.L = v.blk_node_off[b + 1] - r.q0;
  r.e0 = v.blk_e0[b];
  r.ne = v.blk_e0[b + 1] - v.blk_e0[b];
  return r;
}

// q_e = sigma^-2 (r_e - sqrt(w_e) (z_i - z_j)) with z in double-float, the node
// sums s_p = sum_{e: p = i-end} q_e - sum_{e: p = j-end} q_e (= d loglik / d T_p),
// and r^T Sigma^-1 r = sum_e r_e q_e (FP64 per block).
__global__ void k_final(StepView v) {
  extern __shared__ float smf[];
  __shared__ double smd[33];
  if (aborted_cta(v)) return;
  float* zh = smf;
  float* zl = zh + v.L_max;
  float* qs = zl + v.L_max;
  const int s = blockIdx.x;
  const BlockRange br = block_range(v, s);
  for (int l = threadIdx.x; l < br.L; l += blockDim.x) {
    if (v.whiten) {
      const int32_t u = v.loc2u[br.q0 + l];
      zh[l] = v.z[u];
      zl[l] = v.z_lo[u];
    } else {
      zh[l] = 0.f;
      zl[l] = 0.f;
    }
  }
  __syncthreads();
  double quad = 0.0;
  for (int e = threadIdx.x; e < br.ne; e += blockDim.x) {
    const uint32_t lij = v.obs_l[br.e0 + e];
    const int li = lij & 0xFFFF, lj = lij >> 16;
    const df32 d = df_add(df32{zh[li], zl[li]}, df32{-zh[lj], -zl[lj]});
    const df32 bz = df_mul_f(d, v.obs_sw[br.e0 + e]);
    const float r = v.r_obs[br.e0 + e];
    float qe;
    if (v.loss == SPIDER_LOSS_L1) {
      // stage 1: d(-sum |r|)/dr = -sign(r); the quadratic slot carries 2|r| so
      // that the log posterior's -1/2 (quad) is -sum |r|
      qe = r > 0.f ? 1.f : (r < 0.f ? -1.f : 0.f);
      quad += 2.0 * fabs((double)r);
    } else {
      const df32 t = df_add_f(df32{-bz.hi, -bz.lo}, r);
      qe = v.inv_s2 * t.hi;
      quad += (double)r * (double)qe;
    }
    qs[e] = qe;
    v.q_obs[br.e0 + e] = qe;
  }
  quad = block_sum<double>(quad, smd);
  if (threadIdx.x == 0) v.dblk[s] = quad;
  const uint16_t* he = v.blk_he + 2 * br.e0;
  for (int l = threadIdx.x; l < br.L; l += blockDim.x) {
    const int32_t q = br.q0 + l;
    const int h0 = v.node_he[q];
    const int h1 = (l + 1 < br.L) ? (int)v.node_he[q + 1] : 2 * br.ne;
    float a = 0.f;
    for (int h = h0; h < h1; ++h) {
      const int code = he[h];
      a += (code & 1) ? -qs[code >> 1] : qs[code >> 1];
    }
    if (!v.multi[q]) v.s_u[v.loc2u[q]] = a;
    else v.part_a[q] = a;
  }
}

// s_p * (N_s/n_s) times (dT/dx_p, 1) into the global pair slots, stamped.
__global__ void k_merge_s(StepView v) {
  if (aborted(v)) return;
  const int tag = v.prm->tag;
  const int32_t P_u = v.counters[kCntPairs];
  for (int32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < P_u; u += gridDim.x * blockDim.x) {
    const int32_t q = v.uniq_q[u];
    const int32_t p = v.node_pair[q];
    const int32_t m = v.pair_ev[p];
    const int sb = v.ev_sub[m];
    const float scale = (float)((double)v.sub_nobs[sb] / (double)v.sub_nsel[sb]);
    float sp = v.multi[q] ? merge_occ(v, q, v.part_a) : v.s_u[u];
    sp *= scale;
    const float4 J = v.J[u];
    v.gp[p] = make_float4(sp * J.x, sp * J.y, sp * J.z, sp);
    v.pstamp[p] = tag;
    v.estamp[m] = tag;
  }
}

// ------------------------------------------------------------------ events
// centroid of the current state offset, per sub-problem: fixed chunks of
// events summed in a fixed tree, chunks summed in order
__global__ void k_cen_chunk(StepView v) {
  __shared__ float smr[33];
  if (aborted_cta(v)) return;
  const int c = blockIdx.x;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int32_t m = v.chunk_ev0[c] + threadIdx.x; m < v.chunk_ev0[c + 1]; m += blockDim.x) {
    const float4 d = v.dth[m];
    a.x += d.x; a.y += d.y; a.z += d.z; a.w += d.w;
  }
  a.x = block_sum<float>(a.x, smr);
  a.y = block_sum<float>(a.y, smr);
  a.z = block_sum<float>(a.z, smr);
  a.w = block_sum<float>(a.w, smr);
  if (threadIdx.x == 0) v.cen_chunk[c] = a;
}

__global__ void k_cen_final(StepView v) {
  __shared__ float smr[33];
  if (aborted_cta(v)) return;
  const int s = blockIdx.x;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int32_t c = v.sub_chunk_off[s] + threadIdx.x; c < v.sub_chunk_off[s + 1]; c += blockDim.x) {
    const float4 d = v.cen_chunk[c];
    a.x += d.x; a.y += d.y; a.z += d.z; a.w += d.w;
  }
  a.x = block_sum<float>(a.x, smr);
  a.y = block_sum<float>(a.y, smr);
  a.z = block_sum<float>(a.z, smr);
  a.w = block_sum<float>(a.w, smr);
  if (threadIdx.x == 0) {
    const float inv = 1.0f / (float)v.sub_nev[s];
    v.sub_cen[s] = make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv);
  }
}

// grad_m = (N_s/n_s) sum_k s_(m,k) (dT/dx, 1) - dtheta_m / sigma_e^2
//          - mean_s(dtheta) / (M_s sigma_c^2)             (priors of Sec. 3.1)
// mode 0: write grad; mode 1: SGLD theta += eps grad + ns sqrt(2 eps) eta (Sec. 3.2)
__global__ void k_event(StepView v) {
  __shared__ double smd[33];
  if (aborted_cta(v)) return;
  const StepParams& pr = *v.prm;
  const int tag = pr.tag, mode = pr.mode;
  const float eps = pr.eps;
  const float4 ise = v.inv_sig_e2, isc = v.inv_sig_c2;
  const float sq = pr.noise_scale * sqrtf(2.0f * eps);
  const uint2 key = seed_key(pr.seed);
  double lp = 0.0;
  int bad = 0, touched = 0;
  for (int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; m < v.M; m += (int64_t)gridDim.x * blockDim.x) {
    const int sb = v.ev_sub[m];
    const float4 cen = v.sub_cen[sb];
    const float invM = 1.0f / (float)v.sub_nev[sb];
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    if (v.estamp[m] == tag) {
      ++touched;
      for (int32_t p = v.pair_off[m], p1 = v.pair_off[m + 1]; p < p1; ++p)
        if (v.pstamp[p] == tag) {
          const float4 c = v.gp[p];
          g.x += c.x; g.y += c.y; g.z += c.z; g.w += c.w;
        }
    }
    const float4 d = v.dth[m];
    g.x -= d.x * ise.x + cen.x * isc.x * invM;
    g.y -= d.y * ise.y + cen.y * isc.y * invM;
    g.z -= d.z * ise.z + cen.z * isc.z * invM;
    g.w -= d.w * ise.w + cen.w * isc.w * invM;
    if (mode == 0) {
      v.grad[m] = g;
      lp += (double)d.x * d.x * ise.x + (double)d.y * d.y * ise.y + (double)d.z * d.z * ise.z +
            (double)d.w * d.w * ise.w;
      if (!(isfinite(g.x) && isfinite(g.y) && isfinite(g.z) && isfinite(g.w))) bad = 1;
    } else {
      float4 nd;
      if (v.update == SPIDER_UPDATE_ADAM) {
        // stage-1 optimiser: Adam ascent on the objective, no noise
        float4 m1 = v.mom1[m], m2 = v.mom2[m];
        const float b1 = v.beta1, b2 = v.beta2;
        m1.x = fmaf(b1, m1.x, (1.f - b1) * g.x); m2.x = fmaf(b2, m2.x, (1.f - b2) * (g.x * g.x));
        m1.y = fmaf(b1, m1.y, (1.f - b1) * g.y); m2.y = fmaf(b2, m2.y, (1.f - b2) * (g.y * g.y));
        m1.z = fmaf(b1, m1.z, (1.f - b1) * g.z); m2.z = fmaf(b2, m2.z, (1.f - b2) * (g.z * g.z));
        m1.w = fmaf(b1, m1.w, (1.f - b1) * g.w); m2.w = fmaf(b2, m2.w, (1.f - b2) * (g.w * g.w));
        v.mom1[m] = m1;
        v.mom2[m] = m2;
        const float bc1 = pr.bc1, bc2 = pr.bc2, pe = v.upd_eps;
        nd.x = d.x + eps * (m1.x * bc1) / (sqrtf(m2.x * bc2) + pe);
        nd.y = d.y + eps * (m1.y * bc1) / (sqrtf(m2.y * bc2) + pe);
        nd.z = d.z + eps * (m1.z * bc1) / (sqrtf(m2.z * bc2) + pe);
        nd.w = d.w + eps * (m1.w * bc1) / (sqrtf(m2.w * bc2) + pe);
      } else {
        const uint4 w = philox4x32_10(
            make_uint4((uint32_t)v.ev_caller[m], (uint32_t)v.sub_chain[sb], (uint32_t)v.sub_catalog[sb], kTagNoise),
            key);
        const float2 n01 = box_muller(w.x, w.y), n23 = box_muller(w.z, w.w);
        if (v.update == SPIDER_UPDATE_PSGLD) {
          // Eq. pSGLD: per-coordinate preconditioner from the running second moment
          float4 m2 = v.mom2[m];
          const float b2 = v.beta2, pe = v.upd_eps, ns = pr.noise_scale;
          m2.x = fmaf(b2, m2.x, (1.f - b2) * (g.x * g.x));
          m2.y = fmaf(b2, m2.y, (1.f - b2) * (g.y * g.y));
          m2.z = fmaf(b2, m2.z, (1.f - b2) * (g.z * g.z));
          m2.w = fmaf(b2, m2.w, (1.f - b2) * (g.w * g.w));
          v.mom2[m] = m2;
          const float Vx = 1.f / (sqrtf(m2.x) + pe), Vy = 1.f / (sqrtf(m2.y) + pe);
          const float Vz = 1.f / (sqrtf(m2.z) + pe), Vw = 1.f / (sqrtf(m2.w) + pe);
          nd.x = d.x + eps * Vx * g.x + ns * sqrtf(2.f * eps * Vx) * n01.x;
          nd.y = d.y + eps * Vy * g.y + ns * sqrtf(2.f * eps * Vy) * n01.y;
          nd.z = d.z + eps * Vz * g.z + ns * sqrtf(2.f * eps * Vz) * n23.x;
          nd.w = d.w + eps * Vw * g.w + ns * sqrtf(2.f * eps * Vw) * n23.y;
        } else {
          nd.x = d.x + eps * g.x + sq * n01.x;
          nd.y = d.y + eps * g.y + sq * n01.y;
          nd.z = d.z + eps * g.z + sq * n23.x;
          nd.w = d.w + eps * g.w + sq * n23.y;
        }
      }
      if (!(isfinite(nd.x) && isfinite(nd.y) && isfinite(nd.z) && isfinite(nd.w))) bad = 1;
      v.dth[m] = nd;
      if (pr.sample_slot >= 0) v.samples[pr.sample_slot * v.M + m] = nd;
    }
  }
  if (bad) set_error(v.counters, SPIDER_E_NONFINITE);
  touched = block_sum<int>(touched, reinterpret_cast<int*>(smd));
  if (threadIdx.x == 0 && touched) atomicAdd(&v.counters[kCntEvents], touched);
  if (mode == 0) {
    lp = block_sum<double>(lp, smd);
    if (threadIdx.x == 0) v.dred[2 * kMaxGrid + blockIdx.x] = lp;
  }
}

// FP64 log posterior: sum_s -1/2 (N_s/n_s) r_s^T Sigma^-1 r_s - 1/2 |dtheta/sigma_e|^2
//                     - 1/2 sum_s |mean_s(dtheta)/sigma_c|^2   (constants dropped)
__global__ void k_logpost(StepView v, int64_t n_b) {
  __shared__ double smd[33];
  if (aborted_cta(v)) return;
  double quad = 0.0, lp = 0.0;
  for (int64_t t = threadIdx.x; t < n_b; t += blockDim.x) {
    const int sb = v.blk_sub[v.sel[t]];
    quad += v.dblk[t] * ((double)v.sub_nobs[sb] / (double)v.sub_nsel[sb]);
  }
  for (int i = threadIdx.x; i < v.cen_grid; i += blockDim.x) lp += v.dred[2 * kMaxGrid + i];
  quad = block_sum<double>(quad, smd);
  lp = block_sum<double>(lp, smd);
  double lc = 0.0;
  const float isc[4] = {v.inv_sig_c2.x, v.inv_sig_c2.y, v.inv_sig_c2.z, v.inv_sig_c2.w};
  for (int sb = threadIdx.x; sb < v.n_sub; sb += blockDim.x) {
    const float4 c = v.sub_cen[sb];
    const double cc[4] = {c.x, c.y, c.z, c.w};
    for (int a = 0; a < 4; ++a) lc += cc[a] * cc[a] * (double)isc[a];
  }
  lc = block_sum<double>(lc, smd);
  if (threadIdx.x == 0) {
    const double ll = -0.5 * quad;
    v.dout[0] = ll;
    v.dout[1] = -0.5 * lp;
    v.dout[2] = -0.5 * lc;
    v.dout[3] = ll - 0.5 * lp - 0.5 * lc;
  }
}

// FP64 diagnostics: |g_m| of the minibatch gradient and sum (g - G)^2
__global__ void k_diag(StepView v, const float4* __restrict__ g, const float4* __restrict__ G,
                       double* norms, double* part) {
  __shared__ double smd[33];
  double acc = 0.0;
  for (int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; m < v.M; m += (int64_t)gridDim.x * blockDim.x) {
    const float4 a = g[m], b = G[m];
    norms[m] = sqrt((double)a.x * a.x + (double)a.y * a.y + (double)a.z * a.z + (double)a.w * a.w);
    const double dx = (double)a.x - b.x, dy = (double)a.y - b.y, dz = (double)a.z - b.z, dw = (double)a.w - b.w;
    acc += dx * dx + dy * dy + dz * dz + dw * dw;
  }
  acc = block_sum<double>(acc, smd);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// theta = theta_0 + dtheta in FP64, written in the caller's event order (the
// read-back of spider_get_state / spider_samples); src is the state offset or
// one stored sample.
__global__ void k_state_out(StepView v, const float4* __restrict__ src, double* __restrict__ out) {
  for (int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; m < v.M; m += (int64_t)gridDim.x * blockDim.x) {
    const float4 d = src[m];
    const double* t = v.th0_d + 4 * m;
    double4 o;
    o.x = t[0] + (double)d.x;
    o.y = t[1] + (double)d.y;
    o.z = t[2] + (double)d.z;
    o.w = t[3] + (double)d.w;
    reinterpret_cast<double4*>(out)[v.ev_out[m]] = o;
  }
}

// the gradient (FP32) in the caller's event order
__global__ void k_grad_out(StepView v, float4* __restrict__ out) {
  for (int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; m < v.M; m += (int64_t)gridDim.x * blockDim.x)
    out[v.ev_out[m]] = v.grad[m];
}

__global__ void k_philox_words(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                               int64_t n, uint32_t* out) {
  int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n) return;
  uint4 w = philox4x32_10(make_uint4(c0 + (uint32_t)m, c1, c2, c3), seed_key(seed));
  reinterpret_cast<uint4*>(out)[m] = w;
}

}  // namespace

// ------------------------------------------------------------------ launchers
#define CK_LAUNCH(call)                      \
  do {                                       \
    cudaError_t _e = (call);                 \
    if (_e != cudaSuccess) return _e;        \
  } while (0)

static inline int grid_for(int64_t n, int t = kThreads) { return (int)((n + t - 1) / t); }

cudaError_t launch_select(const StepView& v, int64_t n_b, cudaStream_t st, int bthreads) {
  k_select<<<grid_for(n_b), kThreads, 0, st>>>(v, n_b);
  k_owner<<<(unsigned)n_b, bthreads, 0, st>>>(v);
  k_scan_owner<<<1, 1024, 0, st>>>(v, n_b);
  k_assign<<<(unsigned)n_b, bthreads, 0, st>>>(v);
  k_link<<<(unsigned)n_b, bthreads, 0, st>>>(v);
  return cudaGetLastError();
}

size_t resid_smem(const StepView& v) { return (size_t)(3 * v.L_max + 2 * v.B) * sizeof(float); }
size_t final_smem(const StepView& v) { return (size_t)(2 * v.L_max + v.B) * sizeof(float); }

// The limits are those of the largest block there can be (4096 observations of
// 8192 local nodes), whatever this context needs: they belong to the kernels,
// and a context with smaller blocks must not lower them for an older one.
cudaError_t configure_step_kernels() {
  constexpr int kObs = 4096, kNodes = 2 * kObs;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_resid, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)((3 * kNodes + 2 * kObs) * sizeof(float)))))
    return e;
  return cudaFuncSetAttribute(k_final, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)((2 * kNodes + kObs) * sizeof(float)));
}

// ev (or null): events recorded after k_resid and after k_merge_rhs
cudaError_t launch_resid(const StepView& v, int64_t n_b, int gu, cudaStream_t st, const cudaEvent_t* ev,
                         int bthreads) {
  k_resid<<<(unsigned)n_b, bthreads, resid_smem(v), st>>>(v);
  if (ev) CK_LAUNCH(cudaEventRecord(ev[0], st));
  if (v.whiten) k_merge_rhs<<<gu, kThreads, 0, st>>>(v);
  if (ev) CK_LAUNCH(cudaEventRecord(ev[1], st));
  return cudaGetLastError();
}

// ev (or null): events recorded after k_final, k_merge_s, the centroid, k_event
cudaError_t launch_finish(const StepView& v, int64_t n_b, int gu, bool logpost, cudaStream_t st,
                          const cudaEvent_t* ev, int bthreads) {
  k_final<<<(unsigned)n_b, bthreads, final_smem(v), st>>>(v);
  if (ev) CK_LAUNCH(cudaEventRecord(ev[0], st));
  k_merge_s<<<gu, kThreads, 0, st>>>(v);
  if (ev) CK_LAUNCH(cudaEventRecord(ev[1], st));
  k_cen_chunk<<<v.n_chunks, kThreads, 0, st>>>(v);
  k_cen_final<<<v.n_sub, kThreads, 0, st>>>(v);
  if (ev) CK_LAUNCH(cudaEventRecord(ev[2], st));
  k_event<<<v.cen_grid, kThreads, 0, st>>>(v);
  if (ev) CK_LAUNCH(cudaEventRecord(ev[3], st));
  if (logpost) k_logpost<<<1, kThreads, 0, st>>>(v, n_b);
  return cudaGetLastError();
}

cudaError_t launch_diag(const StepView& v, const float4* g, const float4* G, double* norms, double* part,
                        int grid, cudaStream_t st) {
  k_diag<<<grid, kThreads, 0, st>>>(v, g, G, norms, part);
  return cudaGetLastError();
}

cudaError_t launch_state_out(const StepView& v, const float4* src, double* out, int grid, cudaStream_t st) {
  k_state_out<<<grid, kThreads, 0, st>>>(v, src, out);
  return cudaGetLastError();
}

cudaError_t launch_grad_out(const StepView& v, float4* out, int grid, cudaStream_t st) {
  k_grad_out<<<grid, kThreads, 0, st>>>(v, out);
  return cudaGetLastError();
}

cudaError_t launch_philox_words(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                int64_t n, uint32_t* out, cudaStream_t st) {
  k_philox_words<<<grid_for(n), kThreads, 0, st>>>(seed, c0, c1, c2, c3, n, out);
  return cudaGetLastError();
}

}  // namespace spider
