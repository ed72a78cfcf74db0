// Travel times T(x; s) and source Jacobians dT/dx for a list of
// (event, station) pairs (Sec. 2.1 and the forward model of Eq. forwardmodel).
//
//  * homogeneous medium: T = r / v, dT/dx = (x - s) / (v r), with r and T in
//    double-float so that dd differences keep sub-microsecond accuracy;
//  * linear-gradient medium v = v0 + g z: T = arccosh(1 + g^2 r^2/(2 v_x v_s))/g
//    in FP32;
//  * MLP stand-in for EikoNet (Sec. 3.2): T = r * tau(x, s), tau = 6 -> 4 x H
//    SiLU -> 1, with the source Jacobian by a hand-written reverse sweep
//    (delta_L = w_out * silu'(z_L), delta_{l-1} = (W_l^T delta_l) * silu'(z_{l-1}),
//    dtau/dx = W_1[:, :3]^T delta_1) and dT/dx = tau (x - s)/r + r dtau/dx.
//    This file holds the FP32 SIMT form; the tensor-core forms live in k_mlp_tc.cu.
#include <cuda_runtime.h>

#include <cstdint>

#include "dfloat.cuh"
#include "kernels.h"
#include "mlp32.h"
#include "pairs.cuh"
#include "spider.h"

namespace spider {

namespace {

__global__ void k_tt_homogeneous(NetView net, PairSource src, TTOut out) {
  const int64_t P = pair_count(src);
  const df32 inv_v = {net.inv_v_hi, net.inv_v_lo};
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < P;
       u += (int64_t)gridDim.x * blockDim.x) {
    PairGeo g;
    load_pair(src, u, g);
    df32 d[3];
    const df32 r = geometry(g, d);
    const df32 T = df_mul(r, inv_v);
    store_time(out, u, T.hi, T.lo);
    if (out.J) {
      const float f = net.inv_v_hi / r.hi;
      out.J[u] = make_float4(d[0].hi * f, d[1].hi * f, d[2].hi * f, 0.f);
    }
  }
}

__global__ void k_tt_gradient(NetView net, PairSource src, TTOut out) {
  const int64_t P = pair_count(src);
  const float v0 = net.v0, gg = net.g;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < P;
       u += (int64_t)gridDim.x * blockDim.x) {
    PairGeo g;
    load_pair(src, u, g);
    df32 d[3];
    const df32 r = geometry(g, d);
    const float zs = g.shi[2] + (g.slo[2] + g.soff[2]);
    const float zr = g.rhi[2] + g.rlo[2];
    const float vs = v0 + gg * zs, vr = v0 + gg * zr;
    const float X = gg * gg * r.hi * r.hi / (2.f * vs * vr);
    const float sq = sqrtf(X * (2.f + X));
    const float T = log1pf(X + sq) / gg;
    store_time(out, u, T, 0.f);
    if (out.J) {
      const float dTdX = 1.f / (gg * sq);
      const float c = dTdX * gg * gg / (vs * vr);
      out.J[u] = make_float4(c * d[0].hi, c * d[1].hi, c * d[2].hi - dTdX * X * gg / vs, 0.f);
    }
  }
}

// ------------------------------------------------------------------ FP32 MLP
__device__ __forceinline__ void silu_fp32(float z, float& h, float& ds) {
  const float s = 1.0f / (1.0f + expf(-z));
  h = z * s;
  ds = s * (1.0f + z * (1.0f - s));
}

// d = a * b + d on two FP32 lanes: each lane rounds as fmaf does
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t pack2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float half2_of(uint64_t v, int hi) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return hi ? b : a;
}
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Persistent FP32 SIMT MLP.  Wide form: tiles of 64 pairs; a warp computes 64
// pairs x 32 hidden units, a lane 2 pairs x 32 units as 32 packed FMAs (two units
// each) a step of k.  The packed FMA runs at the FP32 rate with half the issue
// slots, which leaves the other half to the loads: one 8-byte load of the lane's
// two activations (doubled in registers) and eight 16-byte loads of the warp's 32
// weights, the same for every lane.  That is about 18 wavefronts of the SM's shared
// memory against the 16 cycles its FMA lanes take (a 16-byte load takes two even where
// all lanes read one address; counted at 250,007 pairs and H = 128: shared memory busy
// 72 % of the time, FMA lanes 62 %), so shared memory is what bounds it, with 14 warps
// an SM to overlap the two.
// Narrow form, for launches that leave SMs without a tile: tiles of 32 pairs, a
// lane one pair x 8 units, so a tile is spread over eight times the lanes.
// Every output is one chain of fused multiply-adds over k in ascending order,
// and the units are summed in ascending order in groups of H / 8, in both forms.
// The weights stream through three chunks of 8 rows (asynchronous copies, one
// barrier per chunk) in one sequence over the six products of every tile, so the
// next product's first rows arrive during the epilogue.  silu'(z) of layers 1-3
// goes to a per-CTA scratch slot (rewritten every tile, so it stays in L2).
// 300,000 pairs at H = 256: 8.41 -> 4.93 ms (28 -> 48 TFLOP/s of the 80 the FP32
// lanes could do); 250,007 at H = 128: 1.58 -> 1.14 ms; 47 at H = 64: 47 -> 38 us.
// The shapes are in mlp32.h.
template <int PL>
struct Lanes {
  float v[PL];
};
template <int PL>
__device__ __forceinline__ Lanes<PL> ld_lanes(const float* p) {
  Lanes<PL> r;
  if constexpr (PL == 2) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    r.v[0] = t.x;
    r.v[1] = t.y;
  } else {
    r.v[0] = *p;
  }
  return r;
}
template <int PL>
__device__ __forceinline__ void st_lanes(float* p, const Lanes<PL>& r) {
  if constexpr (PL == 2) *reinterpret_cast<float2*>(p) = make_float2(r.v[0], r.v[1]);
  else *p = r.v[0];
}

template <int H, bool WIDE>
__global__ void __launch_bounds__(Mlp32<H, WIDE>::kThreads, Mlp32<H, WIDE>::kCtas)
    k_tt_mlp_fp32(NetView net, PairSource src, TTOut out, float* __restrict__ scratch) {
  using C = Mlp32<H, WIDE>;
  constexpr int PL = C::kPl, UW = C::kUw, TP = C::kTile;
  using L = Lanes<PL>;
  extern __shared__ __align__(16) float sm[];
  float* act = sm;                                   // [H][TP]
  float* wbuf = act + H * TP;                        // [kStagesW][kKC][H]
  float* xin = wbuf + kStagesW * C::kChunkW;         // [6][TP]
  float* red = xin + 6 * TP;                         // [kGroups][4][TP]
  float* hold = red + kGroups * 4 * TP;              // [H][TP], narrow form
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  float* dsg = scratch + (size_t)blockIdx.x * 3 * H * TP;
  const int64_t P = pair_count(src);
  const int64_t ntiles = (P + TP - 1) / TP;
  const int64_t mine = ntiles > blockIdx.x ? (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  const int64_t chunks = mine * C::kTotal;
  const float4* wsrc = reinterpret_cast<const float4*>(net.Wd);
  constexpr int kVec = C::kChunkW / 4;               // 16-byte words of a chunk
  int64_t loaded = 0;
  int lc = 0, ls = 0;                                // next chunk to load: index in the images, stage
  auto load = [&]() {
    if (loaded < chunks) {
      float4* d = reinterpret_cast<float4*>(wbuf) + ls * kVec;
      const float4* g = wsrc + (size_t)lc * kVec;
#pragma unroll
      for (int i = 0; i < (kVec + C::kThreads - 1) / C::kThreads; ++i) {
        const int k = i * C::kThreads + tid;
        if (kVec % C::kThreads == 0 || k < kVec) copy16(d + k, g + k);
      }
      ++loaded;
      lc = lc + 1 == C::kTotal ? 0 : lc + 1;
      ls = ls + 1 == kStagesW ? 0 : ls + 1;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int i = 0; i < kStagesW - 1; ++i) load();
  int cs = 0;                                        // stage of the next chunk to use
  uint64_t acc[PL][UW / 2];                          // [pair][two units]
  // acc = act^T x the next H rows of the weight sequence
  auto product = [&]() {
#pragma unroll
    for (int p = 0; p < PL; ++p)
#pragma unroll
      for (int q = 0; q < UW / 2; ++q) acc[p][q] = 0ull;
#pragma unroll 1
    for (int c = 0; c < H / kKC; ++c) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kStagesW - 2) : "memory");
      __syncthreads();
      load();
      const float* wb = wbuf + cs * C::kChunkW + UW * w;
      const float* ab = act + c * kKC * TP + PL * lane;
      cs = cs + 1 == kStagesW ? 0 : cs + 1;
#pragma unroll
      for (int kk = 0; kk < kKC; ++kk) {
        const L a = ld_lanes<PL>(ab + kk * TP);
        uint64_t a2[PL];
#pragma unroll
        for (int p = 0; p < PL; ++p) a2[p] = pack2(a.v[p], a.v[p]);
#pragma unroll
        for (int q = 0; q < UW / 4; ++q) {
          const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(wb + kk * H + 4 * q);
#pragma unroll
          for (int p = 0; p < PL; ++p) fma2(acc[p][2 * q], a2[p], b.x);
#pragma unroll
          for (int p = 0; p < PL; ++p) fma2(acc[p][2 * q + 1], a2[p], b.y);
        }
      }
    }
    __syncthreads();                                 // every read of act for this product is done
  };
  auto value = [&](int p, int u) { return half2_of(acc[p][u >> 1], u & 1); };
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t u0 = tile * TP;
    __syncthreads();
    for (int t = tid; t < TP; t += C::kThreads) {
      const int64_t u = u0 + t;
      PairGeo g;
      load_pair(src, u < P ? u : u0, g);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        xin[c * TP + t] = g.shi[c] + (g.slo[c] + g.soff[c]);
        xin[(3 + c) * TP + t] = g.rhi[c] + g.rlo[c];
      }
    }
    __syncthreads();
    // layer 1 (6 -> H)
    {
      L x[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) x[c] = ld_lanes<PL>(xin + c * TP + PL * lane);
#pragma unroll 4
      for (int u = 0; u < UW; ++u) {
        const int n = UW * w + u;
        const float b = __ldg(net.b1 + n);
        float wc[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) wc[c] = __ldg(net.W1 + n * 6 + c);
        L h, ds;
#pragma unroll
        for (int p = 0; p < PL; ++p) {
          float z = b;
#pragma unroll
          for (int c = 0; c < 6; ++c) z = fmaf(wc[c], x[c].v[p], z);
          silu_fp32(z, h.v[p], ds.v[p]);
        }
        st_lanes<PL>(act + n * TP + PL * lane, h);
        st_lanes<PL>(dsg + n * TP + PL * lane, ds);
      }
    }
    // layers 2..4
#pragma unroll 1
    for (int lyr = 0; lyr < 3; ++lyr) {
      product();
      L t{};                                         // partial sum of tau (layer 4)
#pragma unroll
      for (int u = 0; u < UW; ++u) {
        const int n = UW * w + u;
        const float b = __ldg(net.bh[lyr] + n);
        L h, ds;
#pragma unroll
        for (int p = 0; p < PL; ++p) silu_fp32(value(p, u) + b, h.v[p], ds.v[p]);
        if (lyr < 2) {
          st_lanes<PL>(act + n * TP + PL * lane, h);
          st_lanes<PL>(dsg + ((lyr + 1) * H + n) * TP + PL * lane, ds);
        } else {
          const float w5 = __ldg(net.W5 + n);
          if constexpr (WIDE) {
            if (u % C::kUpg == 0) t = L{};
#pragma unroll
            for (int p = 0; p < PL; ++p) t.v[p] = fmaf(w5, h.v[p], t.v[p]);
            if ((u + 1) % C::kUpg == 0) st_lanes<PL>(red + (n / C::kUpg) * 4 * TP + PL * lane, t);
          } else {
            st_lanes<PL>(hold + n * TP + PL * lane, h);
          }
#pragma unroll
          for (int p = 0; p < PL; ++p) ds.v[p] = w5 * ds.v[p];
          st_lanes<PL>(act + n * TP + PL * lane, ds);          // delta_4
        }
      }
    }
    // backward: delta_{l-1} = (W_l^T delta_l) * silu'(z_{l-1}), l = 4, 3
#pragma unroll 1
    for (int lyr = 2; lyr >= 1; --lyr) {
      product();
#pragma unroll
      for (int u = 0; u < UW; ++u) {
        const int n = UW * w + u;
        L d = ld_lanes<PL>(dsg + (lyr * H + n) * TP + PL * lane);
#pragma unroll
        for (int p = 0; p < PL; ++p) d.v[p] = value(p, u) * d.v[p];
        st_lanes<PL>(act + n * TP + PL * lane, d);
      }
    }
    // delta_1 = (W_2^T delta_2) * silu'(z_1); dtau/dx_src = W_1[:, :3]^T delta_1
    product();
    {
      L g3[3] = {};
#pragma unroll
      for (int u = 0; u < UW; ++u) {
        const int n = UW * w + u;
        L d = ld_lanes<PL>(dsg + n * TP + PL * lane);
#pragma unroll
        for (int p = 0; p < PL; ++p) d.v[p] = value(p, u) * d.v[p];
        if constexpr (WIDE) {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            if (u % C::kUpg == 0) g3[c] = L{};
            const float wc = __ldg(net.W1 + n * 6 + c);
#pragma unroll
            for (int p = 0; p < PL; ++p) g3[c].v[p] = fmaf(wc, d.v[p], g3[c].v[p]);
            if ((u + 1) % C::kUpg == 0) st_lanes<PL>(red + ((n / C::kUpg) * 4 + 1 + c) * TP + PL * lane, g3[c]);
          }
        } else {
          st_lanes<PL>(act + n * TP + PL * lane, d);
        }
      }
    }
    __syncthreads();
    if constexpr (!WIDE) {
      // a group's units lie on several warps: one thread per pair and group
      for (int i = tid; i < kGroups * TP; i += C::kThreads) {
        const int p = i % TP, g = i / TP;
        float t = 0.f, g3[3] = {0.f, 0.f, 0.f};
#pragma unroll 4
        for (int u = 0; u < C::kUpg; ++u) {
          const int n = g * C::kUpg + u;
          t = fmaf(__ldg(net.W5 + n), hold[n * TP + p], t);
          const float d1 = act[n * TP + p];
#pragma unroll
          for (int c = 0; c < 3; ++c) g3[c] = fmaf(__ldg(net.W1 + n * 6 + c), d1, g3[c]);
        }
        red[g * 4 * TP + p] = t;
#pragma unroll
        for (int c = 0; c < 3; ++c) red[(g * 4 + 1 + c) * TP + p] = g3[c];
      }
      __syncthreads();
    }
    for (int t = tid; t < TP; t += C::kThreads) {
      const int64_t u = u0 + t;
      if (u >= P) continue;
      float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int ww = 0; ww < kGroups; ++ww)
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c] += red[(ww * 4 + c) * TP + t];
      PairGeo g;
      load_pair(src, u, g);
      df32 d[3];
      const df32 r = geometry(g, d);
      // T = r * (b5 + dtau): the bias part in double-float, the network part in FP32
      const df32 T = df_add_f(df_mul_f(r, net.b5), r.hi * s[0]);
      store_time(out, u, T.hi, T.lo);
      if (out.J) {
        const float tau = net.b5 + s[0];
        const float f = tau / r.hi;
        out.J[u] = make_float4(f * d[0].hi + r.hi * s[1], f * d[1].hi + r.hi * s[2], f * d[2].hi + r.hi * s[3], 0.f);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <int H, bool WIDE>
cudaError_t launch_form(const NetView& net, const PairSource& src, TTOut out, int grid, float* scratch,
                        cudaStream_t st) {
  using C = Mlp32<H, WIDE>;
  cudaError_t e =
      cudaFuncSetAttribute(k_tt_mlp_fp32<H, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kSmem);
  if (e != cudaSuccess) return e;
  k_tt_mlp_fp32<H, WIDE><<<grid, C::kThreads, C::kSmem, st>>>(net, src, out, scratch);
  return cudaGetLastError();
}

template <int H>
cudaError_t launch_mlp_fp32(const NetView& net, const PairSource& src, TTOut out, int num_sms, int ctas_per_sm,
                            float* scratch, cudaStream_t st) {
  // never above the scratch slots
  if (narrow_form(H, src.n_host, num_sms))
    return launch_form<H, false>(net, src, out, narrow_ctas(H) * num_sms, scratch, st);
  return launch_form<H, true>(net, src, out, (ctas_per_sm == 1 ? 1 : mlp_fp32_ctas(H)) * num_sms, scratch, st);
}

}  // namespace

size_t tt_scratch_floats(const NetView& net, int num_sms) {
  if (net.kind != SPIDER_TT_MLP) return 0;
  const size_t fp32 = (size_t)mlp_fp32_ctas(net.H) * num_sms * 3 * net.H * kTP;
  const size_t tc = (size_t)num_sms * 3 * 128 * net.H / 2; // three 128 x H BF16 slots per SM
  return net.precision == SPIDER_FP32 ? fp32 : tc;
}

bool tt_supported_width(int H) { return H == 32 || H == 64 || H == 128 || H == 256; }

cudaError_t launch_tt(const NetView& net, const PairSource& src, TTOut out, int num_sms, float* scratch,
                      cudaStream_t st, int ctas_per_sm) {
  if (net.kind == SPIDER_TT_HOMOGENEOUS) {
    k_tt_homogeneous<<<4 * num_sms, 256, 0, st>>>(net, src, out);
    return cudaGetLastError();
  }
  if (net.kind == SPIDER_TT_LINEAR_GRADIENT) {
    k_tt_gradient<<<4 * num_sms, 256, 0, st>>>(net, src, out);
    return cudaGetLastError();
  }
  if (net.precision != SPIDER_FP32) {
    cudaError_t e = launch_mlp_tc(net, src, out, num_sms, scratch, st);
    if (e != cudaErrorNotSupported) return e;
    return cudaErrorNotSupported;
  }
  switch (net.H) {
    case 32: return launch_mlp_fp32<32>(net, src, out, num_sms, ctas_per_sm, scratch, st);
    case 64: return launch_mlp_fp32<64>(net, src, out, num_sms, ctas_per_sm, scratch, st);
    case 128: return launch_mlp_fp32<128>(net, src, out, num_sms, ctas_per_sm, scratch, st);
    case 256: return launch_mlp_fp32<256>(net, src, out, num_sms, ctas_per_sm, scratch, st);
    default: return cudaErrorNotSupported;
  }
}

cudaError_t launch_times(const NetView& net, const PairSource& src, float* T_hi, float* T_lo, float* J, float2* stage,
                         int num_sms, float* scratch, cudaStream_t st) {
  const size_t P = (size_t)src.n_host;
  auto apart = [](const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
    return !a || !b || x + na <= y || y + nb <= x;
  };
  const void* other[3] = {src.src, src.rcv, J};
  bool direct = true;
  for (const void* o : other) direct = direct && apart(T_hi, 4 * P, o, 16 * P) && apart(T_lo, 4 * P, o, 16 * P);
  direct = direct && apart(T_hi, 4 * P, T_lo, 4 * P);
  if (direct) return launch_tt(net, src, TTOut{nullptr, reinterpret_cast<float4*>(J), T_hi, T_lo}, num_sms, scratch, st, 2);
  float2* T2 = stage;
  cudaError_t e = cudaSuccess;
  if (!T2 && (e = cudaMallocAsync(&T2, P * sizeof(float2), st)) != cudaSuccess) return cudaErrorMemoryAllocation;
  e = launch_tt(net, src, TTOut{T2, reinterpret_cast<float4*>(J), nullptr, nullptr}, num_sms, scratch, st, 2);
  if (e == cudaSuccess)
    e = cudaMemcpy2DAsync(T_hi, sizeof(float), T2, sizeof(float2), sizeof(float), P, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && T_lo)
    e = cudaMemcpy2DAsync(T_lo, sizeof(float), reinterpret_cast<float*>(T2) + 1, sizeof(float2), sizeof(float), P,
                          cudaMemcpyDeviceToDevice, st);
  if (!stage) {
    const cudaError_t e2 = cudaFreeAsync(T2, st);
    if (e == cudaSuccess) e = e2;
  }
  return e;
}

}  // namespace spider
