// Device-side views shared by the step kernels (plain pointers, passed by value).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace spider {

// counters[] slots (int32, device)
enum : int {
  kCntPairs = 0,     // P_u: unique pairs of the current minibatch
  kCntObs = 1,       // n: observations of the current minibatch
  kCntIters = 2,     // largest CG iteration count of a component on several CTAs
  kCntError = 3,     // first device-side error (SPIDER_E_*), sticky until read
  kCntBarArrive = 4, // grid barrier arrivals of this evaluation
  kCntComps = 5,     // connected components of the minibatch graph
  kCntCompIters = 6, // largest CG iteration count of a component on one warp or CTA, or rounds of a stored inverse
  kCntEvents = 7,    // events touched by the minibatch (with at least one pair)
  kCntSlots = 8
};

// Travel-time network on the device.
struct NetView {
  int kind;          // SPIDER_TT_*
  int H;
  int precision;     // SPIDER_FP32 / BF16 / FP8
  float v0, g;
  float inv_v_hi, inv_v_lo;   // 1/v0 as a double-float
  const float* W1;   // H x 6 (out, in)
  const float* b1;   // H
  // FP32: the six products' weights in the order the kernel reads them:
  // W2^T, W3^T, W4^T ([in][out], forward), W4, W3, W2 ([out][in], reverse)
  const float* Wd;
  const float* bh[3];  // b2..b4
  const float* W5;     // H
  float b5;
  const void* tc;      // tensor-core operand images (BF16 / FP8), null in FP32
  const float* tc_scale;  // per-layer FP8 dequantisation scales (6), null otherwise
  int32_t* err;           // device error flag the tensor-core kernel reports bounded-wait timeouts to
};

// Where the pairs of a travel-time launch come from.
struct PairSource {
  // problem mode: pair u -> uniq_pair[u] -> (event, station)
  const int32_t* uniq_pair;
  const int32_t* pair_ev;
  const int32_t* pair_st;
  const float4* th0_hi;   // event theta_0 (hi)
  const float4* th0_lo;   // event theta_0 (lo)
  const float4* dth;      // event state offset theta - theta_0
  const float4* sta_hi;
  const float4* sta_lo;
  // raw mode (uniq_pair == nullptr): absolute FP32 positions per pair
  const float4* src;
  const float4* rcv;
  const float* src3;      // the same as rows of three (src == nullptr)
  const float* rcv3;
  const int32_t* n_dev;   // device count (problem mode) or nullptr
  int64_t n_host;         // host count (raw mode) / upper bound
};

struct TTOut {
  float2* T2;   // (T_hi, T_lo), or null: hi and lo (may be null) apart
  float4* J;    // (dT/dx, dT/dy, dT/dz, 0), may be null
  float* hi;
  float* lo;
  bool sum;     // hi takes T_hi + T_lo rounded
};

// Per-step parameters, read by the kernels from device memory (the host
// writes them before each step, so a captured step graph can be relaunched).
struct StepParams {
  uint64_t seed;
  float eps;
  float noise_scale;
  int32_t tag;
  int32_t mode;          // 0: gradient only, 1: SGLD update
  int32_t full;          // 1: every block of every sub-problem
  int32_t pad;
  int64_t sample_slot;   // -1: no sample this step
  float bc1, bc2;        // Adam bias corrections 1 / (1 - beta^t)
  uint64_t wait_ns;      // limit of every bounded device-side wait (grid barriers)
};

// Step state and tables.
struct StepView {
  int64_t M, N, S, NB, B, P, Q;
  int L_max;
  const StepParams* prm;
  // sub-problems (catalog x chain); a single catalog is one sub-problem
  int n_sub;
  const int32_t* blk_e0;          // NB + 1 first observation of each block
  const int32_t* blk_sub;         // NB
  const int32_t* ev_sub;          // M
  const int32_t* sub_blk_off;     // n_sub + 1
  const int32_t* sub_sel_full;    // n_sub + 1 prefix of blocks selected per step, full batch
  const int32_t* sub_sel_mb;      // n_sub + 1 prefix of blocks selected per step, minibatch
  const int32_t* sub_nobs;        // n_sub observations
  const int32_t* sub_nev;         // n_sub events
  const int32_t* sub_chain;       // n_sub Philox counter word 1
  const int32_t* sub_catalog;     // n_sub Philox counter word 2
  int32_t* sub_nsel;              // n_sub observations in this step's minibatch
  float4* sub_cen;                // n_sub centroid of the current state offset
  int n_chunks;
  const int32_t* chunk_ev0;       // n_chunks + 1 event chunks for the centroid sums
  const int32_t* sub_chunk_off;   // n_sub + 1
  float4* cen_chunk;              // n_chunks
  const float4* th0_hi;
  const float4* th0_lo;
  const double* th0_d;        // M x 4 theta_0 in FP64 (read-back only)
  const int32_t* ev_out;      // M: caller's event index (global) of each internal event
  float4* dth;
  const int32_t* ev_caller;   // caller's index of each (internal) event: the noise counter
  const float4* sta_hi;
  const float4* sta_lo;
  const int32_t* pair_ev;
  const int32_t* pair_st;
  const int32_t* pair_off;
  const uint32_t* obs_l;
  const float* obs_dt;
  const float* obs_sw;
  const int32_t* blk_node_off;
  const int32_t* node_pair;
  const uint16_t* node_he;
  const uint16_t* blk_he;
  const int32_t* inc_off;
  const int32_t* inc_q;
  const int32_t* inc_b;
  // per-step scratch
  int32_t* sel;
  int32_t* blk_stamp;
  int32_t* owner_q;
  int32_t* next_q;   // the pair's next selected occurrence, -1 after the last
  uint8_t* multi;
  int32_t* loc2u;
  int32_t* blk_owner_cnt;
  int32_t* blk_owner_off;
  int32_t* uniq_pair;
  int32_t* uniq_q;
  float2* T2;
  float4* J;
  float* r_obs;
  float* q_obs;
  float* part_a;     // per-occurrence partials (multi nodes): hi part
  float* part_b;     //   degree partials
  float* part_c;     //   lo part
  float* rhs;        // u = B^T r (hi)
  float* rhs_lo;     //           (lo)
  float* diag;       // lambda + diag(B^T B)
  float* z;          // solution (hi)
  float* z_lo;       //          (lo)
  uint8_t* umulti;  // per unique pair: 1 if it has occurrences in several selected blocks
  float* s_u;
  float4* gp;
  int32_t* pstamp;
  int32_t* estamp;
  float4* grad;
  int32_t* counters;
  double* dblk;      // FP64 sum r^2 per selected block (NB)
  double* dred;      // FP64 diagnostics partials, 4 x kMaxGrid
  double* dout;      // FP64 results: [0] loglik (scaled), [1] logprior, [2] logcen, [3] logpost
  // pieces of every block (k_whiten.cu, k_solve.cu; null without whitening)
  const int32_t* blk_piece_off;   // NB + 1
  const uint16_t* node_piece;     // Q: piece of a local node, numbered within its block
  const uint16_t* node_ppos;      // Q: position of a local node inside its piece
  const int32_t* piece_node_off;  // G + 1
  const uint16_t* piece_nodes;    // Q: block-local index of each piece member
  const int32_t* mem_rp;          // Q + 1: edges of each member (piece_nodes order)
  const uint16_t* edge_pos;       // 2N: position of the other end inside the piece
  const float* edge_sw;           // 2N: sqrt w of the edge
  const int64_t* piece_inv_off;   // G + 1 (null when the inverses were not built)
  const float* piece_inv;         // (lambda I + B^T B)^-1 of every piece, n x n each
  // components of the step
  const int32_t* node_mem;        // Q: member (piece_nodes order) of a local node
  int32_t* owner_b;               // Q: block of the owner occurrence
  int32_t* plab;                  // G: piece labels
  int32_t* prow;                  // G: owner occurrences of the piece
  uint8_t* pmulti;                // G: the piece has a node shared with another selected block
  int32_t* pcount;                // G: pieces of the component, at its root piece
  int32_t* urows;                 // G: rows of the component, at its root piece
  int32_t* unit_of;               // G: unit of a root piece
  int32_t *unit_off, *unit_np, *unit_fill, *unit_rows;   // G: per unit: piece list, pieces, fill cursor, rows
  int32_t* unit_slot;             // G: multi-CTA units: first row slot
  int4* msync;                    // 2 x kMaxGrid: barrier words of the multi-CTA class
  int32_t *unit_pieces, *unit_pblk, *unit_prow;   // G: piece lists: id, block, rows
  int32_t* unit_pbase;            // G: multi-CTA units: rows before the piece in its sorted run
  int32_t* unit_first;            // G: the same in the unit (pcount's memory, done with when units are listed)
  int32_t* cls_list;              // kLists x cls_cap: units of each size class
  int64_t cls_cap;
  int32_t* clean_list;            // G: pieces of the step solved with their inverse
  int32_t* clean_blk;             // G: their blocks
  int32_t* wfast;                 // [kWSlots + 64] counters and cursors, then the labelling rounds' flags
  int32_t* rowof;                 // P: row of a unique pair inside its component
  int32_t* mrow;                  // Q: the same per member occurrence
  float2* ent;                    // pool_entries: matrix entries (sqrt w, column) by slice, padding included
  // row slots of the multi-CTA class
  int32_t *rs_u, *rs_m, *rs_q, *rs_len;
  int4* rs_slice;                 // per slice: where its entries are
  float *rs_y, *rs_r, *rs_p, *rs_ap, *rs_dz, *rs_di, *rs_zh, *rs_zl;
  float4* samples;
  float4* mom1;      // Adam first moment (M), null otherwise
  float4* mom2;      // pSGLD / Adam second moment (M), null for SGLD
  int64_t sample_cap;
  // constants
  float lam;        // sigma^2 / kappa^2
  float inv_s2;     // 1 / sigma^2
  int whiten;       // kappa > 0 and the whitened loss
  int loss;         // SPIDER_LOSS_*
  int update;       // SPIDER_UPDATE_*
  float beta1, beta2, upd_eps;
  float4 inv_sig_e2;   // 1 / sigma_e^2
  float4 inv_sig_c2;   // 1 / sigma_c^2
  int cen_grid;     // CTAs of the event kernel
};

constexpr int kMaxGrid = 4096;
// size classes of the components solved by conjugate gradients: one warp, CTAs of
// 8, 16 and 32 warps, several CTAs; the late list holds pieces whose stored
// inverse did not converge
enum : int {
  kClsWarp = 0, kClsSmall = 1, kClsMid = 2, kClsCta = 3, kClsMulti = 4, kClasses = 5, kClsLate = 5, kLists = 6
};
constexpr int kWarpRows = 64, kSmallRows = 256, kMidRows = 512, kCtaRows = 1024;
constexpr int kWarpPieces = 32, kSmallPieces = 256, kMidPieces = 512, kCtaPieces = 1024;
// Lines between the classes: the rows that 1 warp (two per lane), 8, 16 and 32
// warps (one per lane) hold in registers, and the pieces whose tables fit beside
// them in shared memory.
__host__ __device__ constexpr int solve_class(int rows, int pieces) {
  return rows <= kWarpRows && pieces <= kWarpPieces     ? kClsWarp
         : rows <= kSmallRows && pieces <= kSmallPieces ? kClsSmall
         : rows <= kMidRows && pieces <= kMidPieces     ? kClsMid
         : rows <= kCtaRows && pieces <= kCtaPieces     ? kClsCta
                                                        : kClsMulti;
}
// wfast[] slots
enum : int {
  kWUnits = 0,      // components solved by conjugate gradients
  kWPieces = 1,     // their pieces
  kWGeneral = 2,    // 1: a component needed several CTAs, or a stored inverse did not converge
  kWClean = 3,      // pieces solved with their stored inverse
  kWCursorC = 4,    // their work cursor
  kWRowSlots = 5,   // row slots taken by the multi-CTA class
  kWEntries = 6,    // grains taken from the pool of entries
  kWClass0 = 8,     // units per class list
  kWCursor0 = 16,   // work cursors of the class lists
  kWSlots = 24
};
constexpr int kCenChunk = 4096;   // events per centroid partial sum

}  // namespace spider
