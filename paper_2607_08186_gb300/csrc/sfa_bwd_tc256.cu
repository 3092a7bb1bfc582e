// Stream-Factorized Attention backward (main pass) on the sm_103a tensor cores,
// head dim 256 (the 80B configuration's heads, Table 6).
//
// The gradient is the one of the head-dim-128 kernel (derivative of the forward of
// Eq. 4 / Fig. 2, which the paper trains through, Sec. 3.1); the plan differs because
// at head dim 256 dK and dV of one 128-row key tile alone would fill the 512 TMEM
// columns.  Each gradient therefore has its own work items, in one launch:
//   DV  key rows stationary:   S^T = K Q^T, P^T;                  dV += P^T dO
//   DK  key rows stationary:   S^T = K Q^T, dP^T = V dO^T, dS^T;  dK += dS^T Q
//   DQ  query rows stationary: S = Q K^T,   dP = dO V^T,   dS;    dQ += dS K
// S is computed three times and dP twice (8 GEMMs for 5 algorithmic ones), but every
// gradient is accumulated in TMEM over its whole loop and leaves once: no fp32 dQ
// accumulator in HBM, no reduce-adds, no shared-memory copy of dS.
//
// What bounds it: the tensor pipe.  A 128 x 128 x 16 MMA with both operands in shared
// memory reads 8 KB there in its 64 cycles, all of the SM's 128 B per clock, before any
// TMA write; so a pair of CTAs works on 256 stationary rows (cta_group::2, M = 256):
// each CTA holds its own 128 rows of A but only half of every B tile, 6 KB per 64
// cycles, and the pair loads each streamed tile once.  Per 128 streamed rows a CTA's
// shared memory moves 320 KB (2500 cycles) under 3072 cycles of MMA (DV: 192 KB under
// 2048).
// Measured, 80B-class WITHIN layer (B=1, L=4096, n=4, 24 over 2 heads; fwd + bwd): 4.16 ms
// with the fused form before (one CTA per key tile and head-dim half, S and dP computed
// by both halves, dQ added into an fp32 accumulator by TMA reduce: 3.34 ms of it, about
// 4900 cycles per 128 x 64 tile against 3250 of its shared-memory traffic), 2.85 ms with
// this one (2.1 ms); final-stream CROSS layer of the same heads 3.84 -> 2.49 ms.
// A step takes 2110 (DV), 3100 (DQ) and 3590 (DK) cycles.  With the ring in half tiles, so
// two waits and two commits per operand in the issuer, it was 2480, 3110 and 4110: a wait
// takes about 100 cycles, 215 right after a commit, and the few MMAs queued ahead do not
// cover several in a row (2.76 -> 2.66 ms, the forward included).  What is left in DK is the
// latency of its Q and dO tiles, of which the ring holds one step (3190 with every load of the same
// tile), and the row terms' loads.  Streaming the query tiles of all heads from the last
// tile down, so that the CTAs of a group share them in L2, gained nothing (0.97 to 1.0x).
//
// A pair's work item (cluster of two CTAs, 320 threads each, one CTA per SM):
//   A1, A2   stationary operands, 128 rows x 256 per CTA (DV: A1 only), loaded once
//   ring     streamed operands in 32 KB slots, in the order the issuer consumes them.  As
//            B of S and dP (K-major, N = 128) CTA r holds streamed rows [64r, 64r+64); as
//            B of the output GEMM (MN-major, N = 256) head-dim columns [128r, 128r+128).
//   TMEM     output in columns 256..511; DQ, DK: S in 0..127, dP in 128..255 (dS packed
//            bf16 over it, each 64-column half at the start of its own columns); DV: S
//            double-buffered in 0..255 (P^T packed over its buffer likewise).
//   issue    DQ, DK: S(0) dP(0) S(1), then per step t: out(t) dP(t+1) S(t+2).  The
//            softmax takes S(t+1) into registers while out(t) and dP(t+1) run and dP(t+1)
//            while S(t+2) runs, so the pipe does not wait for it.
//            DV: S(0), then per step t: S(t+1) out(t).
// Roles per CTA: warp 0 TMA producer; warp 1 MMA issuer (the pair's first CTA only: the
// whole warp runs the loop, one elected lane issues) and TMEM owner; warps 2..9 softmax, two
// threads per stationary row (TMEM lane), each half of the streamed columns.  A full barrier
// lives in the first CTA and counts both CTAs' bytes; commits are multicast to both CTAs.
// DQ's two 128-row tiles are the same rows of two heads of one K/V group where the group
// has an even number of heads (same key range), else consecutive tiles of one head; DK's
// and DV's are consecutive key tiles.
// Order of the items: DK (three GEMMs per step) and DV, key tiles with the most query
// tiles first, then DQ, whose items are short and fill the tail.  When there are too few
// key items to balance the SMs, each takes only a chunk of the group's query heads
// (head_chunks below), writing fp32 partial sums that dkv_finalize_kernel adds in chunk
// order: the same bits on every run, as for every output of this kernel.
// Every mbarrier wait is bounded; copies still in flight when a wait gives up were issued
// a whole timeout (about a second) earlier.
#include "tc_common.cuh"

namespace hdsfa {

typedef __nv_bfloat16 bf16;

namespace tcbwd256 {
constexpr int BM = 128, BN = 128, DH = 256, NTHREADS = 320;
constexpr int PR = 64, PC = 128;               // rows of a TMA box; head-dim columns of a CTA's output B half
constexpr int HB = 64;                         // streamed columns of one softmax thread
constexpr int SLOT = PR * DH;                  // a ring slot: half of a streamed tile, four [64 rows][64] swizzle blocks
constexpr int NSLOT = 3, NSLOT_DV = 5;         // DV streams through A2's space as well
constexpr uint32_t COL_OUT = 256, COL_D = 128;  // output; dP (DV: the second S buffer)
enum Kind { kDK = 0, kDV = 1, kDQ = 2 };

struct Smem {
  bf16 a1[BM * DH];           // four [128 rows][64] swizzle blocks
  bf16 a2[BM * DH];           // DV: ring slots 0 and 1
  bf16 ring[NSLOT][SLOT];
  float nlse2[2][BN];         // DK, DV: -lse*log2(e) of the streamed query tile, by step parity (loaded by bulk copy)
  float ndelta[2][BN];        // DK: -delta of it
  uint64_t full[NSLOT_DV], empty[NSLOT_DV], a1_full, a2_full;
  uint64_t s_full[2], s_empty, dp_full, p_full[2], out_done, term_full[2], term_empty[2];
  uint32_t tmem_base;
  int abort;
};
// The layout needs 1024-byte alignment; the kernel checks the actual pad on entry.
constexpr int kSmemBytes = sizeof(Smem) + 1024 < 232448 ? (int)sizeof(Smem) + 1024 : 232448;
static_assert(sizeof(Smem) <= 232448, "head-dim-256 backward shared memory exceeds 227 KB");

struct Params {
  CUtensorMap tm_q, tm_do, tm_k, tm_v;  // boxes of 64 rows x 64 columns
  const float* lse2;   // -lse*log2(e), [B][Hq][ns][Lvp]
  const float* delta;  // -delta, the same layout
  bf16* dq;            // dQ (scaled), or null: dq_acc
  float* dq_acc;       // unscaled fp32 dQ, added to what is there, when dq is null
  bf16* dk;
  bf16* dv;
  float* dkv;   // head chunks > 1: fp32 partial sums [chunks][2][B][q_ns][Lv][Hkv][DH] (dV, dK)
  int hchunks;  // query-head chunks per K/V head
  int grp, hper;  // query heads per K/V head, and per chunk
  int nkv;      // DK items (= DV items); DQ items follow
  int head_pairs;
  // DK / DV item -> key-tile pair, chunk, batch, K/V head; DQ item -> rank, batch, head; group
  FastDiv d_tile, d_hc, d_kns, d_rank, d_hns, d_ns, d_grp;
  SfaGeom g;
  float scale, scale_log2;
  int32_t* status;
};

// One work item: its kind, stationary rows and the streamed steps.
struct Item {
  int kind;
  int b, s, sk, kvh, hc;
  int row0, head;    // this CTA's first stationary row; its query head (DQ)
  int h_base, grp;   // DK, DV: first query head and number of heads of the chunk
  int lo, nst;       // first streamed tile and tiles per head
  int T;             // steps: DQ nst, DK / DV grp * nst
};

HD_DEVINLINE Item make_item(const Params& P, int idx, int rank) {
  const SfaGeom& G = P.g;
  Item it;
  it.kind = idx < P.nkv ? kDK : idx < 2 * P.nkv ? kDV : kDQ;
  it.hc = 0;
  if (it.kind != kDQ) {
    if (it.kind == kDV) idx -= P.nkv;
    const int HC = P.hchunks, per_tile = HC * G.Hkv * G.q_ns * G.B;
    const int j = fast_div(idx, P.d_tile), rem = idx - j * per_tile;  // key-tile pair slowest
    const int hsb = fast_div(rem, P.d_hc);
    it.hc = rem - hsb * HC;
    it.b = fast_div(hsb, P.d_kns);
    const int hs = hsb - it.b * G.Hkv * G.q_ns;
    it.kvh = fast_div(hs, P.d_ns);
    it.s = hs - it.kvh * G.q_ns;
    const int grp_all = P.grp, hper = P.hper;
    it.grp = min(hper, grp_all - it.hc * hper);
    it.h_base = it.kvh * grp_all + it.hc * hper;
    it.head = it.h_base;
    const int n0 = j * 2 * BM;
    it.row0 = n0 + rank * BM;
    // query rows that can see a key of the pair: key row r*qstep + qoff >= n0, and under
    // a window r*qstep + qoff < n0 + 2*BM - 1 + window
    it.lo = (n0 <= G.qoff ? 0 : (n0 - G.qoff + G.qstep - 1) / G.qstep) / BN;
    int hi = (G.Lq - 1) / BN;
    if (G.window > 0) hi = min(hi, ((n0 + 2 * BM - 2 + G.window - G.qoff) / G.qstep) / BN);
    it.nst = hi - it.lo + 1;
    it.T = it.nst > 0 ? it.grp * it.nst : 0;
  } else {
    idx -= 2 * P.nkv;
    const int hp = P.head_pairs, rows = hp ? BM : 2 * BM, nh = hp ? G.Hq / 2 : G.Hq;
    const int ntile = (G.Lq + rows - 1) / rows, per_rank = nh * G.q_ns * G.B;
    const int tr = fast_div(idx, P.d_rank), mt = ntile - 1 - tr, hsb = idx - tr * per_rank;
    it.b = fast_div(hsb, P.d_hns);
    const int hs = hsb - it.b * nh * G.q_ns, hx = fast_div(hs, P.d_ns);
    it.s = hs - hx * G.q_ns;
    it.head = hp ? 2 * hx + rank : hx;
    it.kvh = fast_div(it.head, P.d_grp);
    it.h_base = it.head;
    it.grp = 1;
    const int m0 = mt * rows;
    it.row0 = hp ? m0 : m0 + rank * BM;
    // key tiles some row of the pair sees
    const int rq_first = m0 * G.qstep + G.qoff, rq_last = (min(m0 + rows, G.Lq) - 1) * G.qstep + G.qoff;
    it.lo = G.window > 0 ? max(0, rq_first - G.window + 1) / BN : 0;
    it.nst = min(rq_last, G.Lv - 1) / BN - it.lo + 1;
    it.T = it.nst;
  }
  it.sk = it.s + G.kv_s0;
  return it;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTHREADS, 1) bwd256_kernel(const __grid_constant__ Params P) {
  extern __shared__ uint8_t smem_raw[];
  {
    uint32_t dyn;
    asm("mov.u32 %0, %%dynamic_smem_size;\n" : "=r"(dyn));
    const uintptr_t base = reinterpret_cast<uintptr_t>(smem_raw);
    if (((base + 1023) & ~uintptr_t(1023)) - base + sizeof(Smem) > dyn) {  // uniform: nothing touched yet
      if (threadIdx.x == 0) set_status(P.status, HD_DEVBIT_TIMEOUT);
      return;
    }
  }
  Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const SfaGeom& G = P.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)(blockIdx.x & 1);  // = %cluster_ctarank
  attn_dep_wait(1);
  const Item it = make_item(P, (int)(blockIdx.x >> 1), rank);
  const int kind = it.kind, T = it.T;
  const size_t half = (size_t)G.B * G.q_ns * G.Lv * G.Hkv * DH;  // elements of a slice half
  if (T <= 0) {  // no query sees these key tiles (the same for both CTAs): their rows are zero
    for (int i = threadIdx.x; i < BM * (DH / 8); i += NTHREADS) {
      const int kr = it.row0 + i / (DH / 8), c = i % (DH / 8);
      if (kr >= G.Lv) continue;
      if (P.hchunks > 1) {
        float* w = P.dkv + (2 * it.hc + (kind == kDK)) * half +
                   ((((long long)it.b * G.q_ns + it.s) * G.Lv + kr) * G.Hkv + it.kvh) * DH + c * 8;
        reinterpret_cast<float4*>(w)[0] = make_float4(0.f, 0.f, 0.f, 0.f);
        reinterpret_cast<float4*>(w)[1] = make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
        bf16* w = (kind == kDK ? P.dk : P.dv) +
                  (((long long)it.b * G.nL + (long long)kr * G.rs + it.sk) * G.Hkv + it.kvh) * DH + c * 8;
        *reinterpret_cast<uint4*>(w) = make_uint4(0, 0, 0, 0);
      }
    }
    return;
  }

  if (threadIdx.x == 0) {
    for (int i = 0; i < NSLOT_DV; ++i) {
      mbar_init(&sm.full[i], 1);
      mbar_init(&sm.empty[i], 1);
    }
    mbar_init(&sm.a1_full, 1);
    mbar_init(&sm.a2_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sm.s_full[i], 1);
      mbar_init(&sm.term_full[i], 1);
      mbar_init(&sm.term_empty[i], 8);  // the CTA's softmax warps
      mbar_init(&sm.p_full[i], 16);  // one arrival per softmax warp of the pair
    }
    mbar_init(&sm.s_empty, 16);
    mbar_init(&sm.dp_full, 1);
    mbar_init(&sm.out_done, 1);
    sm.abort = 0;
    fence_mbar_init();
  }
  __syncwarp();
  cluster_arrive();  // the barriers of this CTA are initialised
  if (warp == 1) {
    tma_prefetch(&P.tm_q);
    tma_prefetch(&P.tm_do);
    tma_prefetch(&P.tm_k);
    tma_prefetch(&P.tm_v);
    tmem_alloc_pair(&sm.tmem_base, 512);
    tc_fence_before();
  }
  cluster_wait();
  uint32_t tmem = 0;
  if (warp != 0) {  // the producer does not wait for the TMEM allocation
    named_bar_sync(1, NTHREADS - 32);
    tc_fence_after();
    tmem = sm.tmem_base;
  }
  volatile int* abort = &sm.abort;
  const int nslot = kind == kDV ? NSLOT_DV : NSLOT;
  bf16* const ring0 = kind == kDV ? sm.a2 : sm.ring[0];  // a2 and ring are adjacent

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      const CUtensorMap *tA1 = kind == kDQ ? &P.tm_q : &P.tm_k, *tA2 = kind == kDQ ? &P.tm_do : &P.tm_v;
      const CUtensorMap* tB1 = kind == kDQ ? &P.tm_k : &P.tm_q;
      const CUtensorMap* tB2 = kind == kDQ ? &P.tm_v : &P.tm_do;
      const CUtensorMap* tB3 = kind == kDV ? &P.tm_do : tB1;
      const int ahead = kind == kDQ ? it.head : it.kvh, astr = kind == kDQ ? it.s : it.sk;
      const int bstr = kind == kDQ ? it.sk : it.s;
      auto load_a = [&](bf16* dst, const CUtensorMap* tm, uint64_t* bar) {
        if (rank == 0) mbar_arrive_expect_tx(bar, 2 * BM * DH * 2);
        const uint32_t lb = lead_addr(bar);
        for (int c = 0; c < DH / 64; ++c)
          for (int r = 0; r < BM / PR; ++r)
            tma_load_pair(dst + c * BM * 64 + r * PR * 64, tm, lb, c * 64, ahead, astr, it.row0 + r * PR, it.b);
      };
      int terms_issued = 0;
      int slot = 0, ph = 1;  // empty-barrier phase: the first lap does not wait
      bool ok = true;
      // a unit.  as_n: B of S / dP (this CTA's 64 rows, the whole head dim, block c its
      // columns 64c); else B of the output GEMM (all 128 rows, this CTA's head-dim half,
      // blocks 2p, 2p + 1 the two 64-column blocks of rows 64p)
      auto load_unit = [&](const CUtensorMap* tm, int t, bool as_n) {
        const int hd = kind == kDQ ? it.kvh : it.h_base + t / it.nst;
        const int r0 = (it.lo + (kind == kDQ ? t : t % it.nst)) * BN;
        if (!mbar_wait(&sm.empty[slot], ph, abort, P.status)) {
          ok = false;
          return;
        }
        if (rank == 0) mbar_arrive_expect_tx(&sm.full[slot], 2 * SLOT * 2);
        const uint32_t lb = lead_addr(&sm.full[slot]);
        bf16* dst = ring0 + slot * SLOT;
        for (int c = 0; c < 4; ++c) {
          const int row = as_n ? r0 + rank * PR : r0 + (c >> 1) * PR;
          const int col = as_n ? c * 64 : rank * PC + (c & 1) * 64;
          tma_load_pair(dst + c * PR * 64, tm, lb, col, hd, bstr, row, it.b);
        }
        if (++slot == nslot) {
          slot = 0;
          ph ^= 1;
        }
      };
      // the row terms of step t (DK, DV), into the buffer that step t-2 has read
      auto load_terms = [&](int t) {
        if (t >= 2 && !mbar_wait(&sm.term_empty[t & 1], ((t >> 1) - 1) & 1, abort, P.status)) {
          ok = false;
          return;
        }
        const long long off = (((long long)it.b * G.Hq + it.h_base + t / it.nst) * G.q_ns + it.s) *
                                  row_terms_pitch(G.Lq) + (long long)(it.lo + t % it.nst) * BN;
        mbar_arrive_expect_tx(&sm.term_full[t & 1], kind == kDK ? 2 * BN * 4 : BN * 4);
        bulk_load(sm.nlse2[t & 1], P.lse2 + off, BN * 4, &sm.term_full[t & 1]);
        if (kind == kDK) bulk_load(sm.ndelta[t & 1], P.delta + off, BN * 4, &sm.term_full[t & 1]);
        terms_issued = t + 1;
      };
      load_a(sm.a1, tA1, &sm.a1_full);
      load_unit(tB1, 0, true);
      if (kind != kDQ) load_terms(0);
      if (kind == kDV) {
        for (int t = 0; ok && t < T; ++t) {
          if (t + 1 < T) load_unit(tB1, t + 1, true);
          if (ok && t + 1 < T) load_terms(t + 1);
          if (ok) load_unit(tB3, t, false);
        }
      } else {
        load_a(sm.a2, tA2, &sm.a2_full);
        load_unit(tB2, 0, true);
        if (ok && T > 1) load_unit(tB1, 1, true);
        for (int t = 0; ok && t < T; ++t) {
          load_unit(tB3, t, false);
          if (ok && kind == kDK && t + 1 < T) load_terms(t + 1);
          if (ok && t + 1 < T) load_unit(tB2, t + 1, true);
          if (ok && t + 2 < T) load_unit(tB1, t + 2, true);
        }
      }
      for (int t = max(0, terms_issued - 2); t < terms_issued; ++t) mbar_drain(&sm.term_full[t & 1], (t >> 1) & 1);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (first CTA)
    if (rank == 0) {
      constexpr uint32_t idS = idesc_bf16(2 * BM, BN, 0, 0);  // S, dP: both operands K-major
      constexpr uint32_t idO = idesc_bf16(2 * BM, DH, 0, 1);  // output: A in TMEM, B MN-major
      // descriptors encoded once; a block, slot or k-step adds its byte offset / 16
      const uint64_t a1d = sdesc_sw128(smem_u32(sm.a1), 16, 1024), a2d = sdesc_sw128(smem_u32(sm.a2), 16, 1024);
      const uint64_t bK = sdesc_sw128(smem_u32(ring0), 16, 1024);        // slots K-major
      const uint64_t bM = sdesc_sw128(smem_u32(ring0), PR * 128, 1024);  // slots MN-major
      int slot = 0, ph = 0;
      auto wait_w = [&](uint64_t* bar, int par) -> bool {
        if (!__all_sync(0xffffffffu, mbar_wait(bar, par & 1, abort, P.status))) return false;
        tc_fence_after();
        return true;
      };
      auto next_slot = [&]() {
        if (++slot == nslot) {
          slot = 0;
          ph ^= 1;
        }
      };
      // D[256 x 128] = A B^T over the head dim, then a signal that it is complete
      auto gemm_n = [&](uint32_t col, uint64_t ad, uint64_t* done) -> bool {
        if (!wait_w(&sm.full[slot], ph)) return false;
        const uint64_t bd = bK + (uint64_t)(slot * (SLOT * 2 / 16));
#pragma unroll
        for (int kk = 0; kk < DH / 16; ++kk)
          mma2_ss(tmem + col, ad + (uint64_t)((kk >> 2) * (BM * 128 / 16) + (kk & 3) * 2),
                  bd + (uint64_t)((kk >> 2) * (PR * 128 / 16) + (kk & 3) * 2), idS, kk > 0 ? 1u : 0u);
        commit2(done);
        commit2(&sm.empty[slot]);
        next_slot();
        return true;
      };
      // out[256 x 256] += A[tmem] B over the 128 streamed rows.  B is waited for before A
      // (each wait costs about 100 cycles of a chain that ends with A).
      auto gemm_out = [&](uint32_t acol, uint64_t* a_full, int a_par, bool acc0) -> bool {
        if (!wait_w(&sm.full[slot], ph) || !wait_w(a_full, a_par)) return false;
        const uint64_t bd = bM + (uint64_t)(slot * (SLOT * 2 / 16));
#pragma unroll
        for (int kk = 0; kk < BN / 16; ++kk)
          // P / dS: each 64-column half packed at the start of its own columns
          mma2_ts(tmem + COL_OUT, tmem + acol + (kk >> 2) * HB + (kk & 3) * 8,
                  bd + (uint64_t)((kk >> 2) * (PR * PC * 2 / 16) + (kk & 3) * 16 * 128 / 16), idO,
                  (acc0 || kk > 0) ? 1u : 0u);
        commit2(&sm.empty[slot]);
        next_slot();
        return true;
      };
      bool ok = wait_w(&sm.a1_full, 0) && gemm_n(0, a1d, &sm.s_full[0]);
      if (kind == kDV) {
        for (int t = 0; ok && t < T; ++t) {
          // S(t+1) over P^T(t-1), which out(t-1), issued before, has read
          if (t + 1 < T) ok = gemm_n(((t + 1) & 1) * COL_D, a1d, &sm.s_full[(t + 1) & 1]);
          ok = ok && gemm_out((t & 1) * COL_D, &sm.p_full[t & 1], t >> 1, t > 0);
        }
      } else {
        ok = ok && wait_w(&sm.a2_full, 0) && gemm_n(COL_D, a2d, &sm.dp_full);
        if (ok && T > 1) ok = wait_w(&sm.s_empty, 0) && gemm_n(0, a1d, &sm.s_full[0]);
        for (int t = 0; ok && t < T; ++t) {
          ok = gemm_out(COL_D, &sm.p_full[0], t, t > 0);
          // dP(t+1) over dS(t), which out(t), issued before, has read
          if (ok && t + 1 < T) ok = gemm_n(COL_D, a2d, &sm.dp_full);
          if (ok && t + 2 < T) ok = wait_w(&sm.s_empty, t + 1) && gemm_n(0, a1d, &sm.s_full[0]);
        }
      }
      // every MMA issued above completes before TMEM / smem are released
      commit2(&sm.out_done);
      mbar_drain(&sm.out_done, 0);
    }
  } else {
    // ------------------------------------------------------------ softmax / epilogue
    // Two threads per stationary row (TMEM lane), each half hc of the 128 streamed columns.
    const int q4 = warp & 3, hc = (warp - 2) >> 2;
    const int r = it.row0 + q4 * 32 + lane;  // stationary row: query row (DQ) or key row (DK, DV)
    const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16) + HB * hc;  // this thread's half
    const float c2 = P.scale_log2;
    const uint64_t c2x2 = f2pack(c2, c2);
    const uint32_t lead_s_empty = lead_addr(&sm.s_empty);
    const uint32_t lead_p[2] = {lead_addr(&sm.p_full[0]), lead_addr(&sm.p_full[1])};
    auto publish = [&](uint32_t bar) {  // this warp's TMEM accesses are done: tell the issuer
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_lead(bar);
    };
    auto load_half = [&](uint32_t tcol, float* x) {
#pragma unroll
      for (int c = 0; c < HB / 32; ++c) tmem_ld32(tcol + c * 32, reinterpret_cast<uint32_t*>(x) + c * 32);
      tmem_ld_wait();
    };
    // dS = P (dP - delta), packed bf16 over the first half of this thread's dP columns,
    // all of them read before (the loads run one 16-column chunk ahead)
    auto d_half = [&](const float* x, auto nd) {
      uint32_t d[2][16];
      tmem_ld16(tl + COL_D, d[0]);
#pragma unroll
      for (int c = 0; c < HB / 16; ++c) {
        uint32_t* dc = d[c & 1];
        tmem_ld_wait();
        if (c + 1 < HB / 16) tmem_ld16(tl + COL_D + (c + 1) * 16, d[(c + 1) & 1]);
        uint32_t pk[8];
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
          float y0, y1;
          f2unpack(fmul2(fadd2(f2pack(__uint_as_float(dc[e]), __uint_as_float(dc[e + 1])), nd(c * 8 + (e >> 1))),
                         f2pack(x[c * 16 + e], x[c * 16 + e + 1])),
                   y0, y1);
          pk[e >> 1] = cvt_bf16x2(y0, y1);
        }
        tmem_st8(tl + COL_D + c * 8, pk);
      }
      tmem_st_wait();
    };
    bool ok = true;

    if (kind == kDQ) {
      const int rq = r * G.qstep + G.qoff;             // key row of this query
      const int rq0 = it.row0 * G.qstep + G.qoff;      // ... of the tile's first query
      const int rq1 = (it.row0 + BM - 1) * G.qstep + G.qoff;
      float nl = -INFINITY, nd = 0.f;  // rows past Lq: P = 0
      if (r < G.Lq) {
        const long long off = (((long long)it.b * G.Hq + it.head) * G.q_ns + it.s) * row_terms_pitch(G.Lq) + r;
        nl = P.lse2[off];
        nd = P.delta[off];
      }
      const uint64_t nl2 = f2pack(nl, nl), nd2 = f2pack(nd, nd);
      for (int t = 0; t < T; ++t) {
        const int c0 = (it.lo + t) * BN + HB * hc;  // first key of this half
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.s_full[0], t & 1, abort, P.status))) {
          ok = false;
          break;
        }
        tc_fence_after();
        float x[HB];
        load_half(tl, x);
        publish(lead_s_empty);
#pragma unroll
        for (int e = 0; e < HB; e += 2) {
          float a0, a1;
          f2unpack(ffma2(f2pack(x[e], x[e + 1]), c2x2, nl2), a0, a1);
          x[e] = ex2_approx(a0);
          x[e + 1] = ex2_approx(a1);
        }
        // halves with a key past the first query's key row, at or below the last query's
        // window edge, or past the end (keys there are zero, but exp2(-lse2) may overflow)
        if (c0 + HB - 1 > rq0 || (G.window > 0 && c0 <= rq1 - G.window) || c0 + HB > G.Lv) {
          const int hi = min(rq, G.Lv - 1) - c0, lo = G.window > 0 ? rq - G.window + 1 - c0 : 0;
#pragma unroll
          for (int e = 0; e < HB; ++e)
            if (e > hi || e < lo) x[e] = 0.f;
        }
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.dp_full, t & 1, abort, P.status))) {
          ok = false;
          break;
        }
        tc_fence_after();
        d_half(x, [&](int) { return nd2; });
        publish(lead_p[0]);
      }
    } else {
      // DK, DV: this thread's key row r.  The streamed tile's row terms come through shared
      // memory and are taken into registers before the MMA results they belong to are
      // waited for: a broadcast load queues behind the MMAs' operand reads.
      const int kr = r;
      // key row kr sees the queries q in [vis_lo, vis_hi): q*qstep + qoff >= kr (causal),
      // and for LOCAL q*qstep + qoff < kr + window.  Queries past Lq have -lse2 = -inf; a
      // key row past Lv is not stored.
      const int vis_lo = kr <= G.qoff ? 0 : (kr - G.qoff + G.qstep - 1) / G.qstep;
      int vis_hi = G.Lq;
      if (G.window > 0) {
        const int e = kr + G.window - G.qoff;  // q*qstep < e
        vis_hi = min(vis_hi, e <= 0 ? 0 : (e + G.qstep - 1) / G.qstep);
      }
      int qi = 0;  // query tile of the step within its head
      for (int t = 0; t < T; ++t) {
        const int qm = (it.lo + qi) * BN;
        if (++qi == it.nst) qi = 0;
        const int sb = kind == kDV ? (t & 1) : 0;
        const uint32_t tS = tl + sb * COL_D;
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.term_full[t & 1], (t >> 1) & 1, abort, P.status))) {
          ok = false;
          break;
        }
        ulonglong2 tm[HB / 4];
#pragma unroll
        for (int e = 0; e < HB / 4; ++e) tm[e] = reinterpret_cast<const ulonglong2*>(sm.nlse2[t & 1] + HB * hc)[e];
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.s_full[sb], (kind == kDV ? t >> 1 : t) & 1, abort, P.status))) {
          ok = false;
          break;
        }
        tc_fence_after();
        float x[HB];
        load_half(tS, x);
        if (kind == kDK) publish(lead_s_empty);
#pragma unroll
        for (int e = 0; e < HB; e += 2) {
          float a0, a1;
          f2unpack(ffma2(f2pack(x[e], x[e + 1]), c2x2, (e & 2) ? tm[e >> 2].y : tm[e >> 2].x), a0, a1);
          x[e] = ex2_approx(a0);
          x[e + 1] = ex2_approx(a1);
        }
        // the diagonal band and (LOCAL) tiles that reach the window edge of the first key
        if (qm * G.qstep + G.qoff < it.row0 + BM ||
            (G.window > 0 && (qm + BN - 1) * G.qstep + G.qoff - G.window >= it.row0)) {
          const int lo = vis_lo - qm - HB * hc, hi = vis_hi - qm - HB * hc;
#pragma unroll
          for (int e = 0; e < HB; ++e)
            if (e < lo || e >= hi) x[e] = 0.f;
        }
        if (kind == kDV) {
#pragma unroll
          for (int c = 0; c < HB / 32; ++c) {
            uint32_t pk[16];
#pragma unroll
            for (int e = 0; e < 32; e += 2) pk[e >> 1] = cvt_bf16x2(x[c * 32 + e], x[c * 32 + e + 1]);
            tmem_st16(tS + c * 16, pk);
          }
          tmem_st_wait();
        } else {
          const ulonglong2* nd4 = reinterpret_cast<const ulonglong2*>(sm.ndelta[t & 1] + HB * hc);
          ulonglong2 td[HB / 4];
#pragma unroll
          for (int e = 0; e < HB / 8; ++e) td[e] = nd4[e];
          if (!__all_sync(0xffffffffu, mbar_wait(&sm.dp_full, t & 1, abort, P.status))) {
            ok = false;
            break;
          }
          tc_fence_after();
          d_half(x, [&](int e2) {
            if (e2 < HB / 4 && !(e2 & 7)) {  // one chunk ahead of their use, in the registers the first half leaves
#pragma unroll
              for (int e = 0; e < 4; ++e) td[HB / 8 + (e2 >> 1) + e] = nd4[HB / 8 + (e2 >> 1) + e];
            }
            return (e2 & 1) ? td[e2 >> 1].y : td[e2 >> 1].x;
          });
        }
        publish(lead_p[sb]);
        if (lane == 0) mbar_arrive(&sm.term_empty[t & 1]);
      }
    }

    // epilogue: this thread's half (128 columns) of its row of the output
    if (ok && __all_sync(0xffffffffu, mbar_wait(&sm.out_done, 0, abort, P.status))) {
      tc_fence_after();
      const uint32_t to = tmem + ((uint32_t)(q4 * 32) << 16) + COL_OUT + PC * hc;
      const float mul = kind == kDV ? 1.f : P.scale;
      const bool f32_out = kind == kDQ ? P.dq == nullptr : P.hchunks > 1;
      const int nrow = kind == kDQ ? G.Lq : G.Lv;
      if (f32_out) {
        float* dst;
        float m = mul;
        if (kind == kDQ) {  // unscaled (sfa_bwd_finalize applies the scale) and added: one sum per call
          dst = P.dq_acc + (((long long)it.b * G.q_nL + (long long)r * G.q_rs + it.s) * G.Hq + it.head) * DH;
          m = 1.f;
        } else {
          dst = P.dkv + (2 * it.hc + (kind == kDK)) * half +
                ((((long long)it.b * G.q_ns + it.s) * G.Lv + r) * G.Hkv + it.kvh) * DH;
        }
        dst += PC * hc;
#pragma unroll 1
        for (int c = 0; c < PC / 32; ++c) {
          uint32_t o[32];
          tmem_ld32(to + c * 32, o);
          tmem_ld_wait();
          if (r < nrow) {
#pragma unroll
            for (int e = 0; e < 32; e += 4) {
              const float4 w = make_float4(__uint_as_float(o[e]) * m, __uint_as_float(o[e + 1]) * m,
                                           __uint_as_float(o[e + 2]) * m, __uint_as_float(o[e + 3]) * m);
              if (kind == kDQ)
                red_add4(dst + c * 32 + e, w.x, w.y, w.z, w.w);
              else
                *reinterpret_cast<float4*>(dst + c * 32 + e) = w;
            }
          }
        }
      } else {
        // rows leave through shared memory (A1 is no longer read): each thread writes its
        // half row as bf16, 16-byte units XOR-swizzled by the row, then every store
        // instruction of the warp writes 256-byte halves of two rows
        constexpr int UPR = DH * 2 / 16;  // 16-byte units per row
        uint8_t* stg = reinterpret_cast<uint8_t*>(sm.a1) + q4 * (32 * DH * 2);
#pragma unroll 2
        for (int c = 0; c < PC / 32; ++c) {
          uint32_t o[32];
          tmem_ld32(to + c * 32, o);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; e += 8) {
            uint4 w;
            w.x = cvt_bf16x2(__uint_as_float(o[e + 0]) * mul, __uint_as_float(o[e + 1]) * mul);
            w.y = cvt_bf16x2(__uint_as_float(o[e + 2]) * mul, __uint_as_float(o[e + 3]) * mul);
            w.z = cvt_bf16x2(__uint_as_float(o[e + 4]) * mul, __uint_as_float(o[e + 5]) * mul);
            w.w = cvt_bf16x2(__uint_as_float(o[e + 6]) * mul, __uint_as_float(o[e + 7]) * mul);
            const int u = hc * (UPR / 2) + c * 4 + e / 8;
            *reinterpret_cast<uint4*>(stg + lane * (DH * 2) + ((u ^ (lane & 7)) << 4)) = w;
          }
        }
        __syncwarp();
        bf16* base;
        long long rstride;  // elements between rows
        if (kind == kDQ) {
          base = P.dq + (((long long)it.b * G.q_nL + it.s) * G.Hq + it.head) * DH;
          rstride = (long long)G.q_rs * G.Hq * DH;
        } else {
          base = (kind == kDK ? P.dk : P.dv) + (((long long)it.b * G.nL + it.sk) * G.Hkv + it.kvh) * DH;
          rstride = (long long)G.rs * G.Hkv * DH;
        }
        const int r0 = it.row0 + q4 * 32, u = hc * (UPR / 2) + (lane & 15);
#pragma unroll 8
        for (int i = lane >> 4; i < 32; i += 2)
          if (r0 + i < nrow)
            *reinterpret_cast<uint4*>(base + (long long)(r0 + i) * rstride + u * 8) =
                *reinterpret_cast<const uint4*>(stg + i * (DH * 2) + ((u ^ (i & 7)) << 4));
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();  // neither CTA's barriers or TMEM are used any more
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
}
// Head chunks: dv / dk rows (bf16) from the chunks' fp32 partial sums, added in chunk
// order, 8 columns per thread.
__global__ void __launch_bounds__(256) dkv_finalize_kernel(const float* dkv, bf16* __restrict__ dk,
                                                           bf16* __restrict__ dv, SfaGeom g, int chunks) {
  attn_dep_wait(8);
  const long long n8 = (long long)g.B * g.q_ns * g.Lv * g.Hkv * (DH / 8);
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n8) return;
  const int c8 = (int)(i % (DH / 8));
  long long r = i / (DH / 8);
  const int kvh = (int)(r % g.Hkv);
  r /= g.Hkv;
  const int kr = (int)(r % g.Lv);
  r /= g.Lv;
  const int s = (int)(r % g.q_ns), b = (int)(r / g.q_ns);
  const long long orow = (((long long)b * g.nL + (long long)kr * g.rs + s + g.kv_s0) * g.Hkv + kvh) * DH + c8 * 8;
  const size_t half = (size_t)n8 * 8;
#pragma unroll
  for (int which = 0; which < 2; ++which) {
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
    for (int hc = 0; hc < chunks; ++hc) {
      const float4* src = reinterpret_cast<const float4*>(dkv + (2 * hc + which) * half + i * 8);
      const float4 a = src[0], e = src[1];
      x.x += a.x; x.y += a.y; x.z += a.z; x.w += a.w;
      y.x += e.x; y.y += e.y; y.z += e.z; y.w += e.w;
    }
    uint4 w;
    w.x = cvt_bf16x2(x.x, x.y);
    w.y = cvt_bf16x2(x.z, x.w);
    w.z = cvt_bf16x2(y.x, y.y);
    w.w = cvt_bf16x2(y.z, y.w);
    *reinterpret_cast<uint4*>((which ? dk : dv) + orow) = w;
  }
}

// DK / DV items of one chunk count.
static long long key_items(const SfaGeom& g) {
  return (long long)((g.Lv + 2 * BM - 1) / (2 * BM)) * g.Hkv * g.q_ns * g.B;
}

// Query-head chunks of the DK and DV items: the count with the least estimated time over
// the chip's 76 CTA pairs, as the larger of a pair's share of all items and the longest
// item (DK of the key pair with the most query tiles), plus the finalize pass where there
// are chunks.  In units of 1000 cycles, measured at L = 4096: a step of DK, DV and DQ 3.6,
// 2.1 and 3.1, an item's fixed part 10, the finalize pass 8 and its traffic (8 bytes
// written and read per element and chunk at about 3.4 KB per cycle).  `room`: slices of
// partial sums there is space for.  (One chunk too many costs little on long items, but
// three sequences of 98 positions, fwd + bwd: 63 us with 12 chunks, two waves of short items, 50 us with 4.)
static int head_chunks(const SfaGeom& g, long long room, long long ndq) {
  const int grp = g.Hq / g.Hkv;
  const long long items = key_items(g);
  constexpr int kPairs = kSmCount / 2;
  if (grp < 2 || room < 2 || items >= 2 * kPairs) return 1;
  // query tiles per head that each key pair streams (fewer than 2 * kPairs pairs)
  const int npair = (g.Lv + 2 * BM - 1) / (2 * BM);
  double sum = 0, most = 0;
  for (int j = 0; j < npair; ++j) {
    const int n0 = j * 2 * BM;
    const int lo = (n0 <= g.qoff ? 0 : (n0 - g.qoff + g.qstep - 1) / g.qstep) / BN;
    int hi = (g.Lq - 1) / BN;
    if (g.window > 0 && n0 + 2 * BM - 2 + g.window - g.qoff < (hi + 1) * BN * g.qstep)
      hi = (n0 + 2 * BM - 2 + g.window - g.qoff) / g.qstep / BN;
    const double nst = hi >= lo ? hi - lo + 1 : 0;
    sum += nst;
    most = nst > most ? nst : most;
  }
  const double per = (double)items / npair;  // items of one key pair
  // DQ: as many row-tile products as DK, two row tiles to an item
  const double dq = ndq * 10.0 + 3.1 * sum * per * grp;
  int best = 1;
  double best_cost = 0;
  for (int hs = 1; hs <= grp && hs <= room; ++hs) {
    const int hper = (grp + hs - 1) / hs;
    if ((grp + hper - 1) / hper != hs) continue;  // another count gives the same chunks
    const double total = dq + 2.0 * items * hs * 10.0 + 5.7 * sum * per * grp;
    const double longest = 10.0 + 3.6 * hper * most;
    const double share = total / kPairs;
    double cost = share > longest ? share : longest;
    if (hs > 1) cost += 8.0 + 16.0 * hs * g.B * g.q_ns * (double)g.Lv * g.Hkv * DH / 3.4e6;
    if (best_cost == 0 || cost < best_cost) {
      best = hs;
      best_cost = cost;
    }
  }
  return best;
}
}  // namespace tcbwd256

// dq_out: bf16 dQ (scaled); null: unscaled fp32 dQ added into dq_ws.  With dq_out the space of
// dq_ws is free and holds the chunks' partial sums when it is larger than dkv_ws.
cudaError_t launch_sfa_bwd_main_tc256(const void* q, const void* k, const void* v, const void* dout, void* dq_out,
                                      void* dk, void* dv, const float* lse2_ws, const float* delta_ws, float* dq_ws,
                                      float* dkv_ws, const SfaGeom& g, float scale, int32_t* status,
                                      cudaStream_t st) {
  using namespace tcbwd256;
  Params p;
  const SfaGeom gq = query_geom(g);
  if (!make_rows_tmap(&p.tm_q, q, gq, g.Hq, DH, PR) || !make_rows_tmap(&p.tm_do, dout, gq, g.Hq, DH, PR) ||
      !make_rows_tmap(&p.tm_k, k, g, g.Hkv, DH, PR) || !make_rows_tmap(&p.tm_v, v, g, g.Hkv, DH, PR))
    return cudaErrorInvalidValue;
  p.lse2 = lse2_ws;
  p.delta = delta_ws;
  p.dq = (bf16*)dq_out;
  p.dq_acc = dq_ws;
  p.dk = (bf16*)dk;
  p.dv = (bf16*)dv;
  const long long slice = (long long)g.B * g.q_ns * g.Lv * g.Hkv * DH;  // elements of dV (or dK) of one chunk
  const int ws_chunks = bwd_head_chunks(g, DH);
  long long room = ws_chunks > 1 ? ws_chunks : 0;
  p.dkv = dkv_ws;
  const long long acc_room = dq_out ? (long long)g.B * g.q_nL * g.Hq * DH / (2 * slice) : 0;
  if (acc_room > room) {
    room = acc_room;
    p.dkv = dq_ws;
  }
  p.head_pairs = (g.Hq / g.Hkv) % 2 == 0;
  const int rows = p.head_pairs ? BM : 2 * BM, nh = p.head_pairs ? g.Hq / 2 : g.Hq;
  const long long ndq = (long long)((g.Lq + rows - 1) / rows) * nh * g.q_ns * g.B;
  p.hchunks = head_chunks(g, room, ndq);
  p.grp = g.Hq / g.Hkv;
  p.hper = (p.grp + p.hchunks - 1) / p.hchunks;
  p.d_tile = make_fast_div((uint32_t)(p.hchunks * g.Hkv * g.q_ns * g.B));
  p.d_hc = make_fast_div((uint32_t)p.hchunks);
  p.d_kns = make_fast_div((uint32_t)(g.Hkv * g.q_ns));
  p.d_rank = make_fast_div((uint32_t)(nh * g.q_ns * g.B));
  p.d_hns = make_fast_div((uint32_t)(nh * g.q_ns));
  p.d_ns = make_fast_div((uint32_t)g.q_ns);
  p.d_grp = make_fast_div((uint32_t)p.grp);
  if (p.hchunks > 1 && p.dkv == nullptr) return cudaErrorInvalidValue;
  p.g = g;
  p.scale = scale;
  p.scale_log2 = scale * 1.4426950408889634f;
  p.status = status;
  p.nkv = (int)(key_items(g) * p.hchunks);
  const long long grid = 2 * (2LL * p.nkv + ndq);
  cudaError_t e = cudaFuncSetAttribute(bwd256_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e != cudaSuccess) return e;
  e = launch_attn(bwd256_kernel, grid, NTHREADS, kSmemBytes, st, p);
  if (e != cudaSuccess || p.hchunks == 1) return e;
  const long long n8 = slice / 8;
  return launch_attn(dkv_finalize_kernel, (n8 + 255) / 256, 256, 0, st, p.dkv, (bf16*)dk, (bf16*)dv, g, p.hchunks);
}

}  // namespace hdsfa
