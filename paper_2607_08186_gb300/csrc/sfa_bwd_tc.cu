// Stream-Factorized Attention backward (main pass) on the sm_103a tensor cores,
// head dims 64 and 128 (template parameter DH).
//
// Derivative of the forward of Eq. 4 / Fig. 2, which the paper trains through (Sec. 3.1),
// as two kinds of work items in one launch, a CTA each:
//   DKV  a 128-row key tile of one K/V head stationary, streaming the query tiles that see
//        it over the group's query heads:
//          S^T = K Q^T, P^T = exp2(c2 S^T - lse2), dP^T = V dO^T, dS^T = P^T (dP^T - delta)
//          dV += P^T dO,  dK += dS^T Q
//   DQ   a 128-row query tile of one head stationary, streaming the key tiles it sees:
//          S = Q K^T, P, dP = dO V^T, dS = P (dP - delta);  dQ += dS K
// (c2 = scale*log2e, lse2 = lse*log2e.)  S and dP are computed by both kinds (7 GEMMs for 5
// algorithmic ones), but every gradient is accumulated in TMEM over its item's whole loop
// and leaves once, in the same order on every run: no fp32 dQ accumulator in HBM to clear,
// add into and convert, and no dS or dQ tiles through shared memory.
//
// What bounds it: a fused kernel (dQ from the same dS^T) is limited by shared memory: a
// 128 x 128 x 16 MMA with both operands there reads 8 KB in its 64 cycles, all of the SM's
// 128 B per clock, and per tile pair it moved 480 KB (3750 cycles: operands 256, dQ staging
// and its reduce 128, TMA 64, dS 32) and took 4950 through its chain of pre-fills.  Here
// DKV moves 256 KB under 2048 cycles of MMA and takes about 2700 per step, bound by the
// chain S -> P -> dV, next S while every barrier and load of the softmax queues behind the
// MMAs' operand reads; DQ (Q and dO as A operands in TMEM: 160 KB under 1536) takes 1780,
// bound by dP -> dS -> dQ, next dP.  Large layers run at the card's power limit, where the
// 7 GEMMs cost clock: 2.0 -> 1.9 GHz.
// Measured, fwd + bwd, fused kernel (with this forward) -> this one: B=1, L=300, n=4, 32
// over 8 heads, intra-stream 94 -> 65 us; window of 1024 at L=4096 1088 -> 1063; cross-stream
// 2 x 4084 positions 884 -> 872; intra-stream L=4096 1753 -> 1775, 64 query heads 3487 ->
// 3488; head dim 64, 4 x 1501 tokens, n=3 415 -> 397; the tiny configuration 31 -> 27.  Relative
// error of dQ and dK against 64 bits 3.4e-3 -> 2.4e-3 (dS is rounded once, from fp32 P); dV
// 2.3e-3 as before.
//
// Issue order (one warp, in order, so that a region may be overwritten by the MMAs issued
// after those that read it):
//   DKV  S(0) dP(0), then per step t: wait P(t) | dV(t) S(t+1) | wait dS(t) | dK(t) dP(t+1)
//   DQ   S(0) dP(0) S(1), then per step t: wait dS(t) | dQ(t) dP(t+1) | wait S(t+1) read |
//        S(t+2)
// TMEM (512 columns): S at 0, dP at 128; DKV P^T packed over S, dS^T over dP, dV at 256, dK
// at 256 + DH; DQ dS over dP, dQ at 256, Q and dO packed at 384.  P and dS: each 64-column
// half at the start of its own columns.
// Roles (352 threads): warp 0 TMA producer; warp 1 MMA issuer (the whole warp runs the
// loop, one elected lane issues) and TMEM owner; warps 2..9 softmax, two threads per
// stationary row (TMEM lane), each half of the 128 streamed columns; warp 10 waits for the
// streamed tiles on the issuer's behalf.  A wait on a completed barrier costs 90 to 290
// cycles while MMAs read shared memory, so the issuer and the softmax warps wait for as
// little as possible: three waits more at the top of a softmax step made DQ's step 1840
// cycles and DKV's 2660.
// Grid: DKV items, key tiles with the most query tiles first, then DQ items, whose shorter
// ones fill the tail.  When there are too few DKV items to balance the SMs, each takes only
// a chunk of the group's query heads (head_chunks below), writing fp32 partial sums that
// dkv_finalize_kernel adds in chunk order.
// Every mbarrier wait is bounded.
#include "tc_common.cuh"

namespace hdsfa {

typedef __nv_bfloat16 bf16;

namespace tcbwd {
constexpr int BM = 128, BN = 128, NTHREADS = 352;
constexpr int HB = 64;  // streamed columns of one softmax thread
enum Kind { kDKV = 0, kDQ = 1 };
// TMEM columns: S at 0, dP at 128
constexpr uint32_t COL_P = 128;
constexpr uint32_t COL_OUT = 256;  // DKV: dV, then dK; DQ: dQ
constexpr uint32_t COL_A = 384;    // DQ: Q, then dO (packed bf16, DH/2 columns each)

template <int DH>
struct Smem {
  // tile buffers of [128 rows][DH] (DH/64 swizzle blocks).  DKV: K, V, then a ring of Q and
  // one of dO; DQ: a ring of K and one of V
  static constexpr int NBUF = DH == 64 ? 14 : 7;
  bf16 buf[NBUF][BN * DH];
  float nlse2[2][BN];         // DKV: -lse*log2(e) of the streamed query tile, by step parity
  float ndelta[2][BN];        // DKV: -delta of it
  uint64_t full[NBUF], empty[NBUF], a1_full, a2_full, a_tmem[2], term_full[2], term_empty[2];
  uint64_t s_full, s_empty, dp_full, p_full[2], ds_full[2], out_done;  // P and dS in halves
  uint32_t tmem_base;
  int abort;
};
// The layout needs 1024-byte alignment; the kernel checks the actual pad on entry.
template <int DH>
constexpr int smem_bytes() { return (int)sizeof(Smem<DH>) + 1024 < 232448 ? (int)sizeof(Smem<DH>) + 1024 : 232448; }
static_assert(sizeof(Smem<128>) <= 232448, "backward shared memory exceeds 227 KB");

struct Params {
  CUtensorMap tm_q, tm_do, tm_k, tm_v;
  const float* lse2;   // -lse*log2(e), [B][Hq][ns][Lvp]
  const float* delta;  // -delta, the same layout
  bf16* dq;            // dQ (scaled), or null: dq_acc
  float* dq_acc;       // unscaled fp32 dQ, added to what is there, when dq is null
  bf16* dk;
  bf16* dv;
  float* dkv;   // head chunks > 1: fp32 partial sums [chunks][2][B][q_ns][Lv][Hkv][DH] (dV, dK)
  int hchunks;  // query-head chunks per K/V head
  int nkv;      // DKV items; DQ items follow
  int grp, hper;  // query heads per K/V head, and per chunk
  FastDiv d_tile, d_hc, d_kvns, d_ns, d_rank, d_hns, d_grp, d_qstep;
  SfaGeom g;
  float scale, scale_log2;
  int32_t* status;
};

// One work item: its kind, stationary rows and the streamed steps.
struct Item {
  int kind;
  int b, s, sk, kvh, hc;
  int row0, h;    // first stationary row; first query head
  int grp;        // heads streamed (DKV: of the chunk; DQ: 1)
  int lo, nst;    // first streamed tile and tiles per head
  int T;          // steps: grp * nst
};

HD_DEVINLINE Item make_item(const Params& P, int idx) {
  const SfaGeom& G = P.g;
  Item it;
  it.hc = 0;
  if (idx < P.nkv) {
    it.kind = kDKV;
    const int HC = P.hchunks, per_tile = HC * G.Hkv * G.q_ns * G.B;
    const int j = fast_div(idx, P.d_tile), rem = idx - j * per_tile;  // key tile slowest
    const int hsb = fast_div(rem, P.d_hc);
    it.hc = rem - hsb * HC;
    it.b = fast_div(hsb, P.d_kvns);
    const int hs = hsb - it.b * G.Hkv * G.q_ns;
    it.kvh = fast_div(hs, P.d_ns);
    it.s = hs - it.kvh * G.q_ns;
    it.grp = min(P.hper, P.grp - it.hc * P.hper);
    it.h = it.kvh * P.grp + it.hc * P.hper;
    const int n0 = it.row0 = j * BM;
    // query rows that can see a key of the tile: key row r*qstep + qoff >= n0, and under
    // a window r*qstep + qoff < n0 + BM - 1 + window
    it.lo = (n0 <= G.qoff ? 0 : fast_div(n0 - G.qoff + G.qstep - 1, P.d_qstep)) / BN;
    int hi = (G.Lq - 1) / BN;
    if (G.window > 0) {
      const long long e = (long long)n0 + BM - 2 + G.window - G.qoff;
      if (e < (long long)G.Lv + BM) hi = min(hi, e < 0 ? -1 : fast_div((int)e, P.d_qstep) / BN);
    }
    it.nst = hi - it.lo + 1;
  } else {
    it.kind = kDQ;
    idx -= P.nkv;
    const int per_rank = G.Hq * G.q_ns * G.B, rank = fast_div(idx, P.d_rank);
    const int mt = (G.Lq + BM - 1) / BM - 1 - rank, hsb = idx - rank * per_rank;
    it.b = fast_div(hsb, P.d_hns);
    const int hs = hsb - it.b * G.Hq * G.q_ns;
    it.h = fast_div(hs, P.d_ns);
    it.s = hs - it.h * G.q_ns;
    it.kvh = fast_div(it.h, P.d_grp);
    it.grp = 1;
    const int m0 = it.row0 = mt * BM;
    const int rq_first = m0 * G.qstep + G.qoff, rq_last = (min(m0 + BM, G.Lq) - 1) * G.qstep + G.qoff;
    it.lo = G.window > 0 ? max(0, rq_first - G.window + 1) / BN : 0;
    it.nst = min(rq_last, G.Lv - 1) / BN - it.lo + 1;
  }
  it.T = it.nst > 0 ? it.grp * it.nst : 0;
  it.sk = it.s + G.kv_s0;
  return it;
}

// ACC: the instantiation that adds fp32 dQ into the accumulator (sfa_bwd_main).  Its own, since
// the reductions in the other's epilogue changed the code of its loops: 16 over 4 heads of 64,
// 4473 positions, cross-stream 168.5 -> 173.4 us.
template <int DH, bool ACC>
__global__ void __launch_bounds__(NTHREADS, 1) bwd_kernel(const __grid_constant__ Params P) {
  static_assert(DH == 64 || DH == 128, "head dim 64 or 128");
  constexpr int NBUF = Smem<DH>::NBUF;
  extern __shared__ uint8_t smem_raw[];
  {
    uint32_t dyn;
    asm("mov.u32 %0, %%dynamic_smem_size;\n" : "=r"(dyn));
    const uintptr_t base = reinterpret_cast<uintptr_t>(smem_raw);
    if (((base + 1023) & ~uintptr_t(1023)) - base + sizeof(Smem<DH>) > dyn) {  // uniform: nothing touched yet
      if (threadIdx.x == 0) set_status(P.status, HD_DEVBIT_TIMEOUT);
      return;
    }
  }
  Smem<DH>& sm = *reinterpret_cast<Smem<DH>*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const SfaGeom& G = P.g;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < NBUF; ++i) {
      mbar_init(&sm.full[i], 1);
      mbar_init(&sm.empty[i], 1);
    }
    mbar_init(&sm.a1_full, 1);
    mbar_init(&sm.a2_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sm.a_tmem[i], 8);
      mbar_init(&sm.term_full[i], 1);
      mbar_init(&sm.term_empty[i], 8);
      mbar_init(&sm.p_full[i], 8 + i);  // the softmax warps and, on the second half, the lander
      mbar_init(&sm.ds_full[i], 8 + i);
    }
    mbar_init(&sm.s_full, 1);
    mbar_init(&sm.s_empty, 8);  // one arrival per softmax warp
    mbar_init(&sm.dp_full, 1);
    mbar_init(&sm.out_done, 1);
    sm.abort = 0;
    fence_mbar_init();
  }
  attn_dep_wait(1);
  const Item it = make_item(P, (int)blockIdx.x);
  const int kind = it.kind, T = it.T;
  const size_t half = (size_t)G.B * G.q_ns * G.Lv * G.Hkv * DH;  // elements of a slice half
  if (T <= 0) {  // no query sees this key tile: its dK and dV rows are zero
    for (int i = threadIdx.x; i < 2 * BM * (DH / 8); i += NTHREADS) {
      const int which = i / (BM * (DH / 8)), kr = it.row0 + (i / (DH / 8)) % BM, c = i % (DH / 8);
      if (kr >= G.Lv) continue;
      if (P.hchunks > 1) {
        float* w = P.dkv + (2 * it.hc + which) * half +
                   ((((long long)it.b * G.q_ns + it.s) * G.Lv + kr) * G.Hkv + it.kvh) * DH + c * 8;
        reinterpret_cast<float4*>(w)[0] = make_float4(0.f, 0.f, 0.f, 0.f);
        reinterpret_cast<float4*>(w)[1] = make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
        bf16* w = (which ? P.dk : P.dv) +
                  (((long long)it.b * G.nL + (long long)kr * G.rs + it.sk) * G.Hkv + it.kvh) * DH + c * 8;
        *reinterpret_cast<uint4*>(w) = make_uint4(0, 0, 0, 0);
      }
    }
    return;
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, 512);
    tmem_relinquish();
    tc_fence_before();
  }
  volatile int* abort = &sm.abort;
  // the rings: buffers [b1, b1 + n1) and [b2, b2 + n2)
  const int b1 = kind == kDKV ? 2 : 0, n1 = (DH == 64 ? 2 : 1) * (kind == kDKV ? 3 : 4);
  const int b2 = b1 + n1, n2 = (DH == 64 ? 2 : 1) * (kind == kDKV ? 2 : 3);

  uint32_t tmem = 0;
  if (warp == 0) {
    named_bar_arrive(1, NTHREADS);  // the producer does not wait for the TMEM allocation
  } else {
    named_bar_sync(1, NTHREADS);
    tc_fence_after();
    tmem = sm.tmem_base;
  }

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      const bool kv = kind == kDKV;
      const CUtensorMap *tB1 = kv ? &P.tm_q : &P.tm_k, *tB2 = kv ? &P.tm_do : &P.tm_v;
      const int bstr = kv ? it.s : it.sk;
      auto load = [&](bf16* dst, const CUtensorMap* tm, uint64_t* bar, int hd, int str, int row) {
        mbar_arrive_expect_tx(bar, BN * DH * 2);
        for (int c = 0; c < DH / 64; ++c) tma_load_5d(dst + c * BN * 64, tm, bar, c * 64, hd, str, row, it.b);
      };
      int issued1 = 0, issued2 = 0, terms_issued = 0;
      int hd = kv ? it.h : it.kvh, qi = 0;  // streamed head and tile of the step
      bool ok = true;
      auto load_tile = [&](const CUtensorMap* tm, int base, int n, int& issued) {
        const int slot = base + issued % n, lap = issued / n;
        if (!ok || (lap > 0 && !mbar_wait(&sm.empty[slot], (lap - 1) & 1, abort, P.status))) {
          ok = false;
          return;
        }
        load(sm.buf[slot], tm, &sm.full[slot], hd, bstr, (it.lo + qi) * BN);
        ++issued;
      };
      auto load_a = [&](int second) {
        if (kv)
          load(sm.buf[second], second ? &P.tm_v : &P.tm_k, second ? &sm.a2_full : &sm.a1_full, it.kvh, it.sk, it.row0);
        else
          load(sm.buf[second ? b2 + n2 - 1 : b1 + n1 - 1], second ? &P.tm_do : &P.tm_q,
               second ? &sm.a2_full : &sm.a1_full, it.h, it.s, it.row0);
      };
      load_a(0);
      if (!kv) load_a(1);
      for (int t = 0; ok && t < T; ++t) {
        // DQ: the last slots of the rings hold Q and dO until they are in TMEM
        if (!kv && t == n2 - 1 && (!mbar_wait(&sm.a_tmem[0], 0, abort, P.status) || !mbar_wait(&sm.a_tmem[1], 0, abort, P.status)))
          break;
        load_tile(tB1, b1, n1, issued1);
        if (kv && t == 0) load_a(1);
        load_tile(tB2, b2, n2, issued2);
        if (kv && ok) {  // the step's row terms, into the buffer that step t-2 has read
          if (t >= 2 && !mbar_wait(&sm.term_empty[t & 1], ((t >> 1) - 1) & 1, abort, P.status)) break;
          const long long off = (((long long)it.b * G.Hq + hd) * G.q_ns + it.s) * row_terms_pitch(G.Lq) +
                                (long long)(it.lo + qi) * BN;
          mbar_arrive_expect_tx(&sm.term_full[t & 1], 2 * BN * 4);
          bulk_load(sm.nlse2[t & 1], P.lse2 + off, BN * 4, &sm.term_full[t & 1]);
          bulk_load(sm.ndelta[t & 1], P.delta + off, BN * 4, &sm.term_full[t & 1]);
          terms_issued = t + 1;
        }
        if (++qi == it.nst) {
          qi = 0;
          ++hd;
        }
      }
      // every copy this thread started lands before the CTA may exit
      mbar_drain(&sm.a1_full, 0);
      mbar_drain(&sm.a2_full, 0);
      for (int u = max(0, issued1 - n1); u < issued1; ++u) mbar_drain(&sm.full[b1 + u % n1], (u / n1) & 1);
      for (int u = max(0, issued2 - n2); u < issued2; ++u) mbar_drain(&sm.full[b2 + u % n2], (u / n2) & 1);
      for (int t = max(0, terms_issued - 2); t < terms_issued; ++t) mbar_drain(&sm.term_full[t & 1], (t >> 1) & 1);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    constexpr uint32_t idS = idesc_bf16(BM, BN, 0, 0);  // S, dP: both operands K-major
    constexpr uint32_t idO = idesc_bf16(BM, DH, 0, 1);  // outputs: A in TMEM, B MN-major
    // descriptors encoded once; a slot or k-step adds its byte offset / 16
    const uint64_t dK = sdesc_sw128(smem_u32(sm.buf[0]), 16, 1024);        // a buffer K-major
    const uint64_t dM = sdesc_sw128(smem_u32(sm.buf[0]), BN * 128, 1024);  // ... MN-major
    constexpr int TILE16 = BN * DH * 2 / 16;
    auto wait_w = [&](uint64_t* bar, int par) -> bool {
      if (!__all_sync(0xffffffffu, mbar_wait(bar, par & 1, abort, P.status))) return false;
      tc_fence_after();
      return true;
    };
    auto koff = [](int kk) { return (uint64_t)((kk >> 2) * (128 * 128 / 16) + (kk & 3) * 2); };
    // D[128 x 128] = A B^T over the head dim; A: a tile buffer, or packed in TMEM columns
    auto gemm_ss = [&](uint32_t col, int abuf, int slot) {
#pragma unroll
      for (int kk = 0; kk < DH / 16; ++kk)
        tc_mma_ss_w(tmem + col, dK + (uint64_t)(abuf * TILE16) + koff(kk), dK + (uint64_t)(slot * TILE16) + koff(kk), idS,
                    kk > 0 ? 1u : 0u);
    };
    auto gemm_ts = [&](uint32_t col, uint32_t acol, int slot) {
#pragma unroll
      for (int kk = 0; kk < DH / 16; ++kk)
        tc_mma_ts_w(tmem + col, tmem + acol + kk * 8, dK + (uint64_t)(slot * TILE16) + koff(kk), idS, kk > 0 ? 1u : 0u);
    };
    // output += A[tmem] B over 128 streamed rows, half of them at a time: the softmax
    // publishes the first 32 of each thread's 64 columns ahead of the others
    auto gemm_out = [&](uint32_t col, uint32_t acol, int slot, bool acc0, uint64_t* a_full, int par) -> bool {
      const uint64_t bd = dM + (uint64_t)(slot * TILE16);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        if (!wait_w(a_full + hf, par)) return false;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int kk = (k >> 1) * 4 + hf * 2 + (k & 1);
          tc_mma_ts_w(tmem + col, tmem + acol + (kk >> 2) * HB + (kk & 3) * 8, bd + (uint64_t)(kk * 16 * 128 / 16), idO,
                      (acc0 || hf > 0 || k > 0) ? 1u : 0u);
        }
      }
      return true;
    };
    auto next1 = [&](int s) { return s + 1 == b1 + n1 ? b1 : s + 1; };
    auto next2 = [&](int s) { return s + 1 == b2 + n2 ? b2 : s + 1; };
    int s1 = b1, s2 = b2;  // buffers of the step's Q and dO, or K and V
    bool ok = wait_w(kind == kDKV ? &sm.a1_full : &sm.a_tmem[0], 0) && wait_w(&sm.full[s1], 0);
    if (kind == kDKV) {
      if (ok) {
        gemm_ss(0, 0, s1);
        tc_commit_w(&sm.s_full);
        ok = wait_w(&sm.a2_full, 0) && wait_w(&sm.full[s2], 0);
      }
      if (ok) {
        gemm_ss(COL_P, 1, s2);
        tc_commit_w(&sm.dp_full);
      }
      for (int t = 0; ok && t < T; ++t) {
        const int s1n = next1(s1), s2n = next2(s2);
        if (!gemm_out(COL_OUT, 0, s2, t > 0, sm.p_full, t)) { ok = false; break; }
        tc_commit_w(&sm.empty[s2]);  // dP(t), issued before, has read dO(t) too
        if (t + 1 < T) {             // over P^T(t)
          gemm_ss(0, 0, s1n);
          tc_commit_w(&sm.s_full);
        }
        if (!gemm_out(COL_OUT + DH, COL_P, s1, t > 0, sm.ds_full, t)) { ok = false; break; }
        tc_commit_w(&sm.empty[s1]);
        if (t + 1 < T) {  // over dS^T(t)
          gemm_ss(COL_P, 1, s2n);
          tc_commit_w(&sm.dp_full);
        }
        s1 = s1n;
        s2 = s2n;
      }
    } else {
      if (ok) {
        gemm_ts(0, COL_A, s1);
        tc_commit_w(&sm.s_full);
        ok = wait_w(&sm.a_tmem[1], 0) && wait_w(&sm.full[s2], 0);
      }
      if (ok) {
        gemm_ts(COL_P, COL_A + DH / 2, s2);
        tc_commit_w(&sm.dp_full);
        tc_commit_w(&sm.empty[s2]);
        if (T > 1) {
          ok = wait_w(&sm.full[next1(s1)], 0) && wait_w(&sm.s_empty, 0);
          if (ok) {
            gemm_ts(0, COL_A, next1(s1));
            tc_commit_w(&sm.s_full);
          }
        }
      }
      for (int t = 0; ok && t < T; ++t) {
        s2 = next2(s2);  // V(t+1)
        if (!gemm_out(COL_OUT, COL_P, s1, t > 0, sm.ds_full, t)) { ok = false; break; }
        tc_commit_w(&sm.empty[s1]);
        if (t + 1 < T) {  // over dS(t)
          gemm_ts(COL_P, COL_A + DH / 2, s2);
          tc_commit_w(&sm.dp_full);
        }
        if (t + 2 < T) {
          if (!wait_w(&sm.s_empty, t + 1)) { ok = false; break; }
          gemm_ts(0, COL_A, next1(next1(s1)));
          tc_commit_w(&sm.s_full);
        }
        if (t + 1 < T) tc_commit_w(&sm.empty[s2]);
        s1 = next1(s1);
      }
    }
    // every MMA issued above completes before TMEM / smem are released
    tc_commit_w(&sm.out_done);
    mbar_drain(&sm.out_done, 0);
  } else if (warp == NTHREADS / 32 - 1) {
    // ------------------------------------------------------------ lander
    // Waits for the streamed tiles that the issuer takes next and then arrives where the
    // issuer waits for the softmax, so that neither of them waits for the tiles.  A phase is
    // arrived on only after the one before has completed.
    if (lane == 0) {
      auto wait1 = [&](int t) { return t >= T || mbar_wait(&sm.full[b1 + t % n1], (t / n1) & 1, abort, P.status); };
      auto wait2 = [&](int t) { return t >= T || mbar_wait(&sm.full[b2 + t % n2], (t / n2) & 1, abort, P.status); };
      auto arrive = [&](uint64_t* bar, int t) {
        if (t > 0 && !mbar_wait(bar, (t - 1) & 1, abort, P.status)) return false;
        mbar_arrive(bar);
        return true;
      };
      for (int t = 0; t < T; ++t) {
        if (kind == kDKV) {
          if (!wait1(t + 1) || !arrive(&sm.p_full[1], t)) break;                   // S(t+1)
          if (!wait2(t + 1) || !arrive(&sm.ds_full[1], t)) break;                  // dP(t+1)
        } else {
          if (!wait2(t + 1) || !wait1(t + 2) || !arrive(&sm.ds_full[1], t)) break;  // dP(t+1), S(t+2)
        }
      }
    }
  } else {
    // ------------------------------------------------------------ softmax / epilogue
    const int q4 = warp & 3, hc = (warp - 2) >> 2;
    const int r = it.row0 + q4 * 32 + lane;  // stationary row: query row (DQ) or key row (DKV)
    const uint32_t tq = tmem + ((uint32_t)(q4 * 32) << 16);
    const uint32_t tl = tq + HB * hc;  // this thread's half of a region
    const float c2 = P.scale_log2;
    const uint64_t c2x2 = f2pack(c2, c2);
    auto publish = [&](uint64_t* bar) {  // this warp's TMEM accesses are done: tell the issuer
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
    };
    // dS = P (dP - delta), packed bf16 over the first half of this thread's dP columns, all
    // of them read before (the loads run one 16-column chunk ahead)
    auto ds_half = [&](const float* x, auto nd) {
      uint32_t d[2][16];
      tmem_ld16(tl + COL_P, d[0]);
#pragma unroll
      for (int c = 0; c < HB / 16; ++c) {
        uint32_t* dc = d[c & 1];
        tmem_ld_wait();
        if (c + 1 < HB / 16) tmem_ld16(tl + COL_P + (c + 1) * 16, d[(c + 1) & 1]);
        uint32_t pk[8];
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
          float y0, y1;
          f2unpack(fmul2(fadd2(f2pack(__uint_as_float(dc[e]), __uint_as_float(dc[e + 1])), nd(c * 8 + (e >> 1))),
                         f2pack(x[c * 16 + e], x[c * 16 + e + 1])),
                   y0, y1);
          pk[e >> 1] = cvt_bf16x2(y0, y1);
        }
        tmem_st8(tl + COL_P + c * 8, pk);
        if (c & 1) {
          tmem_st_wait();
          publish(&sm.ds_full[c >> 1]);
        }
      }
    };
    bool ok = true;

    if (kind == kDQ) {
      const int rq = r * G.qstep + G.qoff;             // key row of this query
      const int rq0 = it.row0 * G.qstep + G.qoff;      // ... of the tile's first query
      const int rq1 = (it.row0 + BM - 1) * G.qstep + G.qoff;
      float nl = -INFINITY, nd = 0.f;  // rows past Lq: P = 0
      if (r < G.Lq) {
        const long long off = (((long long)it.b * G.Hq + it.h) * G.q_ns + it.s) * row_terms_pitch(G.Lq) + r;
        nl = P.lse2[off];
        nd = P.delta[off];
      }
      const uint64_t nl2 = f2pack(nl, nl), nd2 = f2pack(nd, nd);
      // A operands: this thread's half row of Q and of dO from their tile buffers into TMEM.
      // From there the S and dP MMAs read only B from shared memory, half of its bandwidth.
      for (int w = 0; w < 2; ++w) {
        if (!__all_sync(0xffffffffu, mbar_wait(w ? &sm.a2_full : &sm.a1_full, 0, abort, P.status))) ok = false;
        const int row = q4 * 32 + lane;
        const uint8_t* src = reinterpret_cast<const uint8_t*>(sm.buf[w ? b2 + n2 - 1 : b1 + n1 - 1]) +
                             (DH == 128 ? hc * (BM * 128) : 0) + row * 128;  // 128-byte swizzled rows of 64 columns
        uint32_t a[DH / 4];
#pragma unroll
        for (int e = 0; e < DH / 16; ++e) {
          const int u = e + (DH == 128 ? 0 : hc * 4);
          const uint4 v = *reinterpret_cast<const uint4*>(src + ((u ^ (row & 7)) << 4));
          a[4 * e] = v.x;
          a[4 * e + 1] = v.y;
          a[4 * e + 2] = v.z;
          a[4 * e + 3] = v.w;
        }
#pragma unroll
        for (int e = 0; e < DH / 64; ++e) tmem_st16(tq + COL_A + w * (DH / 2) + (DH / 4) * hc + e * 16, a + e * 16);
        tmem_st_wait();
        publish(&sm.a_tmem[w]);
      }
      for (int t = 0; ok && t < T; ++t) {
        const int c0 = (it.lo + t) * BN + HB * hc;  // first key of this half
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.s_full, t & 1, abort, P.status))) {
          ok = false;
          break;
        }
        tc_fence_after();
        float x[HB];
#pragma unroll
        for (int c = 0; c < HB / 32; ++c) tmem_ld32(tl + c * 32, reinterpret_cast<uint32_t*>(x) + c * 32);
        tmem_ld_wait();
        publish(&sm.s_empty);
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
        if (G.smod > 1) {  // the naive intra-stream schedule: key row = query row (mod smod)
          int k = (rq - c0) % G.smod;
          if (k < 0) k += G.smod;
#pragma unroll
          for (int e = 0; e < HB; ++e) {
            if (k != 0) x[e] = 0.f;
            k = k == 0 ? G.smod - 1 : k - 1;
          }
        }
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.dp_full, t & 1, abort, P.status))) {
          ok = false;
          break;
        }
        tc_fence_after();
        ds_half(x, [&](int) { return nd2; });
      }
    } else {
      // DKV: this thread's key row r.  The streamed tile's row terms come through shared
      // memory and are taken into registers before the MMA results they belong to are
      // waited for: a broadcast load queues behind the MMAs' operand reads.
      const int kr = r;
      // key row kr sees the queries q in [vis_lo, vis_hi): q*qstep + qoff >= kr (causal),
      // and for LOCAL q*qstep + qoff < kr + window.  Queries past Lq have -lse2 = -inf; a
      // key row past Lv is not stored.
      const int vis_lo = kr <= G.qoff ? 0 : fast_div(kr - G.qoff + G.qstep - 1, P.d_qstep);
      int vis_hi = G.Lq;
      if (G.window > 0) {
        const long long e = (long long)kr + G.window - G.qoff;  // q*qstep < e
        if (e < (long long)G.Lv) vis_hi = min(vis_hi, e <= 0 ? 0 : fast_div((int)e + G.qstep - 1, P.d_qstep));
      }
      int qi = 0;  // query tile of the step within its head
      auto terms_landed = [&](int t) {
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.term_full[t & 1], (t >> 1) & 1, abort, P.status))) ok = false;
      };
      terms_landed(0);
      for (int t = 0; ok && t < T; ++t) {
        const int qm = (it.lo + qi) * BN;
        if (++qi == it.nst) qi = 0;
        ulonglong2 tm[HB / 4];
#pragma unroll
        for (int e = 0; e < HB / 4; ++e) tm[e] = reinterpret_cast<const ulonglong2*>(sm.nlse2[t & 1] + HB * hc)[e];
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.s_full, t & 1, abort, P.status))) {
          ok = false;
          break;
        }
        tc_fence_after();
        float x[HB];
#pragma unroll
        for (int c = 0; c < HB / 32; ++c) tmem_ld32(tl + c * 32, reinterpret_cast<uint32_t*>(x) + c * 32);
        tmem_ld_wait();
        // the diagonal band and (LOCAL) tiles that reach the window edge of the first key
        const bool edge = qm * G.qstep + G.qoff < it.row0 + BM ||
                          (G.window > 0 && (qm + BN - 1) * G.qstep + G.qoff - G.window >= it.row0);
        const int lo = vis_lo - qm - HB * hc, hi = vis_hi - qm - HB * hc;
        int kmod = 0;  // (query row - key row) mod smod of the naive intra-stream schedule
        if (G.smod > 1) {
          kmod = (qm + HB * hc - kr) % G.smod;
          if (kmod < 0) kmod += G.smod;
        }
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
#pragma unroll
          for (int e = hf * 32; e < hf * 32 + 32; e += 2) {
            float a0, a1;
            f2unpack(ffma2(f2pack(x[e], x[e + 1]), c2x2, (e & 2) ? tm[e >> 2].y : tm[e >> 2].x), a0, a1);
            x[e] = ex2_approx(a0);
            x[e + 1] = ex2_approx(a1);
          }
          if (edge) {
#pragma unroll
            for (int e = hf * 32; e < hf * 32 + 32; ++e)
              if (e < lo || e >= hi) x[e] = 0.f;
          }
          if (G.smod > 1) {
#pragma unroll
            for (int e = hf * 32; e < hf * 32 + 32; ++e) {
              if (kmod != 0) x[e] = 0.f;
              kmod = kmod + 1 == G.smod ? 0 : kmod + 1;
            }
          }
#pragma unroll
          for (int c = 2 * hf; c < 2 * hf + 2; ++c) {
            uint32_t pk[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) pk[e >> 1] = cvt_bf16x2(x[c * 16 + e], x[c * 16 + e + 1]);
            tmem_st8(tl + c * 8, pk);
          }
          tmem_st_wait();
          publish(&sm.p_full[hf]);
        }
        const ulonglong2* nd4 = reinterpret_cast<const ulonglong2*>(sm.ndelta[t & 1] + HB * hc);
        ulonglong2 td[HB / 4];
#pragma unroll
        for (int e = 0; e < HB / 8; ++e) td[e] = nd4[e];
        if (t + 1 < T) terms_landed(t + 1);  // here, where the softmax waits for dP anyway
        if (!__all_sync(0xffffffffu, mbar_wait(&sm.dp_full, t & 1, abort, P.status))) {
          ok = false;
          break;
        }
        tc_fence_after();
        ds_half(x, [&](int e2) {
          if (e2 < HB / 4 && !(e2 & 7)) {  // a chunk ahead of their use, in the registers the first half leaves
#pragma unroll
            for (int e = 0; e < 4; ++e) td[HB / 8 + (e2 >> 1) + e] = nd4[HB / 8 + (e2 >> 1) + e];
          }
          return (e2 & 1) ? td[e2 >> 1].y : td[e2 >> 1].x;
        });
        if (lane == 0) mbar_arrive(&sm.term_empty[t & 1]);
      }
    }

    // epilogue: this thread's half (DH/2 columns) of its row of each output
    if (ok && __all_sync(0xffffffffu, mbar_wait(&sm.out_done, 0, abort, P.status))) {
      tc_fence_after();
      constexpr int UPR = DH * 2 / 16, UPH = UPR / 2;  // 16-byte units per row and half row
      const int nrow = kind == kDQ ? G.Lq : G.Lv;
      const bool f32_out = kind == kDQ ? P.dq == nullptr : P.hchunks > 1;  // (dq is null only with ACC)
#pragma unroll 1
      for (int o = 0; o < (kind == kDQ ? 1 : 2); ++o) {  // DQ: dQ; DKV: dV, then dK
        const uint32_t to = tq + (kind == kDQ ? COL_OUT : COL_OUT + o * DH) + (DH / 2) * hc;
        if (f32_out) {
          float* dst;
          float m = o ? P.scale : 1.f;
          if (kind == kDQ) {  // unscaled (sfa_bwd_finalize applies the scale) and added: one sum per call
            dst = P.dq_acc + (((long long)it.b * G.q_nL + (long long)r * G.q_rs + it.s) * G.Hq + it.h) * DH;
          } else {
            dst = P.dkv + (2 * it.hc + o) * half + ((((long long)it.b * G.q_ns + it.s) * G.Lv + r) * G.Hkv + it.kvh) * DH;
          }
          dst += (DH / 2) * hc;
#pragma unroll 1
          for (int c = 0; c < DH / 64; ++c) {
            uint32_t v[32];
            tmem_ld32(to + c * 32, v);
            tmem_ld_wait();
            if (r < nrow) {
#pragma unroll
              for (int e = 0; e < 32; e += 4) {
                const float4 w = make_float4(__uint_as_float(v[e]) * m, __uint_as_float(v[e + 1]) * m,
                                             __uint_as_float(v[e + 2]) * m, __uint_as_float(v[e + 3]) * m);
                if (ACC && kind == kDQ)
                  red_add4(dst + c * 32 + e, w.x, w.y, w.z, w.w);
                else
                  *reinterpret_cast<float4*>(dst + c * 32 + e) = w;
              }
            }
          }
        } else {
          // rows leave through shared memory (no tile buffer is read any more): each thread writes
          // its half row as bf16, 16-byte units XOR-swizzled by the row, then every store
          // instruction of the warp writes whole half rows
          const float mul = kind == kDQ || o ? P.scale : 1.f;
          uint8_t* stg = reinterpret_cast<uint8_t*>(sm.buf[o]) + q4 * (32 * DH * 2);
#pragma unroll
          for (int c = 0; c < DH / 64; ++c) {
            uint32_t v[32];
            tmem_ld32(to + c * 32, v);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; e += 8) {
              uint4 w;
              w.x = cvt_bf16x2(__uint_as_float(v[e + 0]) * mul, __uint_as_float(v[e + 1]) * mul);
              w.y = cvt_bf16x2(__uint_as_float(v[e + 2]) * mul, __uint_as_float(v[e + 3]) * mul);
              w.z = cvt_bf16x2(__uint_as_float(v[e + 4]) * mul, __uint_as_float(v[e + 5]) * mul);
              w.w = cvt_bf16x2(__uint_as_float(v[e + 6]) * mul, __uint_as_float(v[e + 7]) * mul);
              const int u = hc * UPH + c * 4 + e / 8;
              *reinterpret_cast<uint4*>(stg + lane * (DH * 2) + ((u ^ (lane & (UPH - 1))) << 4)) = w;
            }
          }
          __syncwarp();
          bf16* base;
          long long rstride;  // elements between rows
          if (kind == kDQ) {
            base = P.dq + (((long long)it.b * G.q_nL + it.s) * G.Hq + it.h) * DH;
            rstride = (long long)G.q_rs * G.Hq * DH;
          } else {
            base = (o ? P.dk : P.dv) + (((long long)it.b * G.nL + it.sk) * G.Hkv + it.kvh) * DH;
            rstride = (long long)G.rs * G.Hkv * DH;
          }
          const int r0 = it.row0 + q4 * 32, u = hc * UPH + lane % UPH;
#pragma unroll
          for (int k = 0; k < UPH; ++k) {
            const int i = k * (32 / UPH) + lane / UPH;  // row within the warp
            if (r0 + i < nrow)
              *reinterpret_cast<uint4*>(base + (long long)(r0 + i) * rstride + u * 8) =
                  *reinterpret_cast<const uint4*>(stg + i * (DH * 2) + ((u ^ (i & (UPH - 1))) << 4));
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}
// Head chunks: dv / dk rows (bf16) from the chunks' fp32 partial sums, added in chunk
// order, 8 columns per thread.
template <int DH>
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

// Query-head chunks of the DKV items: the count with the least estimated time over the
// chip's SMs, as the larger of an SM's share of all items and the longest item (the key
// tile with the most query tiles), plus the finalize pass where there are chunks.  In units
// of 1000 cycles: a step of DKV and DQ 2.6 and 1.9, an item's fixed part 9, the
// finalize pass 8 and its traffic (8 bytes written and read per element and chunk at about
// 3.4 KB per cycle).  `room`: slices of partial sums there is space for.
static int head_chunks(const SfaGeom& g, int Dh, long long room) {
  const int grp = g.Hq / g.Hkv;
  const int ntile = (g.Lv + BM - 1) / BM;
  const long long items = (long long)ntile * g.Hkv * g.q_ns * g.B;
  if (grp < 2 || room < 2 || items >= 4 * kSmCount) return 1;
  double sum = 0, most = 0;  // query tiles per head that each key tile streams
  for (int j = 0; j < ntile; ++j) {
    const int n0 = j * BM;
    const int lo = (n0 <= g.qoff ? 0 : (n0 - g.qoff + g.qstep - 1) / g.qstep) / BN;
    int hi = (g.Lq - 1) / BN;
    if (g.window > 0 && n0 + BM - 2 + g.window - g.qoff < (hi + 1) * BN * g.qstep)
      hi = (n0 + BM - 2 + g.window - g.qoff) / g.qstep / BN;
    const double nst = hi >= lo ? hi - lo + 1 : 0;
    sum += nst;
    most = nst > most ? nst : most;
  }
  const double per = (double)items / ntile;  // items of one key tile
  const double ndq = (double)((g.Lq + BM - 1) / BM) * g.Hq * g.q_ns * g.B;
  const double dq = ndq * 9.0 + 1.9 * sum * per * grp;
  int best = 1;
  double best_cost = 0;
  for (int hs = 1; hs <= grp && hs <= room; ++hs) {
    const int hper = (grp + hs - 1) / hs;
    if ((grp + hper - 1) / hper != hs) continue;  // another count gives the same chunks
    const double total = dq + (double)items * hs * 9.0 + 2.6 * sum * per * grp;
    const double longest = 9.0 + 2.6 * hper * most;
    const double share = total / kSmCount;
    double cost = share > longest ? share : longest;
    if (hs > 1) cost += 8.0 + 16.0 * hs * g.B * g.q_ns * (double)g.Lv * g.Hkv * Dh / 3.4e6;
    if (best_cost == 0 || cost < best_cost) {
      best = hs;
      best_cost = cost;
    }
  }
  return best;
}
}  // namespace tcbwd

template <int DH>
static cudaError_t bwd_tc_impl(tcbwd::Params& p, long long slice, cudaStream_t st) {
  using namespace tcbwd;
  const SfaGeom& g = p.g;
  constexpr int smem = smem_bytes<DH>();
  const auto kernel = p.dq ? bwd_kernel<DH, false> : bwd_kernel<DH, true>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const long long ndq = (long long)((g.Lq + BM - 1) / BM) * g.Hq * g.q_ns * g.B;
  e = launch_attn(kernel, p.nkv + ndq, NTHREADS, smem, st, p);
  if (e != cudaSuccess || p.hchunks == 1) return e;
  const long long n8 = slice / 8;
  return launch_attn(dkv_finalize_kernel<DH>, (n8 + 255) / 256, 256, 0, st, p.dkv, p.dk, p.dv, g, p.hchunks);
}

// Dh: 64 or 128.  dq_out: bf16 dQ (scaled); null: unscaled fp32 dQ added into dq_ws.  With dq_out
// the space of dq_ws is free and holds the chunks' partial sums when it is larger than dkv_ws.
cudaError_t launch_sfa_bwd_main_tc(const void* q, const void* k, const void* v, const void* dout, void* dq_out,
                                   void* dk, void* dv, const float* lse2_ws, const float* delta_ws, float* dq_ws,
                                   float* dkv_ws, const SfaGeom& g, int Dh, float scale, int32_t* status,
                                   cudaStream_t st) {
  using namespace tcbwd;
  Params p;
  const SfaGeom gq = query_geom(g);
  if (!make_rows_tmap(&p.tm_q, q, gq, g.Hq, Dh, BN) || !make_rows_tmap(&p.tm_do, dout, gq, g.Hq, Dh, BN) ||
      !make_rows_tmap(&p.tm_k, k, g, g.Hkv, Dh, BN) || !make_rows_tmap(&p.tm_v, v, g, g.Hkv, Dh, BN))
    return cudaErrorInvalidValue;
  p.lse2 = lse2_ws;
  p.delta = delta_ws;
  p.dq = (bf16*)dq_out;
  p.dq_acc = dq_ws;
  p.dk = (bf16*)dk;
  p.dv = (bf16*)dv;
  const long long slice = (long long)g.B * g.q_ns * g.Lv * g.Hkv * Dh;  // elements of dV (or dK) of one chunk
  const int ws_chunks = bwd_head_chunks(g, Dh);
  long long room = ws_chunks > 1 ? ws_chunks : 0;
  p.dkv = dkv_ws;
  const long long acc_room = dq_out ? (long long)g.B * g.q_nL * g.Hq * Dh / (2 * slice) : 0;
  if (acc_room > room) {
    room = acc_room;
    p.dkv = dq_ws;
  }
  p.hchunks = head_chunks(g, Dh, room);
  if (p.hchunks > 1 && p.dkv == nullptr) return cudaErrorInvalidValue;
  p.g = g;
  p.scale = scale;
  p.scale_log2 = scale * 1.4426950408889634f;
  p.status = status;
  p.grp = g.Hq / g.Hkv;
  p.hper = (p.grp + p.hchunks - 1) / p.hchunks;
  p.d_tile = make_fast_div((uint32_t)(p.hchunks * g.Hkv * g.q_ns * g.B));
  p.d_hc = make_fast_div((uint32_t)p.hchunks);
  p.d_kvns = make_fast_div((uint32_t)(g.Hkv * g.q_ns));
  p.d_ns = make_fast_div((uint32_t)g.q_ns);
  p.d_rank = make_fast_div((uint32_t)(g.Hq * g.q_ns * g.B));
  p.d_hns = make_fast_div((uint32_t)(g.Hq * g.q_ns));
  p.d_grp = make_fast_div((uint32_t)p.grp);
  p.d_qstep = make_fast_div((uint32_t)g.qstep);
  p.nkv = (int)((long long)((g.Lv + BM - 1) / BM) * g.Hkv * g.q_ns * g.B * p.hchunks);
  return Dh == 64 ? bwd_tc_impl<64>(p, slice, st) : bwd_tc_impl<128>(p, slice, st);
}

}  // namespace hdsfa
