// Stream-Factorized Attention forward on the sm_103a tensor cores, head dim 256
// (the 80B configuration's heads, Table 6).
//
// Same problem and masks as the head-dim <= 128 forward (Eq. 4, Fig. 2a/2b, and the
// final-stream query geometry of Sec. 3.1).  The tile plan differs because a 128-row query
// tile's O accumulator alone takes 256 of the 512 TMEM columns and its Q tile 64 KB of
// shared memory: one tile per CTA.  A key tile of 128 keys is then 128 KB of K and V for
// 2048 cycles of MMA, and one CTA's worth of it in every SM (64 B/clock each) is more than
// L2 delivers.  So a pair of CTAs works on two query tiles (cta_group::2, M = 256) and each
// CTA loads half of every K and V tile: 32 B/clock.
//   smem   Q (four [128][64] swizzle blocks, 64 KB) and a ring of five 32 KB slots: of a K
//          tile this CTA's 64 keys, of a V tile this CTA's 128 head-dim columns.
//   TMEM   S in two 128-column buffers (P packed bf16 over its S, each 64-key half at the
//          start of its own columns), O over columns 256..511.
//   issue  S(0), then per key tile t: S(t+1), O += P(t) V(t).
// The two query tiles are the same rows of two heads of one K/V group where the group has
// an even number of heads (same key range), else consecutive tiles of one head.
// Roles per CTA (320 threads): warp 0 TMA producer; warp 1 MMA issuer (the pair's first CTA
// only: the whole warp runs the loop, one elected lane issues) and TMEM owner; warps 2..9
// online softmax, two threads per query row (TMEM lane), each half of a tile's keys, in fp32
// with exp2.  The two exchange their maximum through shared memory, so both decide alike; O
// is rescaled in TMEM, 128 columns by each, only when the running maximum grows by more than
// 2^8.  P is published in two parts (the first 32 keys of each half, then the rest), so the
// PV of the first runs while the second is computed.
// A full barrier lives in the first CTA and counts both CTAs' bytes; commits are multicast.
// What bounds it: the tensor pipe; a key tile takes 2060 cycles against 2048 of MMA (one CTA
// with the whole tile in its own shared memory, as this kernel was before: about 3050).
// The rest is each CTA's start (1800 cycles to the first load, 2500 more to the first MMA)
// and end (the last softmax and PV, 2400 to store O).  24 over 2 heads, 4096 positions x 4
// streams: WITHIN 607 -> 499 us, final-stream CROSS 488 -> 411 us.
// Every mbarrier wait is bounded; copies still in flight when a wait gives up were issued
// a whole timeout (about a second) earlier.
#include "tc_common.cuh"

namespace hdsfa {

typedef __nv_bfloat16 bf16;

namespace tcfwd256 {
constexpr int DH = 256, BM = 128, BN = 128, NSLOT = 5, NTHREADS = 320;
constexpr int HB = 64;   // keys of a K tile that a CTA loads, and keys of one softmax thread
constexpr int PC = 128;  // head-dim columns of a V tile that a CTA loads, and of O per softmax thread
constexpr uint32_t COL_O = 256;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleThreshold = 8.0f;  // log2 units: P stays <= 256 between O rescales

struct Smem {
  bf16 q[BM * DH];            // four [128 rows][64] swizzle blocks
  bf16 ring[NSLOT][HB * DH];  // K: four [64 keys][64] swizzle blocks; V: two [128 keys][64]
  float part[2][2][BM];       // by tile parity and key half: a row's maximum (at the end: its sum)
  // S(t) and PV(t) complete: by t mod 4, since the producer, which takes them as the release
  // of K(t) and V(t), may be up to two tiles late
  uint64_t s_full[4], pv_done[4];
  uint64_t full[NSLOT], q_full[DH / 64], p_full[2][2], o_done;
  uint32_t tmem_base;
  int abort;
};
// The layout needs 1024-byte alignment; the kernel checks the actual pad on entry.
constexpr int kSmemBytes = sizeof(Smem) + 1024 < 232448 ? (int)sizeof(Smem) + 1024 : 232448;
static_assert(sizeof(Smem) <= 232448, "head-dim-256 forward shared memory exceeds 227 KB");

struct Params {
  CUtensorMap tm_q, tm_k, tm_v;  // boxes of 128 (Q, V) and 64 (K) rows x 64 columns
  bf16* o;
  float* lse;
  SfaGeom g;
  float scale_log2;
  int32_t* status;
  int head_pairs;  // 1: a pair's two query tiles are the same rows of two heads of one K/V group
  FastDiv d_rank, d_hns, d_ns, d_grp;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NTHREADS, 1) fwd256_kernel(const __grid_constant__ Params P) {
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
  if (threadIdx.x == 0) {
    for (int i = 0; i < NSLOT; ++i) mbar_init(&sm.full[i], 1);
    for (int i = 0; i < 4; ++i) {
      mbar_init(&sm.s_full[i], 1);
      mbar_init(&sm.pv_done[i], 1);
    }
    for (int i = 0; i < DH / 64; ++i) mbar_init(&sm.q_full[i], 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sm.p_full[i][0], 16);  // one arrival per softmax warp of the pair
      mbar_init(&sm.p_full[i][1], 16);
    }
    mbar_init(&sm.o_done, 1);
    sm.abort = 0;
    fence_mbar_init();
  }
  __syncwarp();
  cluster_arrive();  // the barriers of this CTA are initialised
  if (warp == 1) {
    tma_prefetch(&P.tm_q);
    tma_prefetch(&P.tm_k);
    tma_prefetch(&P.tm_v);
    tmem_alloc_pair(&sm.tmem_base, 512);
    tc_fence_before();
  }
  attn_dep_wait(1);
  // linear grid of pairs, query-tile rank slowest: the last query tiles (the most key tiles
  // to visit) of every head, stream and batch launch first
  const int hp = P.head_pairs, rows = hp ? BM : 2 * BM, nh = hp ? G.Hq / 2 : G.Hq;
  const int item = (int)(blockIdx.x >> 1), per_rank = nh * G.q_ns * G.B;
  const int tr = fast_div(item, P.d_rank);
  const int m0 = ((G.Lq + rows - 1) / rows - 1 - tr) * rows;  // first query row of the pair
  const int hsb = item - tr * per_rank;
  const int b = fast_div(hsb, P.d_hns), hs = hsb - b * nh * G.q_ns;
  const int hx = fast_div(hs, P.d_ns), s = hs - hx * G.q_ns;
  const int h = hp ? 2 * hx + rank : hx;       // this CTA's head and first query row
  const int row0 = hp ? m0 : m0 + rank * BM;
  const int sk = s + G.kv_s0, kvh = fast_div(h, P.d_grp);
  // key tiles some row of the pair sees
  const int rq_first = m0 * G.qstep + G.qoff, rq_last = (min(m0 + rows, G.Lq) - 1) * G.qstep + G.qoff;
  const int lo = G.window > 0 ? max(0, rq_first - G.window + 1) / BN : 0;
  const int T = min(rq_last, G.Lv - 1) / BN - lo + 1;  // >= 1: every query sees its own key row
  cluster_wait();
  uint32_t tmem = 0;
  if (warp != 0) {  // the producer does not wait for the TMEM allocation
    named_bar_sync(5, NTHREADS - 32);
    tc_fence_after();
    tmem = sm.tmem_base;
  }
  volatile int* abort = &sm.abort;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      // Units in the ring: K(0), then K(t+1), V(t) for each tile: K(t) is unit 2t-1 and V(t)
      // unit 2t+2 (the last V: 2T-1, which nothing has to wait for).  Unit u takes the slot
      // of unit u - NSLOT, free once the MMAs that read it have completed.
      int u = 0, slot = 0;
      bool ok = true;
      auto take_slot = [&]() -> bool {
        if (u < NSLOT) return true;
        const int w = u - NSLOT, t = w == 0 ? 0 : (w & 1) ? (w + 1) >> 1 : (w >> 1) - 1;
        uint64_t* done = w == 0 || (w & 1) ? &sm.s_full[t & 3] : &sm.pv_done[t & 3];
        return mbar_wait(done, (t >> 2) & 1, abort, P.status);
      };
      auto load_unit = [&](int t, bool is_v) {
        if (!ok || !(ok = take_slot())) return;
        const int r0 = (lo + t) * BN;
        if (rank == 0) mbar_arrive_expect_tx(&sm.full[slot], 2 * HB * DH * 2);
        const uint32_t lb = lead_addr(&sm.full[slot]);
        if (is_v) {
          for (int c = 0; c < PC / 64; ++c)
            tma_load_pair(sm.ring[slot] + c * BN * 64, &P.tm_v, lb, rank * PC + c * 64, kvh, sk, r0, b);
        } else {
          for (int c = 0; c < DH / 64; ++c)
            tma_load_pair(sm.ring[slot] + c * HB * 64, &P.tm_k, lb, c * 64, kvh, sk, r0 + rank * HB, b);
        }
        ++u;
        if (++slot == NSLOT) slot = 0;
      };
      auto load_q = [&](int c) {  // 64 columns: S(0) starts on the first
        if (rank == 0) mbar_arrive_expect_tx(&sm.q_full[c], 2 * BM * 64 * 2);
        tma_load_pair(sm.q + c * BM * 64, &P.tm_q, lead_addr(&sm.q_full[c]), c * 64, h, s, row0, b);
      };
      load_q(0);
      load_unit(0, false);
      for (int c = 1; c < DH / 64; ++c) load_q(c);
      for (int t = 0; ok && t < T; ++t) {
        if (t + 1 < T) load_unit(t + 1, false);
        load_unit(t, true);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (first CTA)
    if (rank == 0) {
      constexpr uint32_t idS = idesc_bf16(2 * BM, BN, 0, 0);  // S = Q K^T, both K-major
      constexpr uint32_t idO = idesc_bf16(2 * BM, DH, 0, 1);  // O += P V: P in TMEM, V MN-major
      // descriptors encoded once; a block, slot or k-step adds its byte offset / 16
      const uint64_t qd = sdesc_sw128(smem_u32(sm.q), 16, 1024);
      const uint64_t kd0 = sdesc_sw128(smem_u32(sm.ring[0]), 16, 1024);
      const uint64_t vd0 = sdesc_sw128(smem_u32(sm.ring[0]), BN * 128, 1024);
      constexpr int SLOT16 = HB * DH * 2 / 16;
      auto wait_w = [&](uint64_t* bar, int par) -> bool {
        if (!__all_sync(0xffffffffu, mbar_wait(bar, par & 1, abort, P.status))) return false;
        tc_fence_after();
        return true;
      };
      auto issue_s = [&](int t, int slot) {
        const uint64_t kd = kd0 + (uint64_t)(slot * SLOT16);
#pragma unroll
        for (int kk = 0; kk < DH / 16; ++kk)
          mma2_ss(tmem + (t & 1) * BN, qd + (uint64_t)((kk >> 2) * (BM * 128 / 16) + (kk & 3) * 2),
                  kd + (uint64_t)((kk >> 2) * (HB * 128 / 16) + (kk & 3) * 2), idS, kk > 0 ? 1u : 0u);
        commit2(&sm.s_full[t & 3]);
      };
      // The first part of P also says that V(t) and K(t+2) have landed (the softmax waits for
      // them where it waits for S anyway): each wait here takes 90 cycles, 215 right after a
      // commit, and is a gap in the tensor pipe when the few MMAs queued ahead run out.
      auto issue_pv = [&](int t, int slot) -> bool {
        const uint64_t vd = vd0 + (uint64_t)(slot * SLOT16);
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          if (!wait_w(&sm.p_full[t & 1][part], t >> 1)) return false;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            // part 0: keys 0..31 of each 64-key half, part 1: keys 32..63
            const int p = k >> 1, kh = 2 * part + (k & 1), kk = 4 * p + kh;
            mma2_ts(tmem + COL_O, tmem + (t & 1) * BN + p * HB + kh * 8, vd + (uint64_t)(kk * 16 * 128 / 16), idO,
                    (t > 0 || part > 0 || k > 0) ? 1u : 0u);
          }
        }
        commit2(&sm.pv_done[t & 3]);
        return true;
      };
      auto next_slot = [](int s) { return s + 1 == NSLOT ? 0 : s + 1; };
      bool ok = wait_w(&sm.full[0], 0);
#pragma unroll 1
      for (int c = 0; c < DH / 64; ++c) {
        ok = ok && wait_w(&sm.q_full[c], 0);
        if (!ok) break;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          mma2_ss(tmem, qd + (uint64_t)(c * (BM * 128 / 16) + k * 2), kd0 + (uint64_t)(c * (HB * 128 / 16) + k * 2), idS,
                  c + k > 0 ? 1u : 0u);
      }
      if (ok) commit2(&sm.s_full[0]);
      int slot = 1;
      if (ok && T > 1) ok = wait_w(&sm.full[1], 0);
      for (int t = 0; ok && t < T; ++t) {
        // S(t+1) over P(t-1), which PV(t-1), issued before, has read
        if (t + 1 < T) {
          issue_s(t + 1, slot);
          slot = next_slot(slot);
        }
        ok = issue_pv(t, slot);
        slot = next_slot(slot);
      }
      // every MMA issued above completes before TMEM / smem are released
      commit2(&sm.o_done);
      mbar_drain(&sm.o_done, 0);
    }
  } else {
    // ------------------------------------------------------------ softmax / epilogue
    const int q4 = warp & 3, hc = (warp - 2) >> 2;
    const int row = q4 * 32 + lane;
    const int r = row0 + row;
    const int rq = r * G.qstep + G.qoff;                            // its key row
    const int rq0 = row0 * G.qstep + G.qoff;                        // key row of the tile's first query
    const int rq1 = (min(row0 + BM, G.Lq) - 1) * G.qstep + G.qoff;  // and of its last
    const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16);
    const uint32_t tO = tl + COL_O + PC * hc;
    const float c2 = P.scale_log2;
    const uint64_t c2x2 = f2pack(c2, c2);
    float m_run = -INFINITY, l_run = 0.f;  // m_run in raw score units
    bool ok = true;
    for (int t = 0; t < T; ++t) {
      const int j = lo + t;
      const uint32_t tS = tl + (uint32_t)((t & 1) * BN + HB * hc);
      const uint32_t bar_p = lead_addr(sm.p_full[t & 1]);
      if (ok && rank == 0 && warp == 2 && lane == 0) {
        // V(t) and K(t+2) have landed, before this thread's arrival on p_full
        const int uv = t + 1 < T ? 2 * t + 2 : 2 * t + 1;
        mbar_wait(&sm.full[uv % NSLOT], (uv / NSLOT) & 1, abort, P.status);
        if (t + 2 < T) mbar_wait(&sm.full[(2 * t + 3) % NSLOT], ((2 * t + 3) / NSLOT) & 1, abort, P.status);
      }
      __syncwarp();
      // tcgen05.ld/st are warp-collective: every wait result is made warp-uniform
      ok = ok && __all_sync(0xffffffffu, mbar_wait(&sm.s_full[t & 3], (t >> 2) & 1, abort, P.status));
      float x[HB], tmax = -INFINITY;
      if (ok) {
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < HB / 32; ++c) tmem_ld32(tS + c * 32, reinterpret_cast<uint32_t*>(x) + c * 32);
        tmem_ld_wait();
        // tiles holding a key past the first query's key row (the diagonal band), a key at
        // or below the last query's window edge, and the ragged last tile
        if ((j + 1) * BN - 1 > rq0 || (G.window > 0 && j * BN <= rq1 - G.window) || (j + 1) * BN > G.Lv) {
          const int k0 = j * BN + HB * hc;
          const int e_hi = min(rq, G.Lv - 1) - k0;
#pragma unroll
          for (int e = 0; e < HB; ++e)
            if (e > e_hi) x[e] = -INFINITY;
          if (G.window > 0) {
            const int e_lo = rq - G.window + 1 - k0;
#pragma unroll
            for (int e = 0; e < HB; ++e)
              if (e < e_lo) x[e] = -INFINITY;
          }
        }
        float mx[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) mx[e] = x[e];
#pragma unroll
        for (int e = 4; e < HB; ++e) mx[e & 3] = fmaxf(mx[e & 3], x[e]);
        tmax = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
        sm.part[t & 1][hc][row] = tmax;
      }
      // the two warps of these 32 rows meet here on every tile, also after a wait gave up
      named_bar_sync(1 + q4, 64);
      if (!ok) continue;
      const float m_new = fmaxf(m_run, fmaxf(tmax, sm.part[t & 1][hc ^ 1][row]));
      const bool rescale = (m_run == -INFINITY) || ((m_new - m_run) * c2 > kRescaleThreshold);
      const float m_use = rescale ? m_new : m_run;
      const float neg = (m_use == -INFINITY) ? 0.f : -m_use * c2;
      const uint64_t neg2 = f2pack(neg, neg);
      uint64_t sum2[4] = {0, 0, 0, 0};
      const bool mine = rescale && m_run != -INFINITY && t > 0;
#pragma unroll
      for (int c = 0; c < HB / 32; ++c) {
        uint32_t pk[16];
#pragma unroll
        for (int e = c * 32; e < c * 32 + 32; e += 2) {
          float a0, a1;
          f2unpack(ffma2(f2pack(x[e], x[e + 1]), c2x2, neg2), a0, a1);
          const float p0 = ex2_approx(a0), p1 = ex2_approx(a1);
          sum2[(e >> 1) & 3] = fadd2(sum2[(e >> 1) & 3], f2pack(p0, p1));
          pk[(e >> 1) & 15] = cvt_bf16x2(p0, p1);
        }
        tmem_st16(tS + c * 16, pk);
        if (c == 0 && __any_sync(0xffffffffu, mine)) {
          // O holds the PVs of every earlier tile only once PV(t-1) has completed (S(t) was
          // issued before it)
          if (!__all_sync(0xffffffffu, mbar_wait(&sm.pv_done[(t - 1) & 3], ((t - 1) >> 2) & 1, abort, P.status))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const float alpha = mine ? ex2_approx((m_run - m_use) * c2) : 1.f;
          l_run *= alpha;
#pragma unroll
          for (int d = 0; d < PC / 16; ++d) {
            uint32_t o[16];
            tmem_ld16(tO + d * 16, o);
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 16; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * alpha);
            tmem_st16(tO + d * 16, o);
          }
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_lead(bar_p + 8 * c);
      }
      float s0, s1, s2, s3;
      f2unpack(fadd2(sum2[0], sum2[1]), s0, s1);
      f2unpack(fadd2(sum2[2], sum2[3]), s2, s3);
      l_run += (s0 + s1) + (s2 + s3);
      m_run = m_use;
    }
    sm.part[T & 1][hc][row] = l_run;  // last read two tiles before the end
    named_bar_sync(1 + q4, 64);
    l_run += sm.part[T & 1][hc ^ 1][row];
    if (ok && __all_sync(0xffffffffu, mbar_wait(&sm.o_done, 0, abort, P.status))) {
      tc_fence_after();
      const float inv = 1.f / l_run;
      // O rows leave through shared memory (Q is no longer read): each thread writes its half
      // row (normalised, bf16), 16-byte units XOR-swizzled by the row, then every store
      // instruction of the warp writes 256-byte halves of two rows
      constexpr int UPR = DH * 2 / 16;  // 16-byte units per row
      uint8_t* stg = reinterpret_cast<uint8_t*>(sm.q) + q4 * (32 * DH * 2);
#pragma unroll 2
      for (int c = 0; c < PC / 32; ++c) {
        uint32_t o[32];
        tmem_ld32(tO + c * 32, o);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 32; e += 8) {
          uint4 w;
          w.x = cvt_bf16x2(__uint_as_float(o[e + 0]) * inv, __uint_as_float(o[e + 1]) * inv);
          w.y = cvt_bf16x2(__uint_as_float(o[e + 2]) * inv, __uint_as_float(o[e + 3]) * inv);
          w.z = cvt_bf16x2(__uint_as_float(o[e + 4]) * inv, __uint_as_float(o[e + 5]) * inv);
          w.w = cvt_bf16x2(__uint_as_float(o[e + 6]) * inv, __uint_as_float(o[e + 7]) * inv);
          const int u = hc * (UPR / 2) + c * 4 + e / 8;
          *reinterpret_cast<uint4*>(stg + lane * (DH * 2) + ((u ^ (lane & 7)) << 4)) = w;
        }
      }
      __syncwarp();
      bf16* base = P.o + (((long long)b * G.q_nL + s) * G.Hq + h) * DH;
      const long long rstride = (long long)G.q_rs * G.Hq * DH;  // elements between query rows
      const int r0 = row0 + q4 * 32, u = hc * (UPR / 2) + (lane & 15);
#pragma unroll 8
      for (int i = lane >> 4; i < 32; i += 2)
        if (r0 + i < G.Lq)
          *reinterpret_cast<uint4*>(base + (long long)(r0 + i) * rstride + u * 8) =
              *reinterpret_cast<const uint4*>(stg + i * (DH * 2) + ((u ^ (i & 7)) << 4));
      if (hc == 0 && r < G.Lq)
        P.lse[((long long)b * G.Hq + h) * G.q_nL + (long long)r * G.q_rs + s] = (m_run * c2 + log2f(l_run)) * kLn2;
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
}  // namespace tcfwd256

cudaError_t launch_sfa_fwd_tc256(const void* q, const void* k, const void* v, void* o, float* lse,
                                 const SfaGeom& g, float scale, int32_t* status, cudaStream_t st) {
  using namespace tcfwd256;
  Params p;
  if (!make_rows_tmap(&p.tm_q, q, query_geom(g), g.Hq, DH, BM) || !make_rows_tmap(&p.tm_k, k, g, g.Hkv, DH, HB) ||
      !make_rows_tmap(&p.tm_v, v, g, g.Hkv, DH, BN))
    return cudaErrorInvalidValue;
  p.o = (bf16*)o;
  p.lse = lse;
  p.g = g;
  p.scale_log2 = scale * kLog2e;
  p.status = status;
  p.head_pairs = (g.Hq / g.Hkv) % 2 == 0;
  const int rows = p.head_pairs ? BM : 2 * BM, nh = p.head_pairs ? g.Hq / 2 : g.Hq;
  p.d_rank = make_fast_div((uint32_t)(nh * g.q_ns * g.B));
  p.d_hns = make_fast_div((uint32_t)(nh * g.q_ns));
  p.d_ns = make_fast_div((uint32_t)g.q_ns);
  p.d_grp = make_fast_div((uint32_t)(g.Hq / g.Hkv));
  cudaError_t e = cudaFuncSetAttribute(fwd256_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e != cudaSuccess) return e;
  const unsigned grid = 2 * (unsigned)((g.Lq + rows - 1) / rows) * (unsigned)(nh * g.q_ns * g.B);
  return launch_attn(fwd256_kernel, grid, NTHREADS, kSmemBytes, st, p);
}

}  // namespace hdsfa
