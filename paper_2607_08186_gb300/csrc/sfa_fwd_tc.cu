// Stream-Factorized Attention forward on the sm_103a tensor cores.
//
// One CTA computes a 128-row query tile of one virtual causal problem (SfaGeom):
// in WITHIN mode the problem is one stream (rows p = t*n + s, Eq. 4), so the tile
// visits only that stream's key tiles; CROSS is causal over all nL positions
// (Fig. 2a); LOCAL adds the window (Fig. 2b).  Key tiles past the diagonal (or
// before the window) are skipped; tiles straddling a mask edge are masked in
// registers.  A final-stream problem has only the L final-stream queries (dense
// [B][L] tensors) against the same keys: query row r stands at key row
// r*qstep + qoff, which sets its tile range and mask.
//
// A CTA owns two 128-row query tiles (groups g = 0, 1).  Where a K/V group has an
// even number of query heads (GQA), they are the same rows of two of its heads, so
// both see the same key tiles and finish together; otherwise rows m0 and m0 + 128 of
// one head (the second tile then runs one key tile longer: measured as about 2 us of
// a WITHIN CTA's 35 us, the first tile's softmax warps idle meanwhile).
// Roles (320 threads):
//   warp 0      TMA producer: both Q tiles once, then the tiles K(lo), V(lo), K(lo+1),
//               V(lo+1), ... into a ring of single K or V tiles.
//   warp 1      MMA issuer: the whole warp runs the issue loop, one elected lane
//               issues; owns TMEM.  Per key tile and group: S_g = Q_g K^T (SS) into the
//               group's 128 TMEM columns, O_g += P_g V (TS: P_g read from TMEM) into its O
//               columns; the next S_g is issued after the PV that reads P_g.
//   warps 2..5, 6..9  softmax of group 0 / 1: one thread per query row (its TMEM
//               lane); online softmax in fp32 with exp2 (packed f32x2 arithmetic),
//               P packed to bf16 over the first 64 columns of S_g and released to the PV
//               in two halves, O_g rescaled in TMEM only when the running max grows by
//               more than 2^8, epilogue.
// K/V tiles use the 128-byte swizzle written by TMA.  Every mbarrier wait is bounded.
//
// What bounds it: a group's own chain P -> PV -> next S -> softmax: 1024 cycles of MMAs,
// about 300 of signals and 1300 of softmax (of those 600 are the SFU's 128 exp2 per row),
// under which the other group's 1024 cycles of MMAs run: about 2550 per key tile and group
// pair, against 2048 of MMAs.  A tensor pipe that waits costs most: the issuer holds
// about five MMAs (360 cycles) in its queue, a wait on a completed barrier takes 90
// cycles, 215 right after a commit, and a second commit 110, since barriers live in the
// shared memory that the S MMAs read at its full rate.  So between the last MMA of a batch
// and the first of the next the issuer only commits once and waits once (for P); a
// softmax warp, idle then, has waited for the K / V tiles, and ring slots are released
// where no wait follows.  K and V tiles have slots of their own, so K(j+1) is on its way
// while V(j) is in use (a two-stage ring of K and V together left S(j+1) waiting for its
// load, 3450 cycles per tile).
// Measured: 470 -> 372 us for an intra-stream layer (B=1, L=4096, n=4, 32 over 8 heads of
// dim 128), 6.26 -> 5.27 ms for a cross-stream one of 32768 positions (1.67 PFLOP/s), 110
// -> 93 us at head dim 64 (B=4, L=1501, n=3, 16 over 4 heads).  A CTA's fixed part, about
// 8500 cycles, is what separates the intra-stream layer from the tile time.
// Slower: one issuer per group (459 us: the groups' MMAs interleave and their softmaxes
// meet on the SFU), the tile waits inside the S batch (440 us) or between the halves of P
// (454 us), two single-tile CTAs per SM (463 us: K and V are loaded twice).
#include "tc_common.cuh"

namespace hdsfa {

typedef __nv_bfloat16 bf16;

namespace tcfwd {
constexpr int BM = 128, BN = 128, NG = 2, NTHREADS = 64 + NG * 128;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleThreshold = 8.0f;  // log2 units: P stays <= 256 between O rescales

template <int DH>
struct Smem {
  bf16 q[NG][BM * DH];  // per query tile: DH/64 swizzle blocks of [BM][64]
  static constexpr int NSLOT = DH == 64 ? 10 : 5;
  bf16 ring[NSLOT][BN * DH];  // one K or V tile each
  uint64_t q_full[NG], full[NSLOT], empty[NSLOT], s_full[NG], p_full[NG][2], o_done[NG], drain;
  uint32_t tmem_base;
  int abort;
};
// The layout needs 1024-byte alignment; the kernel checks the actual pad on entry.
template <int DH>
constexpr int smem_bytes() { return (int)sizeof(Smem<DH>) + 1024 < 232448 ? (int)sizeof(Smem<DH>) + 1024 : 232448; }
static_assert(sizeof(Smem<128>) <= 232448, "forward shared memory exceeds 227 KB");

struct Params {
  CUtensorMap tm_q, tm_k, tm_v;
  bf16* o;
  float* lse;
  SfaGeom g;
  float scale_log2;
  int32_t* status;
  int head_pairs;  // 1: a CTA's two query tiles are the same rows of two heads of one K/V group
  FastDiv d_rank, d_hns, d_ns, d_grp;
};

// Key-tile range [lo, hi] of the query tile starting at row m0 (hi < lo: no rows).
HD_DEVINLINE void tile_range(const SfaGeom& G, int m0, int& lo, int& hi) {
  if (m0 >= G.Lq) {
    lo = 0;
    hi = -1;
    return;
  }
  const int rq_first = m0 * G.qstep + G.qoff, rq_last = (min(m0 + BM, G.Lq) - 1) * G.qstep + G.qoff;
  lo = G.window > 0 ? max(0, rq_first - G.window + 1) / BN : 0;
  hi = min(rq_last / BN, (G.Lv - 1) / BN);
}

// TMEM columns: S_g at g*128 (P_g packed bf16 over its first 64 columns), O_g at 256 + g*DH.
// NAIVE: the naive intra-stream schedule (G.smod > 1): every tile is masked, a pair
// also needing key row = query row (mod smod); its own instantiation, so the other
// modes' softmax carries none of that code.
template <int DH, bool NAIVE>
__global__ void __launch_bounds__(NTHREADS, 1) fwd_kernel(const __grid_constant__ Params P) {
  constexpr int NSLOT = Smem<DH>::NSLOT;
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
    for (int i = 0; i < NSLOT; ++i) {
      mbar_init(&sm.full[i], 1);
      mbar_init(&sm.empty[i], 1);
    }
    for (int g = 0; g < NG; ++g) {
      mbar_init(&sm.q_full[g], 1);
      mbar_init(&sm.s_full[g], 1);
      mbar_init(&sm.p_full[g][0], 4);  // one arrival per softmax warp of the group
      mbar_init(&sm.p_full[g][1], 4);
      mbar_init(&sm.o_done[g], 1);
    }
    mbar_init(&sm.drain, 1);
    sm.abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, 512);
    tmem_relinquish();
    tc_fence_before();
  }
  attn_dep_wait(1);
  // A CTA's two query tiles: with head_pairs the same 128 rows of heads 2x and 2x+1
  // (one K/V group: both tiles see exactly the same key tiles and finish together),
  // else rows m0 and m0 + 128 of one head (the second tile sees one more key tile).
  const int hp = P.head_pairs;
  const int rows_per_cta = hp ? BM : NG * BM;
  const int ncta = (G.Lq + rows_per_cta - 1) / rows_per_cta;
  const int nh = hp ? G.Hq / NG : G.Hq;  // head slots of the grid
  // linear grid, query-tile rank slowest: the last query tiles (the most key tiles to
  // visit) of every head, stream and batch launch first
  const int per_rank = nh * G.q_ns * G.B;
  const int rank = fast_div((int)blockIdx.x, P.d_rank);
  const int mt = ncta - 1 - rank, hsb = (int)blockIdx.x - rank * per_rank;
  const int b = fast_div(hsb, P.d_hns), hs = hsb - b * nh * G.q_ns;
  const int hx = fast_div(hs, P.d_ns), s = hs - hx * G.q_ns;
  int qm[NG], hd[NG];  // first query row and head of each group's tile
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    qm[g] = hp ? mt * BM : mt * NG * BM + g * BM;
    hd[g] = hp ? NG * hx + g : hx;
  }
  const int h = hd[0];
  const int sk = s + G.kv_s0;  // stream of the key problem
  const int kvh = fast_div(h, P.d_grp);
  int lo[NG], hi[NG];
#pragma unroll
  for (int g = 0; g < NG; ++g) tile_range(G, qm[g], lo[g], hi[g]);
  // The window of a final-stream problem whose query step is wider than it can leave key
  // tiles between the two query tiles' ranges that neither of them sees.  Tiles are numbered
  // without that gap (the second tile's lie `gap` further on), so some group takes part at
  // every j: its softmax waits for the tiles on the issuer's behalf, its PV releases K(j).
  static_assert(NG == 2, "one gap");
  const int gap = hi[1] >= lo[1] ? max(0, lo[1] - hi[0] - 1) : 0;
  lo[1] -= gap;
  hi[1] -= gap;
  const int n_lo = lo[0];
  int n_hi = hi[0];
#pragma unroll
  for (int g = 1; g < NG; ++g) n_hi = max(n_hi, hi[g]);

  volatile int* abort = &sm.abort;
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
      int slot = 0, ph = 1, issued = 0;  // empty-barrier phase: the first lap does not wait
      bool ok = true;
      auto load_tile = [&](const CUtensorMap* tm, int j) {
        if (!ok || !mbar_wait(&sm.empty[slot], ph, abort, P.status)) {
          ok = false;
          return;
        }
        mbar_arrive_expect_tx(&sm.full[slot], BN * DH * 2);
        const int row = (j > hi[0] ? j + gap : j) * BN;
        for (int c = 0; c < DH / 64; ++c)
          tma_load_5d(sm.ring[slot] + c * BN * 64, tm, &sm.full[slot], c * 64, kvh, sk, row, b);
        ++issued;
        if (++slot == NSLOT) {
          slot = 0;
          ph ^= 1;
        }
      };
      auto load_q = [&](int g) {
        mbar_arrive_expect_tx(&sm.q_full[g], BM * DH * 2);
        for (int c = 0; c < DH / 64; ++c)
          tma_load_5d(sm.q[g] + c * BM * 64, &P.tm_q, &sm.q_full[g], c * 64, hd[g], s, qm[g], b);
      };
      load_q(0);
      if (n_lo <= n_hi) load_tile(&P.tm_k, n_lo);
      load_q(1);
      for (int j = n_lo; ok && j <= n_hi; ++j) {
        load_tile(&P.tm_v, j);
        if (j < n_hi) load_tile(&P.tm_k, j + 1);
      }
      // every copy this thread started lands before the CTA may exit
      for (int g = 0; g < NG; ++g) mbar_drain(&sm.q_full[g], 0);
      for (int u = max(0, issued - NSLOT); u < issued; ++u) mbar_drain(&sm.full[u % NSLOT], (u / NSLOT) & 1);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // The whole warp runs the loop (warp-uniform operands); one elected lane issues.
    constexpr uint32_t idS = idesc_bf16(BM, BN, 0, 0);  // S[q][kv] = Q K^T (both K-major)
    constexpr uint32_t idO = idesc_bf16(BM, DH, 0, 1);  // O[q][d] += P V   (P in TMEM, V MN-major)
    static_assert(BM == 128 && BN == 128 && NG == 2, "descriptor offsets below");
    // Operand descriptors are encoded once; a slot or k-step adds its byte offset / 16 to
    // the 64-bit descriptor (the address field; shared addresses stay below 256 KB), which
    // keeps the instructions between consecutive MMAs (and so the issue gaps) small.
    const uint64_t qd0 = sdesc_sw128(smem_u32(sm.q[0]), 16, 1024);
    const uint64_t kd0 = sdesc_sw128(smem_u32(sm.ring[0]), 16, 1024);
    const uint64_t vd0 = sdesc_sw128(smem_u32(sm.ring[0]), BN * 128, 1024);
    constexpr int TILE16 = BN * DH * 2 / 16;
    auto wait_w = [&](uint64_t* bar, int par) -> bool {
      if (!__all_sync(0xffffffffu, mbar_wait(bar, par & 1, abort, P.status))) return false;
      tc_fence_after();
      return true;
    };
    auto issue_s = [&](int g, int slot) {
      const uint64_t qd = qd0 + (uint64_t)(g * (BM * DH * 2 / 16)), kd = kd0 + (uint64_t)(slot * TILE16);
#pragma unroll
      for (int kk = 0; kk < DH / 16; ++kk) {
        const uint64_t off = (uint64_t)((kk >> 2) * (128 * 128 / 16) + (kk & 3) * 2);
        tc_mma_ss_w(tmem + g * 128, qd + off, kd + off, idS, kk > 0 ? 1u : 0u);
      }
      tc_commit_w(&sm.s_full[g]);
    };
    // P arrives in two halves of 64 keys: the first half's k-steps run while the softmax
    // computes the second.  The softmax publishes P(j) only after V(j) and K(j+1) have
    // landed, so the issuer waits for nothing else: each of its waits takes 90 cycles, 215
    // right after a commit, and a commit after another 110, against about 360 cycles of
    // queued MMAs.  Releases go where no wait follows at once.
    auto issue_pv = [&](int g, int j, int slot, int k_done) -> bool {
      const uint64_t vd = vd0 + (uint64_t)(slot * TILE16);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        if (!wait_w(&sm.p_full[g][hf], j - lo[g])) return false;
#pragma unroll
        for (int kk = hf * 4; kk < hf * 4 + 4; ++kk)
          tc_mma_ts_w(tmem + 256 + g * DH, tmem + g * 128 + kk * 8, vd + (uint64_t)(kk * 16 * 128 / 16), idO,
                      (j > lo[g] || kk > 0) ? 1u : 0u);
        if (hf == 0 && k_done >= 0) tc_commit_w(&sm.empty[k_done]);
      }
      return true;
    };
    auto next_slot = [](int s) { return s + 1 == NSLOT ? 0 : s + 1; };
    bool ok = true;
    int k_done = -1, v_slot = 1;  // K(j), not yet released; V(j) (K(n_lo) is in slot 0)
    if (n_hi >= n_lo) {
      ok = wait_w(&sm.full[0], 0);
      for (int g = 0; ok && g < NG; ++g) {
        ok = wait_w(&sm.q_full[g], 0);
        if (ok && lo[g] <= n_lo && n_lo <= hi[g]) issue_s(g, 0);
      }
      k_done = 0;
    }
    for (int j = n_lo; ok && j <= n_hi; ++j) {
      const int k_slot = next_slot(v_slot);  // K(j+1)
      for (int g = 0; ok && g < NG; ++g) {
        if (lo[g] <= j && j <= hi[g]) {
          if (!issue_pv(g, j, v_slot, k_done)) { ok = false; break; }
          k_done = -1;
          if (j == hi[g]) tc_commit_w(&sm.o_done[g]);
        }
        if (g == NG - 1) tc_commit_w(&sm.empty[v_slot]);
        // S of the next tile for this group reuses its S/P columns: issued after its PV
        if (j + 1 <= hi[g] && lo[g] <= j + 1) issue_s(g, k_slot);
      }
      k_done = k_slot;
      v_slot = next_slot(k_slot);
    }
    // every MMA issued above completes before TMEM / smem are released
    tc_commit_w(&sm.drain);
    mbar_drain(&sm.drain, 0);
  } else {
    // ------------------------------------------------------------ softmax / epilogue
    const int g = (warp - 2) >> 2;
    const int q4 = warp & 3;
    const int row = q4 * 32 + lane;
    const int r = qm[g] + row;
    const int hg = hd[g];
    const int rq = r * G.qstep + G.qoff;                      // its key row
    const int rq0 = qm[g] * G.qstep + G.qoff;                 // key row of the tile's first query
    // key row of its last query (a key tile above rq1 - window is inside every row's window)
    const int rq1 = (min(qm[g] + BM, G.Lq) - 1) * G.qstep + G.qoff;
    const uint32_t tl = tmem + ((uint32_t)(q4 * 32) << 16);
    const uint32_t tS = tl + g * 128, tO = tl + 256 + g * DH;
    const float c2 = P.scale_log2;
    float m_run = -INFINITY, l_run = 0.f;  // m_run in raw score units
    bool ok = true;
    for (int j = lo[g]; j <= hi[g]; ++j) {
      const int i = j - lo[g];
      const int kb = (g == 0 ? j : j + gap) * BN;  // first key row of the tile
      // this thread's arrivals on p_full also say that V(j) and K(j+1) have landed (waited
      // for here, where the softmax waits for S anyway)
      if (warp == 2 + 4 * g && lane == 0) {
        const int u = 2 * (j - n_lo) + 1;  // V(j)'s place in the ring's order
        mbar_wait(&sm.full[u % NSLOT], (u / NSLOT) & 1, abort, P.status);
        if (j < n_hi) mbar_wait(&sm.full[(u + 1) % NSLOT], ((u + 1) / NSLOT) & 1, abort, P.status);
      }
      __syncwarp();
      // tcgen05.ld/st are warp-collective: every wait result is made warp-uniform
      if (!__all_sync(0xffffffffu, mbar_wait(&sm.s_full[g], i & 1, abort, P.status))) {
        ok = false;
        break;
      }
      tc_fence_after();
      float x[BN];
#pragma unroll
      for (int c = 0; c < BN / 32; ++c) tmem_ld32(tS + c * 32, reinterpret_cast<uint32_t*>(x) + c * 32);
      tmem_ld_wait();
      // tiles holding a key past the first query's key row (the diagonal band), a key at
      // or below the last query's window edge, and the ragged last tile
      const bool need_mask = kb + BN - 1 > rq0 || (G.window > 0 && kb <= rq1 - G.window) ||
                             kb + BN > G.Lv;
      if constexpr (NAIVE) {
        // causal (no window in this schedule) and k = (rq - key row) mod smod == 0,
        // k stepped down the tile's columns
        int k = (rq - kb) % G.smod;
        if (k < 0) k += G.smod;
#pragma unroll
        for (int e = 0; e < BN; ++e) {
          if (k != 0 || kb + e > rq || kb + e >= G.Lv) x[e] = -INFINITY;
          k = k == 0 ? G.smod - 1 : k - 1;
        }
      } else if (need_mask) {
        // keys past the query's own row or the end, and (LOCAL) at or below its window edge
        const int e_hi = min(rq, G.Lv - 1) - kb;
#pragma unroll
        for (int e = 0; e < BN; ++e)
          if (e > e_hi) x[e] = -INFINITY;
        if (G.window > 0) {
          const int e_lo = rq - G.window + 1 - kb;
#pragma unroll
          for (int e = 0; e < BN; ++e)
            if (e < e_lo) x[e] = -INFINITY;
        }
      }
      float mx[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) mx[e] = x[e];
#pragma unroll
      for (int e = 8; e < BN; ++e) mx[e & 7] = fmaxf(mx[e & 7], x[e]);
      const float tmax = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])),
                               fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
      const float m_new = fmaxf(m_run, tmax);
      const bool rescale = (m_run == -INFINITY) || ((m_new - m_run) * c2 > kRescaleThreshold);
      const float m_use = rescale ? m_new : m_run;
      const float neg = (m_use == -INFINITY) ? 0.f : -m_use * c2;
      const uint64_t c2x2 = f2pack(c2, c2), neg2 = f2pack(neg, neg);
      // P (bf16 pairs) over the first 64 columns of this group's S, published in halves
      uint64_t sum2[4] = {0, 0, 0, 0};
      const bool mine = rescale && m_run != -INFINITY && i > 0;
#pragma unroll
      for (int c = 0; c < BN / 32; ++c) {
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
        if (c & 1) {
          if (c == 1 && __any_sync(0xffffffffu, mine)) {
            // O_g already holds every earlier tile's PV (its S of this tile was issued after
            // them).  Looked at here, so that the vote does not delay the exponentials.
            const float alpha = mine ? ex2_approx((m_run - m_use) * c2) : 1.f;
            l_run *= alpha;
#pragma unroll
            for (int d = 0; d < DH / 16; ++d) {
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
          if (lane == 0) mbar_arrive(&sm.p_full[g][c >> 1]);
        }
      }
      float s0, s1, s2, s3;
      f2unpack(fadd2(sum2[0], sum2[1]), s0, s1);
      f2unpack(fadd2(sum2[2], sum2[3]), s2, s3);
      l_run += (s0 + s1) + (s2 + s3);
      m_run = m_use;
    }
    if (ok && hi[g] >= lo[g] && __all_sync(0xffffffffu, mbar_wait(&sm.o_done[g], 0, abort, P.status))) {
      tc_fence_after();
      const float inv = 1.f / l_run;
      // O rows leave through shared memory: each thread writes its row (normalised,
      // bf16) into this warp's 32 rows of the group's Q buffer (no longer read: the last
      // S MMA of the group completed before o_done), 16-byte units XOR-swizzled by the
      // row; then every store instruction writes whole rows (DH*2 bytes each, 2 rows at
      // DH = 128), instead of one 16-byte piece of 32 different rows.
      constexpr int UPR = DH * 2 / 16;  // 16-byte units per row
      uint8_t* stg = reinterpret_cast<uint8_t*>(sm.q[g]) + q4 * (32 * DH * 2);
#pragma unroll
      for (int c = 0; c < DH / 32; ++c) {
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
          const int u = c * 4 + e / 8;
          *reinterpret_cast<uint4*>(stg + lane * (DH * 2) + ((u ^ (lane & 7)) << 4)) = w;
        }
      }
      __syncwarp();
      {
        const long long rstride = (long long)G.q_rs * G.Hq * DH;  // elements between query rows
        bf16* obase = P.o + (((long long)b * G.q_nL + s) * G.Hq + hg) * DH;
        const int r0 = qm[g] + q4 * 32;  // this warp's first row
#pragma unroll
        for (int i = 0; i < 32 * UPR / 32; ++i) {
          const int rr = (i * 32 + lane) / UPR, u = (i * 32 + lane) % UPR;  // row within the warp, unit
          if (r0 + rr < G.Lq)
            *reinterpret_cast<uint4*>(obase + (long long)(r0 + rr) * rstride + u * 8) =
                *reinterpret_cast<const uint4*>(stg + rr * (DH * 2) + ((u ^ (rr & 7)) << 4));
        }
      }
      if (r < G.Lq)
        P.lse[((long long)b * G.Hq + hg) * G.q_nL + (long long)r * G.q_rs + s] = (m_run * c2 + log2f(l_run)) * kLn2;
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
}  // namespace tcfwd

// --------------------------------------------------------------------- host
template <int DH, bool NAIVE>
static cudaError_t tc_fwd_impl(tcfwd::Params& p, cudaStream_t st) {
  constexpr int smem = tcfwd::smem_bytes<DH>();
  cudaError_t e =
      cudaFuncSetAttribute(tcfwd::fwd_kernel<DH, NAIVE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int rows_per_cta = p.head_pairs ? tcfwd::BM : tcfwd::NG * tcfwd::BM;
  const int nh = p.head_pairs ? p.g.Hq / tcfwd::NG : p.g.Hq;
  const unsigned grid = (unsigned)((p.g.Lq + rows_per_cta - 1) / rows_per_cta) * (unsigned)(nh * p.g.q_ns * p.g.B);
  return launch_attn(tcfwd::fwd_kernel<DH, NAIVE>, grid, tcfwd::NTHREADS, smem, st, p);
}

cudaError_t launch_sfa_fwd_tc(const void* q, const void* k, const void* v, void* o, float* lse,
                              const SfaGeom& g, int Dh, float scale, int32_t* status, cudaStream_t st) {
  tcfwd::Params p;
  if (!make_rows_tmap(&p.tm_q, q, query_geom(g), g.Hq, Dh, tcfwd::BM) ||
      !make_rows_tmap(&p.tm_k, k, g, g.Hkv, Dh, tcfwd::BN) ||
      !make_rows_tmap(&p.tm_v, v, g, g.Hkv, Dh, tcfwd::BN))
    return cudaErrorInvalidValue;
  p.o = (bf16*)o;
  p.lse = lse;
  p.g = g;
  p.scale_log2 = scale * tcfwd::kLog2e;
  p.status = status;
  p.head_pairs = (g.Hq / g.Hkv) % tcfwd::NG == 0;
  const int nh = p.head_pairs ? g.Hq / tcfwd::NG : g.Hq;
  p.d_rank = make_fast_div((uint32_t)(nh * g.q_ns * g.B));
  p.d_hns = make_fast_div((uint32_t)(nh * g.q_ns));
  p.d_ns = make_fast_div((uint32_t)g.q_ns);
  p.d_grp = make_fast_div((uint32_t)(g.Hq / g.Hkv));
  if (Dh == 64) return tc_fwd_impl<64, false>(p, st);
  return g.smod > 1 ? tc_fwd_impl<128, true>(p, st) : tc_fwd_impl<128, false>(p, st);
}

}  // namespace hdsfa
