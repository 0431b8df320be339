// Block-diagonal softmax attention with two query tiles in flight and the scores of each computed two steps ahead.
// Same tiles, same 80-key steps in the same order, hence the same bits as attention_rr.cuh.
#pragma once
#include <type_traits>

#include "attention_rr.cuh"

namespace eas {

template <int HD>
struct AttnPpSmem {
  static constexpr int kKeys = 80;
  static constexpr int kWg = 2;                            // softmax warpgroups, tiles per unit
  static constexpr int kKStages = 6, kVStages = HD == 64 ? 6 : 3;
  static constexpr int kRegsLight = 112, kRegsSoftmax = 192, kRegsLaunch = 168;
  static constexpr int HI = HD - 64;                       // 0 or 16 extra columns
  static constexpr int kThreads = 128 * (1 + kWg);
  static constexpr int kLoBytes = 128 * 128;               // Q tile: 128 rows x 64 bf16
  static constexpr int kQBytes = kLoBytes + 128 * HI * 2;  // + 128 rows x 16 bf16, 32-byte swizzle
  static constexpr int kAtomBytes = kKeys * 128;           // keys x 64 bf16
  static constexpr int kKTxBytes = kAtomBytes + kKeys * HI * 2;
  static constexpr int kKBytes = (kKTxBytes + 1023) / 1024 * 1024;
  static constexpr int kVBytes = kAtomBytes * (HI ? 2 : 1);   // head_dim 80: 128 columns wide, as in attention_rr.cuh
  static constexpr int kKOff = kWg * 2 * kQBytes, kVOff = kKOff + kKStages * kKBytes;
  static constexpr int kBarOff = kVOff + kVStages * kVBytes;
  static constexpr int kBytes = kBarOff + 512 + 1024;      // barriers + alignment slack
  static_assert(kBytes <= 232448, "exceeds the shared memory of an SM");
  static_assert(kBytes > 116224, "a second CTA must not fit beside this one");
  static_assert(kQBytes % 1024 == 0 && kVBytes % 1024 == 0 && kAtomBytes % 1024 == 0, "tiles start on swizzle-atom boundaries");
  // tensor-memory columns of warpgroup w from w * kColStride: two score buffers (P over the scores it comes from), O
  static constexpr int kOCol = 2 * kKeys, kColStride = kOCol + HD;
  static_assert(kWg * kColStride <= 512, "tensor memory columns");
  static_assert(128 * kRegsLight + 128 * kWg * kRegsSoftmax <= kThreads * kRegsLaunch, "setmaxnreg budget exceeds the CTA's register allocation");
  static_assert(kThreads * kRegsLaunch <= 65536, "registers");
};

template <int HD>
__global__ void __launch_bounds__(AttnPpSmem<HD>::kThreads, 1) attn_pp_kernel(const __grid_constant__ AttnRrParams p) {
  using L = AttnPpSmem<HD>;
  constexpr int HI = L::HI, NK = L::kKStages, NV = L::kVStages, NWG = L::kWg, KEYS = L::kKeys;
  extern __shared__ uint8_t smem_raw_attn[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw_attn) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
  uint64_t* q_full = bars;                 // [NWG][2]
  uint64_t* s_full = q_full + 2 * NWG;     // [NWG][2] by score buffer: the step's scores and the P V two steps before are complete
  uint64_t* p_ready = s_full + 2 * NWG;    // [NWG][2] P stored, O rescaled if it had to be
  uint64_t* k_full = p_ready + 2 * NWG;    // [NK]
  uint64_t* k_empty = k_full + NK;         // [NK] every issuer hands every stage back
  uint64_t* v_full = k_empty + NK;         // [NV]
  uint64_t* v_empty = v_full + NV;         // [NV]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(v_empty + NV);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  static_assert((6 * NWG + 2 * NK + 2 * NV) * 8 + 8 <= 512, "barrier area");

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2 * NWG; ++i) { mbar_init(&q_full[i], 1); mbar_init(&s_full[i], 1); mbar_init(&p_ready[i], 4); }
    for (int i = 0; i < NK; ++i) { mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], NWG); }
    for (int i = 0; i < NV; ++i) { mbar_init(&v_full[i], 1); mbar_init(&v_empty[i], NWG); }
    *abort_flag = 0;
    mbar_fence_init();
    tma_prefetch_desc(&p.map_q_lo);
    tma_prefetch_desc(&p.map_k_lo);
    if (HI) { tma_prefetch_desc(&p.map_q_hi); tma_prefetch_desc(&p.map_k_hi); }
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  if (p.early_launch) pdl_launch_dependents();

  auto unit_at = [&](uint32_t round) { return attn_unit_at(round); };
  auto q_tile = [&](int w, uint32_t b) { return smem + (w * 2 + b) * L::kQBytes; };
  auto k_tile = [&](uint32_t g) { return smem + L::kKOff + (g % NK) * L::kKBytes; };
  auto v_tile = [&](uint32_t g) { return smem + L::kVOff + (g % NV) * L::kVBytes; };
  attn_warm_parameters<NWG, KEYS>(p);
  pdl_wait();

  if (warp == 0 || warp == 3) {
    // ------------------------------------------------------------------ producers: warp 0 loads K, warp 3 V
    setmaxnreg_dec<L::kRegsLight>();
    if (lane == 0) {
      const bool is_k = warp == 0;
      const uint32_t n_st = is_k ? NK : NV;
      uint64_t* empty = is_k ? k_empty : v_empty;
      uint32_t g = 0, s = 0, ph = 1, round = 0;
      bool ok = true;
      int cursor = 0;
      for (int unit = unit_at(0); unit < p.total_units && ok; unit = unit_at(++round)) {
        const RrUnit u = attn_decode<NWG, KEYS>(p, unit, cursor);
        for (int j = 0; j < u.n_kv && ok; ++j)
          for (int st = 0; st < u.n_streams; ++st, ++g) {
            if (!mbar_wait(&empty[s], ph, abort_flag)) { ok = false; break; }
            // The first K tile (and the Q tiles, loaded by the issuers) ahead of everything else: the rings would fill with 150 KB
            // beside them, two thousand cycles at an SM's rate.
            if (g == (is_k ? 1u : 0u) && !mbar_wait(&k_full[0], 0, abort_flag)) { ok = false; break; }
            const int x = (u.head0 + st) * HD, y = u.row0 + j * KEYS;
            if (is_k) {
              mbar_expect_tx(&k_full[s], L::kKTxBytes);
              tma_load_2d(k_tile(s), &p.map_k_lo, &k_full[s], p.d_model + x, y);
              if (HI) tma_load_2d(k_tile(s) + L::kAtomBytes, &p.map_k_hi, &k_full[s], p.d_model + x + 64, y);
            } else {
              mbar_expect_tx(&v_full[s], L::kVBytes);
              tma_load_2d(v_tile(s), &p.map_k_lo, &v_full[s], 2 * p.d_model + x, y);
              if (HI) tma_load_2d(v_tile(s) + L::kAtomBytes, &p.map_k_lo, &v_full[s], 2 * p.d_model + x + 64, y);
            }
            if (++s == n_st) { s = 0; ph ^= 1u; }
          }
      }
      // The last hand-backs of the stages are asynchronous arrivals (UMMA commits) that nothing else waits for: they have to be
      // in before the CTA's shared memory passes to another one.  (Never used stages pass at once.)
      for (uint32_t e = 0; e < n_st && ok; ++e) {
        ok = mbar_wait(&empty[s], ph, abort_flag);
        if (++s == n_st) { s = 0; ph ^= 1u; }
      }
      if (!ok) {
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000) {}     // let loads in flight land before the CTA retires
      }
    }
  } else if (warp <= NWG) {
    // ------------------------------------------------------------------ UMMA issuers, one warp per warpgroup
    setmaxnreg_dec<L::kRegsLight>();
    const int w = warp - 1;
    constexpr uint32_t idesc_s = make_idesc_bf16(128, KEYS, 0, 0);         // S = Q K^T, both K-major
    constexpr uint32_t idesc_o = make_idesc_bf16(128, HD, 0, 1);           // O += P V, V is MN-major
    const uint32_t tm = tmem_base + w * L::kColStride;
    uint32_t kp = 0, vp = 0;                     // ring positions handed back so far
    uint32_t t = 0, ts = 0;                      // steps: P V issued, scores issued
    uint32_t tile = 0;                           // tiles begun (P V): its Q is in buffer tile & 1
    bool ok = true;

    auto hand_back_k = [&](uint32_t to) -> bool {
      for (; kp < to; ++kp) {
        if (!warp_mbar_wait(&k_full[kp % NK], (kp / NK) & 1u, abort_flag)) return false;
        if (elect_one()) mbar_arrive(&k_empty[kp % NK]);
        __syncwarp();
      }
      return true;
    };
    auto hand_back_v = [&](uint32_t to) -> bool {
      for (; vp < to; ++vp) {
        if (!warp_mbar_wait(&v_full[vp % NV], (vp / NV) & 1u, abort_flag)) return false;
        if (elect_one()) mbar_arrive(&v_empty[vp % NV]);
        __syncwarp();
      }
      return true;
    };
    auto load_q = [&](const RrUnit& u, uint32_t which) {       // Q of the warpgroup's tile number `which`
      const int head = (u.r0 + w) / u.nt, y = u.row0 + ((u.r0 + w) - head * u.nt) * kTcTile;
      if (elect_one()) {
        const uint32_t b = which & 1u;
        mbar_expect_tx(&q_full[w * 2 + b], L::kQBytes);
        tma_load_2d(q_tile(w, b), &p.map_q_lo, &q_full[w * 2 + b], head * HD, y);
        if (HI) tma_load_2d(q_tile(w, b) + L::kLoBytes, &p.map_q_hi, &q_full[w * 2 + b], head * HD + 64, y);
      }
      __syncwarp();
    };
    auto clear_behind = [&](uint32_t g, int rows) {            // see attention_rr.cuh
      uint8_t* v = v_tile(g);
#pragma unroll 4
      for (int c = rows * 8 + lane; c < KEYS * 8; c += 32)      // 16-byte chunks, 8 a row
        *reinterpret_cast<uint4*>(v + c * 16) = make_uint4(0u, 0u, 0u, 0u);
      if (HI) {                                                // columns 64..79: two swizzled chunks a row of the second atom
#pragma unroll 2
        for (int c = rows * 2 + lane; c < KEYS * 2; c += 32)
          *reinterpret_cast<uint4*>(v + L::kAtomBytes + (c >> 1) * 128 + (((c & 1) ^ ((c >> 1) & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
      }
      fence_proxy_async_smem();                                // generic-proxy stores -> visible to the tensor core's operand reads
      __syncwarp();
    };

    uint32_t base = 0, round = 0;                // ring position of the current unit's first K/V tile
    int cursor = 0, cursor_s = 0;
    RrUnit u{}, un{}, us{};                      // this unit, the next one, the one the scores have come to
    bool has = unit_at(0) < p.total_units, has_next = false;
    if (has) un = attn_decode<NWG, KEYS>(p, unit_at(0), cursor);
    while (has && ok) {
      u = un;
      has_next = unit_at(round + 1) < p.total_units;
      if (has_next) un = attn_decode<NWG, KEYS>(p, unit_at(round + 1), cursor);
      if (w >= u.n_q) {
        // no tile in this unit: its stages as they land
        const uint32_t end = base + static_cast<uint32_t>(u.n_kv * u.n_streams);
        while (vp < end && ok) ok = hand_back_k(vp + 1) && hand_back_v(vp + 1);
        base = end;
        ++round;
        has = has_next;
        continue;
      }
      // ---- a chain: tiles of this warpgroup in consecutive units; the scores run two steps ahead through it
      if (t != ts) {                             // the warpgroup has seen the two bare commits of the chain before
        for (int k = 0; k < 2 && ok; ++k, ++t) ok = warp_mbar_wait(&p_ready[w * 2 + (t & 1u)], (t >> 1) & 1u, abort_flag);
        if (!ok) break;
      }
      uint32_t base_s = base, round_s = round, tile_s = tile;
      int js = 0;
      bool s_on = true;
      us = u;
      cursor_s = cursor;                         // (only moves forward: `un` may be decoded again)
      load_q(u, tile);
      if (has_next && w < un.n_q) load_q(un, tile + 1);
      // scores of the next step (or, behind the chain's last one, a bare commit): s_full also says that all P V issued are complete
      auto next_s = [&]() -> bool {
        if (!s_on) {
          if (elect_one()) umma_commit(&s_full[w * 2 + (ts & 1u)]);
          __syncwarp();
          ++ts;
          return true;
        }
        const uint32_t ns = static_cast<uint32_t>(us.n_streams);
        const uint32_t g = base_s + static_cast<uint32_t>(js) * ns + static_cast<uint32_t>((us.r0 + w) / us.nt - us.head0);
        if (js == 0 && !warp_mbar_wait(&q_full[w * 2 + (tile_s & 1u)], (tile_s >> 1) & 1u, abort_flag)) return false;
        if (!hand_back_k(g) || !warp_mbar_wait(&k_full[g % NK], (g / NK) & 1u, abort_flag)) return false;
        kp = g + 1;
        tc_fence_after_sync();
        if (elect_one()) {
          const uint32_t qa = smem_u32(q_tile(w, tile_s & 1u)), ka = smem_u32(k_tile(g)), d = tm + (ts & 1u) * KEYS;
          const uint64_t ad = make_smem_desc(qa, 16, 1024, kSwizzle128B);
          const uint64_t bd = make_smem_desc(ka, 16, 1024, kSwizzle128B);
#pragma unroll
          for (int k = 0; k < 4; ++k) umma_bf16_ss(d, ad + 2 * k, bd + 2 * k, idesc_s, k != 0);
          if (HI) {
            const uint64_t ah = make_smem_desc(qa + L::kLoBytes, 16, 256, kSwizzle32B);
            const uint64_t bh = make_smem_desc(ka + L::kAtomBytes, 16, 256, kSwizzle32B);
            umma_bf16_ss(d, ah, bh, idesc_s, 1);
          }
          umma_commit(&s_full[w * 2 + (ts & 1u)]);
          umma_commit(&k_empty[g % NK]);
        }
        __syncwarp();
        ++ts;
        if (++js == us.n_kv) {
          js = 0;
          base_s += static_cast<uint32_t>(us.n_kv) * ns;
          s_on = false;
          if (unit_at(round_s + 1) < p.total_units) {
            us = attn_decode<NWG, KEYS>(p, unit_at(++round_s), cursor_s);
            s_on = w < us.n_q;
            ++tile_s;
          }
        }
        return true;
      };
      ok = next_s() && next_s();
      bool chain = true;
      while (chain && ok) {                      // tile by tile
        const uint32_t ns = static_cast<uint32_t>(u.n_streams), st = static_cast<uint32_t>((u.r0 + w) / u.nt - u.head0);
        for (int j = 0; j < u.n_kv; ++j) {
          const bool last = j + 1 == u.n_kv;
          const uint32_t g = base + static_cast<uint32_t>(j) * ns + st;
          if (!hand_back_v(g) || !warp_mbar_wait(&v_full[g % NV], (g / NV) & 1u, abort_flag)) { ok = false; break; }
          vp = g + 1;
          if (last && u.S % KEYS != 0) clear_behind(g, u.S - j * KEYS);
          if (!warp_mbar_wait(&p_ready[w * 2 + (t & 1u)], (t >> 1) & 1u, abort_flag)) { ok = false; break; }
          tc_fence_after_sync();
          // 64-column swizzle atoms kAtomBytes apart (leading byte offset; head_dim 64 has one), 8-key groups 1 KB apart
          const uint64_t bd = make_smem_desc(smem_u32(v_tile(g)), L::kAtomBytes, 1024, kSwizzle128B);
          if (elect_one()) {
#pragma unroll
            for (int ks = 0; ks < KEYS / 16; ++ks)               // 16 keys: 8 columns of P, 2 KB of V
              umma_bf16_ts(tm + L::kOCol, tm + (t & 1u) * KEYS + ks * 8, bd + ks * (2048 >> 4), idesc_o, (j != 0 || ks != 0) ? 1u : 0u);
            umma_commit(&v_empty[g % NV]);
          }
          __syncwarp();
          ++t;
          if (last && has_next && w < un.n_q && unit_at(round + 2) < p.total_units) {
            // this tile's scores are complete (the warpgroup has read them): its Q buffer takes the tile after the next
            int c = cursor;
            const RrUnit u2 = attn_decode<NWG, KEYS>(p, unit_at(round + 2), c);
            if (w < u2.n_q) load_q(u2, tile + 2);
          }
          if (!next_s()) { ok = false; break; }
        }
        if (!ok) break;
        ++tile;
        base += static_cast<uint32_t>(u.n_kv) * ns;
        chain = has_next && w < un.n_q;
        if (!chain) ok = hand_back_k(base) && hand_back_v(base);
        ++round;
        has = has_next;
        if (chain) {
          u = un;
          has_next = unit_at(round + 1) < p.total_units;
          if (has_next) un = attn_decode<NWG, KEYS>(p, unit_at(round + 1), cursor);
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax warpgroups
    setmaxnreg_inc<L::kRegsSoftmax>();
    const int w = (warp - 4) >> 2;
    const int quarter = warp & 3;                  // TMEM lane quarter of this warp
    const uint32_t tm = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + w * L::kColStride;
    const uint32_t o_addr = tm + L::kOCol;
    const uint64_t scale2 = pack2(p.scale_log2, p.scale_log2);
    uint32_t t = 0;                                // steps done
    bool ok = true;
    // the finished tile whose output is still in tensor memory
    bool pend = false;
    bf16* pend_dst = nullptr;                      // nullptr: the row is past the item's end
    float pend_l = 1.f;
    auto step_full = [&](uint32_t step) -> bool { return warp_mbar_wait(&s_full[w * 2 + (step & 1u)], (step >> 1) & 1u, abort_flag); };
    auto flush_output = [&]() {
      const float inv = 1.0f / pend_l;
      uint4* dst = reinterpret_cast<uint4*>(pend_dst);
#pragma unroll 1
      for (int c = 0; c < HD / 32; ++c) {
        uint32_t o[32];
        __syncwarp();
        tmem_ld_32x32_at<0>(o_addr + c * 32, o);
        tmem_ld_wait_16<0>(o); tmem_ld_tie_16<16>(o);
        store_row<32>(o, inv, dst, c * 4);
      }
      if constexpr (HD % 32 != 0) {
        uint32_t o[16];
        __syncwarp();
        tmem_ld_32x16(o_addr + HD / 32 * 32, o);
        tmem_ld_wait_16<0>(o);
        store_row<16>(o, inv, dst, HD / 32 * 4);
      }
      __syncwarp();
      pend = false;
    };
    // the chain is over: the two commits behind its scores say that its last P V are complete; the issuer may then use the barriers again
    auto end_chain = [&]() -> bool {
      for (int k = 0; k < 2; ++k, ++t) {
        if (!step_full(t)) return false;
        if (k == 1) {
          tc_fence_after_sync();
          flush_output();
          tc_fence_before_sync();
        }
        __syncwarp();
        mbar_arrive_if(&p_ready[w * 2 + (t & 1u)], lane == 0);
      }
      return true;
    };

    float m_used = 0.f;
    uint64_t l2[2] = {0, 0};                        // row sum, two packed accumulators
    bool begun = false;                             // the tile has a reference maximum
    // The reference maximum moves only when the row maximum grew by more than the threshold (the first step: always); true if a
    // row's that has sums against the old one did, which then wants `rescale_rows`.
    float m_old = 0.f;
    bool moved = false;
    auto take_max = [&](float mx) -> bool {
      m_old = m_used;
      moved = !begun || (mx - m_used) * p.scale_log2 > kRescaleThreshold;
      m_used = moved ? mx : m_used;
      return __ballot_sync(0xffffffffu, moved && begun) != 0u;
    };
    auto settle_output = [&](bool rescale) -> bool {
      // O is read or changed: the P V of the step before has to be complete, which the next step's commit says
      if (!step_full(t + 1)) return false;
      tc_fence_after_sync();
      if (pend) flush_output();
      if (rescale) {
        const float corr = moved ? fast_ex2((m_old - m_used) * p.scale_log2) : 1.0f;
        const uint64_t corr2 = pack2(corr, corr);
        l2[0] = fmul2(l2[0], corr2);
        l2[1] = fmul2(l2[1], corr2);
#pragma unroll 1
        for (int c = 0; c < HD / 8; ++c) {
          uint32_t o[8];
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                       : "=r"(o[0]), "=r"(o[1]), "=r"(o[2]), "=r"(o[3]), "=r"(o[4]), "=r"(o[5]), "=r"(o[6]), "=r"(o[7]) : "r"(o_addr + c * 8) : "memory");
          asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(o[0]), "+r"(o[1]), "+r"(o[2]), "+r"(o[3]), "+r"(o[4]), "+r"(o[5]), "+r"(o[6]), "+r"(o[7])::"memory");
#pragma unroll
          for (int i = 0; i < 8; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * corr);
          tmem_st_32x8_from(o_addr + c * 8, o);
        }
      }
      return true;
    };
    int cursor = 0;
    uint32_t round = 0;
    for (int unit = unit_at(0); unit < p.total_units && ok; unit = unit_at(++round)) {
      const RrUnit u = attn_decode<NWG, KEYS>(p, unit, cursor);
      if (w >= u.n_q) {                             // no tile in this unit
        if (pend) ok = end_chain();
        continue;
      }
      l2[0] = l2[1] = 0;
      begun = false;
      // a step whose first N keys hold all that is left of the item (N = 80: any step)
      auto step = [&](auto width, int left) -> bool {
        constexpr int N = decltype(width)::value;
        if (!step_full(t)) return false;
        tc_fence_after_sync();
        const uint32_t s_addr = tm + (t & 1u) * KEYS;
        uint32_t s[N], pk[KEYS / 2];
        tmem_ld_32x32_at<0>(s_addr, s);
        if constexpr (N == KEYS) {
          tmem_ld_32x32_at<32>(s_addr, s);
          tmem_ld_32x16_at<64>(s_addr, s);
        }
        tmem_ld_wait_16<0>(s); tmem_ld_tie_16<16>(s);
        if constexpr (N == KEYS) { tmem_ld_tie_16<32>(s); tmem_ld_tie_16<48>(s); tmem_ld_tie_16<64>(s); }
        if (__builtin_expect(left < N, N != KEYS)) {           // keys past the item's end
#pragma unroll
          for (int i = 0; i < N; ++i) if (i >= left) s[i] = 0xff800000u;   // -inf
        }
        const bool rescale = take_max(max_of<0, N>(s));
        const float mb = m_used * p.scale_log2;
        const uint64_t nmb2 = pack2(-mb, -mb);
        uint64_t ls[2] = {0, 0};
        exps<0, N>(s, pk, ls, scale2, nmb2);
#pragma unroll
        for (int i = N / 2; i < KEYS / 2; ++i) pk[i] = 0u;
        if (__builtin_expect(pend || rescale, 0) && !settle_output(rescale)) return false;
        l2[0] = fadd2(l2[0], ls[0]);
        l2[1] = fadd2(l2[1], ls[1]);
        // P row: two bf16 per column of this thread's lane, over the scores
        __syncwarp();
        tmem_st_32x32_from(s_addr, pk);
        tmem_st_32x8_from(s_addr + 32, pk + 32);
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        mbar_arrive_if(&p_ready[w * 2 + (t & 1u)], lane == 0);
        ++t;
        begun = true;
        return true;
      };
      int left = u.S;
#pragma unroll 1
      for (; left > 32 && ok; left -= KEYS) ok = step(std::integral_constant<int, KEYS>{}, left);
      if (left > 0 && ok) ok = step(std::integral_constant<int, 32>{}, left);
      if (!ok) break;
      pend = true;
      float l0, l1, l3, l4;
      unpack2(l2[0], l0, l1);
      unpack2(l2[1], l3, l4);
      pend_l = (l0 + l1) + (l3 + l4);
      const int head = (u.r0 + w) / u.nt, qrow = ((u.r0 + w) - head * u.nt) * kTcTile + quarter * 32 + lane;
      pend_dst = qrow < u.S ? p.out + static_cast<long long>(u.row0 + qrow) * p.ldo + head * HD : nullptr;
    }
    if (ok && pend) end_chain();
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0 && *abort_flag) atomicCAS(p.status, DEV_OK, DEV_ERR_WAIT_TIMEOUT);
}

}  // namespace eas
