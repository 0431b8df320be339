// Block-diagonal (variable-length) softmax attention on tcgen05 tensor cores: the default kernel.
//
// A query tile is 128 rows of one head of one item.  A work unit is up to three consecutive query tiles of one item, counted
// head by head; a softmax warpgroup (one thread per query row) works on each.  The key loop walks the item's keys 80 at a
// time; keys past the item's end are masked to probability exactly 0 and their value rows (the next item's) are cleared, since
// 0 x Inf or NaN is not 0: an item's output does not depend on what is packed behind it.  The
// tiles of a unit may belong to several heads (an item of 577 tokens has 5 query tiles a head): each head of the unit is a
// "stream" of K/V tiles of its own, shared by its tiles.
//
//   warp 0       TMA producer of K and V tiles (ring)
//   warps 1..3   UMMA issuers, one per warpgroup: S = Q K^T (128 x 80) into TMEM, O += P V (128 x head_dim) in TMEM; they also
//                load the warpgroup's Q tiles (one buffer each, refilled as soon as its last scores are complete)
//   warps 4..15  three softmax warpgroups
//
// What bounds it, and why three tiles: a tile's chain (scores -> row maximum -> exponentials -> P to tensor memory -> P V and
// the next scores -> back) takes 1750 cycles a step of 80 keys when a tile is alone, of which the exponentials need 640 and the
// tensor pipe 320-400: mostly latency, so what counts is the number of tiles in flight.  Three take 2450 cycles a step
// together (the special-function unit 1920 of them); two with 128 (112) keys a step and P in columns of its own, the former
// kernel, 3100 (2780).  Tensor memory holds three because P takes S's own columns (dead once the row is in registers):
// 3 x (80 + head_dim) columns.  The scores of a tile's next step then have to wait for its P V, but the other warpgroups'
// exponentials fill that time; UMMAs complete in order, so "scores ready" also says that the warpgroup's previous P V is
// complete, and a step has one wait.  Each warpgroup has an issuer of its own: one issuer for all (about 900 cycles of waits,
// issues and commits a step) was what the warpgroups waited for (1.37 times the time).
// Measured, same session, former kernel -> this one: 4 x 8192 tokens, 16 heads of 64: 1493 -> 1265 us; 2 x 8192, heads of 80:
// 803 -> 735 us; ragged 256 ... 4900, heads of 80: 338 -> 272 us; 32 x 577, heads of 64: 106 -> 89 us.
// In forward passes the board sits at its power cap, where instructions cost time even if their pipe has room: taking a
// quarter of the exponentials to the FMA pipe (a cubic), which is neutral in short runs, is 2-3 % slower in 0.3 s runs
// (32768 tokens, heads of 80: 6.03 ms without, 6.22 with), so all of them are on the special-function unit.
// Not better: four warpgroups (64 keys at head_dim 64, 48 at 80), P in columns of its own with 64 or 48 keys and three tiles,
// no row maximum while the standing reference is safe.
//
// OWN_P, the variant for little work (the host's plan decides): two tiles at most, P in columns of its own
// (2 x (80 + 40 + head_dim) columns) and two Q buffers a tile, so that the next scores are issued as soon as the row has
// been read and are there when the exponentials are done: a step of a tile alone takes 1480 instead of 1750 cycles.  Same
// 80-key steps in the same order: the same bits.  One item, kernel time: 577 tokens, 16 heads of 64: 12.1 -> 10.3 us; 1500 tokens, 20
// heads of 64: 27.5 -> 25.7; 468 tokens, 16 heads of 80: 11.5 -> 10.1; 2304 tokens: 39.9 -> 37.6.  With three tiles' worth of work the
// third tile is worth more (4 x 8192 tokens: 1275 us against 1500).
//
// The reference maximum only moves when the row maximum grows by more than 2^8 in the exponent; then the thread rescales
// its O row in TMEM.  Final O / l is written as bf16.  A row's arithmetic does not depend on its unit.
// Persistent: gridDim.x = sm_budget CTAs; the units are dealt to them in rounds of gridDim.x, alternate rounds in
// opposite directions (the host sorts the units by decreasing cost: a fixed direction would hand CTA 0 the costliest
// unit of every round).
#pragma once
#include "ptx.cuh"

namespace eas {

constexpr int kTcTile = 128;            // query rows per tile
constexpr float kRescaleThreshold = 8.0f;
constexpr uint32_t kWarmPiece = 16384;

struct AttnRrParams {
  CUtensorMap map_q_lo;   // qkv [T, 3d], box {64 columns, 128 rows}, 128-byte swizzle
  CUtensorMap map_q_hi;   // box {16 columns, 128 rows}, 32-byte swizzle (head_dim 80: columns 64..79)
  CUtensorMap map_k_lo;   // box {64 columns, KEYS rows}, 128-byte swizzle (K and V tiles)
  CUtensorMap map_k_hi;   // box {16 columns, KEYS rows}, 32-byte swizzle
  bf16* out;
  long long ldo;
  int d_model, n_heads;
  float scale_log2;       // log2(e) / sqrt(head_dim)
  int n_items, total_units;
  int item_start[128];
  int item_len[128];
  int unit_prefix[129];
  // an item's units: item_full of them with kWg query tiles, the others with small_tiles (<= kWg): see attention_plan
  int item_full[128];
  int small_tiles;
  // Constant memory that later launches read (weights), towards L2 beside this one: each CTA asks for its share
  const uint8_t* warm[4];
  uint32_t warm_bytes[4];
  uint32_t* status;
  int early_launch;       // see pdl_launch_dependents
};

template <int HD, bool OWN_P>
struct AttnRrSmem {
  static constexpr int kKeys = 80;
  static constexpr int kWg = OWN_P ? 2 : 3;                // softmax warpgroups, tiles per unit
  static constexpr int kQBufs = OWN_P ? 2 : 1;             // Q tiles per warpgroup
  static constexpr int kStages = HD == 64 ? 6 : 4;
  static constexpr int kRegsLight = OWN_P ? 112 : 80, kRegsSoftmax = OWN_P ? 192 : 144, kRegsLaunch = OWN_P ? 168 : 128;
  static constexpr int HI = HD - 64;                       // 0 or 16 extra columns
  static constexpr int kThreads = 128 * (1 + kWg);
  static constexpr int kLoBytes = 128 * 128;               // Q tile: 128 rows x 64 bf16
  static constexpr int kHiBytes = 128 * HI * 2;            // 128 rows x 16 bf16, 32-byte swizzle
  static constexpr int kQBytes = kLoBytes + kHiBytes;
  static constexpr int kAtomBytes = kKeys * 128;           // keys x 64 bf16
  static constexpr int kKHiBytes = kKeys * HI * 2;
  static constexpr int kKTxBytes = kAtomBytes + kKHiBytes;
  static constexpr int kKBytes = (kKTxBytes + 1023) / 1024 * 1024;
  // head_dim 80: V is loaded 128 columns wide (two 64-column boxes; the extra 48 columns belong to the next head, or are
  // zero past the last one) so that P V is ONE UMMA per 16 keys, N = 80 across the two swizzle atoms.
  static constexpr int kVBytes = kAtomBytes * (HI ? 2 : 1);
  static constexpr int kStageBytes = kKBytes + kVBytes;
  static constexpr int kKvOff = kWg * kQBufs * kQBytes;
  static constexpr int kBarOff = kKvOff + kStages * kStageBytes;
  static constexpr int kBytes = kBarOff + 512 + 1024;      // barriers + alignment slack
  static_assert(kBytes <= 232448, "exceeds the shared memory of an SM");
  static_assert(kBytes > 116224, "a second CTA must not fit beside this one");
  static_assert(kQBytes % 1024 == 0 && kStageBytes % 1024 == 0 && kAtomBytes % 1024 == 0, "tiles start on swizzle-atom boundaries");
  // TMEM columns of warpgroup w from w * kColStride: S, (own) P: two bf16 per column, O.  P otherwise takes S's first columns.
  static constexpr int kPCol = OWN_P ? kKeys : 0, kOCol = kKeys + (OWN_P ? kKeys / 2 : 0), kColStride = kOCol + HD;
  static_assert(kWg * kColStride <= 512, "tensor memory columns");
  static_assert(kKeys == 80, "five UMMA k-steps; a row of scores is 32 + 32 + 16 registers");
  static_assert(kWg <= 3, "the issuers are warps 1 .. kWg of the first warpgroup");
  static_assert(kStages > kWg, "an issuer looks at most kWg ring positions ahead of the stage it holds");
  // setmaxnreg: the pool is the CTA's launch allocation
  static_assert(128 * kRegsLight + 128 * kWg * kRegsSoftmax <= kThreads * kRegsLaunch, "setmaxnreg budget exceeds the CTA's register allocation");
  static_assert(kThreads * kRegsLaunch <= 65536, "registers");
};

// Wait for this thread's tensor-memory loads, tied to registers they fill so that no use can move ahead of it.
template <int OFF, int N>
__device__ __forceinline__ void tmem_ld_wait_16(uint32_t (&r)[N]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[OFF]), "+r"(r[OFF + 1]), "+r"(r[OFF + 2]), "+r"(r[OFF + 3]), "+r"(r[OFF + 4]), "+r"(r[OFF + 5]), "+r"(r[OFF + 6]), "+r"(r[OFF + 7]),
                 "+r"(r[OFF + 8]), "+r"(r[OFF + 9]), "+r"(r[OFF + 10]), "+r"(r[OFF + 11]), "+r"(r[OFF + 12]), "+r"(r[OFF + 13]), "+r"(r[OFF + 14]), "+r"(r[OFF + 15])
               ::"memory");
}
// ties 16 more registers behind the wait above (no instruction)
template <int OFF, int N>
__device__ __forceinline__ void tmem_ld_tie_16(uint32_t (&r)[N]) {
  asm volatile("" : "+r"(r[OFF]), "+r"(r[OFF + 1]), "+r"(r[OFF + 2]), "+r"(r[OFF + 3]), "+r"(r[OFF + 4]), "+r"(r[OFF + 5]), "+r"(r[OFF + 6]), "+r"(r[OFF + 7]),
                    "+r"(r[OFF + 8]), "+r"(r[OFF + 9]), "+r"(r[OFF + 10]), "+r"(r[OFF + 11]), "+r"(r[OFF + 12]), "+r"(r[OFF + 13]), "+r"(r[OFF + 14]), "+r"(r[OFF + 15])
               ::"memory");
}

struct RrUnit {
  int r0, nt, n_q, head0, n_streams, S, n_kv, row0;
};
// this CTA's unit of a round; increasing in `round`
__device__ __forceinline__ int attn_unit_at(uint32_t round) {
  const int g = static_cast<int>(gridDim.x), b = static_cast<int>(blockIdx.x);
  return static_cast<int>(round) * g + ((round & 1u) ? g - 1 - b : b);
}
// units are visited in increasing order: the item is found by stepping forward from the previous unit's (`cursor`)
template <int FULL, int KEYS>
__device__ __forceinline__ RrUnit attn_decode(const AttnRrParams& p, int unit, int& cursor) {
  int lo = cursor;
  while (lo + 1 < p.n_items && p.unit_prefix[lo + 1] <= unit) ++lo;
  cursor = lo;
  RrUnit u;
  u.S = p.item_len[lo];
  u.row0 = p.item_start[lo];
  u.nt = (u.S + kTcTile - 1) / kTcTile;
  u.n_kv = (u.S + KEYS - 1) / KEYS;
  const int k = unit - p.unit_prefix[lo], full = p.item_full[lo];
  u.r0 = k < full ? k * FULL : full * FULL + (k - full) * p.small_tiles;
  u.n_q = min(k < full ? FULL : p.small_tiles, p.n_heads * u.nt - u.r0);
  u.head0 = u.r0 / u.nt;
  u.n_streams = (u.r0 + u.n_q - 1) / u.nt - u.head0 + 1;
  return u;
}

template <int HD, bool OWN_P>
__global__ void __launch_bounds__(AttnRrSmem<HD, OWN_P>::kThreads, 1) attn_rr_kernel(const __grid_constant__ AttnRrParams p) {
  using L = AttnRrSmem<HD, OWN_P>;
  constexpr int HI = L::HI, NST = L::kStages, NWG = L::kWg, KEYS = L::kKeys;
  extern __shared__ uint8_t smem_raw_attn[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw_attn) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
  uint64_t* q_full = bars;                 // [NWG][kQBufs]
  uint64_t* s_full = q_full + 2 * NWG;     // [NWG] scores of a step complete (and everything issued before them)
  uint64_t* p_ready = s_full + NWG;        // [NWG] P stored, O rescaled if it had to be
  uint64_t* s_free = p_ready + NWG;        // [NWG] own P: the warpgroup has read the scores out of tensor memory
  uint64_t* pv_done = s_free + NWG;        // [NWG] own P: P V of a step complete
  uint64_t* k_full = pv_done + NWG;        // [NST]
  uint64_t* v_full = k_full + NST;         // [NST]
  uint64_t* kv_empty = v_full + NST;       // [NST] every issuer hands every stage back
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(kv_empty + NST);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  static_assert((6 * NWG + 3 * NST) * 8 + 8 <= 512, "barrier area");

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NWG * L::kQBufs; ++i) mbar_init(&q_full[i], 1);
    for (int i = 0; i < NWG; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_ready[i], 4); mbar_init(&s_free[i], 4); mbar_init(&pv_done[i], 1); }
    for (int i = 0; i < NST; ++i) { mbar_init(&k_full[i], 1); mbar_init(&v_full[i], 1); mbar_init(&kv_empty[i], NWG); }
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
  // The parameters that the first unit's decoding reads come from a cold constant cache, some 650 cycles in all: ahead of the grid
  // dependency's wait they cost nothing (the kernel alone, 4 x 8192 tokens 1325 -> 1311 us, 8 items of 577 27.8 -> 27.5; whole calls move
  // by less than their runs differ).  The variant for little work
  // has its SMs to itself and is ready too late for that (one item of 468 tokens 8.92 -> 9.00).
  if (!OWN_P && attn_unit_at(0) < p.total_units) {
    int cursor = 0;
    const RrUnit u = attn_decode<NWG, KEYS>(p, attn_unit_at(0), cursor);
    asm volatile("" ::"r"(u.r0), "r"(u.n_q), "r"(u.n_streams), "r"(u.row0), "r"(u.n_kv));
  }
  pdl_wait();

  auto unit_at = [&](uint32_t round) { return attn_unit_at(round); };
  auto decode = [&](int unit, int& cursor) { return attn_decode<NWG, KEYS>(p, unit, cursor); };
  auto stream_of = [](const RrUnit& u, int w) { return (u.r0 + w) / u.nt - u.head0; };
  auto q_tile = [&](int w, uint32_t b) { return smem + (w * L::kQBufs + b) * L::kQBytes; };
  auto k_tile = [&](int s) { return smem + L::kKvOff + s * L::kStageBytes; };
  auto v_tile = [&](int s) { return smem + L::kKvOff + s * L::kStageBytes + L::kKBytes; };

  if (warp == 0) {
    // ------------------------------------------------------------------ K / V producer
    setmaxnreg_dec<L::kRegsLight>();
    if (lane == 0) {
      uint32_t g = 0, round = 0;
      bool ok = true;
      int cursor = 0;
      auto warm_up = [&]() {
#pragma unroll 1
        for (int r = 0; r < 4; ++r)
          for (uint32_t off = blockIdx.x * kWarmPiece; off < p.warm_bytes[r]; off += gridDim.x * kWarmPiece)
            l2_prefetch(p.warm[r] + off, min(kWarmPiece, p.warm_bytes[r] - off));
      };
      for (int unit = unit_at(0); unit < p.total_units && ok; unit = unit_at(++round)) {
        const RrUnit u = decode(unit, cursor);
        for (int j = 0; j < u.n_kv && ok; ++j)
          for (int st = 0; st < u.n_streams; ++st, ++g) {
            const int s = g % NST;
            if (g == NST) warm_up();
            if (!mbar_wait(&kv_empty[s], ((g / NST) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
            const int x = (u.head0 + st) * HD, y = u.row0 + j * KEYS;
            mbar_expect_tx(&k_full[s], L::kKTxBytes);
            tma_load_2d(k_tile(s), &p.map_k_lo, &k_full[s], p.d_model + x, y);
            if (HI) tma_load_2d(k_tile(s) + L::kAtomBytes, &p.map_k_hi, &k_full[s], p.d_model + x + 64, y);
            mbar_expect_tx(&v_full[s], L::kVBytes);
            tma_load_2d(v_tile(s), &p.map_k_lo, &v_full[s], 2 * p.d_model + x, y);
            if (HI) tma_load_2d(v_tile(s) + L::kAtomBytes, &p.map_k_lo, &v_full[s], 2 * p.d_model + x + 64, y);
          }
      }
      if (g <= NST) warm_up();
      // The last hand-backs of the stages are asynchronous arrivals (UMMA commits) that nothing else waits for: they have to be
      // in before the CTA's shared memory passes to another one.  (Never used stages pass at once.)
      for (uint32_t e = g; e < g + NST && ok; ++e) ok = mbar_wait(&kv_empty[e % NST], ((e / NST) & 1u) ^ 1u, abort_flag);
      if (!ok) {
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000) {}     // let loads in flight land before the CTA retires
      }
    }
  } else if (warp <= NWG) {
    // ------------------------------------------------------------------ UMMA issuers, one warp per warpgroup
    // The whole warp walks the steps (uniform control flow: see elect_one) and one elected lane issues.  A step: P V of
    // this step and the scores of the next as soon as P is there; what they need beside P (V, the next K, the next tile's
    // Q) is waited for before P, so that the path from P to the next scores holds one wait.  With P in columns of its own the
    // next scores come first, as soon as the warpgroup has read the previous ones.
    // An issuer sees every K/V stage of the CTA land, in order, also those of streams its tile has no part in (it hands those
    // back with a plain arrival), so that it never mistakes a barrier's phase for an earlier one.  Holding its own stage g it
    // waits for no stage past g + kWg < g + kStages (warpgroup w belongs at most to stream w, and at most kWg - 1 - w streams
    // follow its own), so the waits of the issuers have no cycle.
    setmaxnreg_dec<L::kRegsLight>();
    const int w = warp - 1;
    constexpr uint32_t QB = L::kQBufs;
    constexpr uint32_t idesc_s = make_idesc_bf16(128, KEYS, 0, 0);         // S = Q K^T, both K-major
    constexpr uint32_t idesc_o = make_idesc_bf16(128, HD, 0, 1);           // O += P V, V is MN-major
    const uint32_t tm = tmem_base + w * L::kColStride;
    uint32_t n_q = 0, n_s = 0, n_p = 0;          // Q tiles waited for, s_full phases committed, p_ready phases waited for
    bool started = false;                        // the first scores of this unit's tile are issued already
    bool owed = false;                           // the warpgroup still has to say that it has seen a bare commit
    uint32_t base = 0, round = 0;                // base: ring position of the unit's first K/V tile
    bool ok = true;
    int cursor = 0;
    RrUnit un{};
    if (unit_at(0) < p.total_units) un = decode(unit_at(0), cursor);

    auto load_q = [&](const RrUnit& u) {         // into the buffer of the next tile to be waited for
      const int head = (u.r0 + w) / u.nt, y = u.row0 + ((u.r0 + w) - head * u.nt) * kTcTile;
      if (elect_one()) {
        const uint32_t b = n_q % QB;
        mbar_expect_tx(&q_full[w * QB + b], L::kQBytes);
        tma_load_2d(q_tile(w, b), &p.map_q_lo, &q_full[w * QB + b], head * HD, y);
        if (HI) tma_load_2d(q_tile(w, b) + L::kLoBytes, &p.map_q_hi, &q_full[w * QB + b], head * HD + 64, y);
      }
      __syncwarp();
    };
    auto q_landed = [&]() -> bool {
      if (!warp_mbar_wait(&q_full[w * QB + n_q % QB], (n_q / QB) & 1u, abort_flag)) return false;
      ++n_q;
      return true;
    };
    auto k_landed = [&](uint32_t g) -> bool { return warp_mbar_wait(&k_full[g % NST], (g / NST) & 1u, abort_flag); };
    auto hand_back = [&](uint32_t from, uint32_t to) -> bool {   // stages of other streams
      for (uint32_t g = from; g < to; ++g) {
        if (!k_landed(g)) return false;
        if (elect_one()) mbar_arrive(&kv_empty[g % NST]);
        __syncwarp();
      }
      return true;
    };
    // Only the first `rows` value rows of the V tile at ring position g belong to the item: clears the others (their probabilities
    // are 0, but 0 x Inf or NaN is not).  Every issuer of the stream does so before its own P V; later ones store the zeros that
    // are there already.  Once a tile, beside the softmax of its last step and before the next tile's Q is waited for.  (P V of
    // the last step over fewer keys would have less to clear, but the branch costs every step: +1 % at 8192 keys.)
    auto clear_behind = [&](uint32_t g, int rows) {
      uint8_t* v = v_tile(g % NST);
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
    // by the elected lane: scores of the current tile (the last one waited for) against the K tile at ring position g
    auto mma_s = [&](uint32_t g) {
      const uint32_t qa = smem_u32(q_tile(w, (n_q - 1u) % QB)), ka = smem_u32(k_tile(g % NST));
      const uint64_t ad = make_smem_desc(qa, 16, 1024, kSwizzle128B);
      const uint64_t bd = make_smem_desc(ka, 16, 1024, kSwizzle128B);
#pragma unroll
      for (int k = 0; k < 4; ++k) umma_bf16_ss(tm, ad + 2 * k, bd + 2 * k, idesc_s, k != 0);
      if (HI) {
        const uint64_t ah = make_smem_desc(qa + L::kLoBytes, 16, 256, kSwizzle32B);
        const uint64_t bh = make_smem_desc(ka + L::kAtomBytes, 16, 256, kSwizzle32B);
        umma_bf16_ss(tm, ah, bh, idesc_s, 1);
      }
      umma_commit(&s_full[w]);
    };

    for (int unit = unit_at(0); unit < p.total_units && ok; unit = unit_at(++round)) {
      const RrUnit u = un;
      const bool has_next = unit_at(round + 1) < p.total_units;
      if (has_next) un = decode(unit_at(round + 1), cursor);
      const uint32_t ns = static_cast<uint32_t>(u.n_streams);
      const uint32_t next_base = base + static_cast<uint32_t>(u.n_kv) * ns;
      if (w >= u.n_q) {
        ok = hand_back(base, next_base);
        base = next_base;
        continue;
      }
      const bool chain = has_next && w < un.n_q;      // the next unit's first scores follow this unit's last ones
      const uint32_t st = static_cast<uint32_t>(stream_of(u, w)), st_next = chain ? static_cast<uint32_t>(stream_of(un, w)) : 0u;
      if (!started) {
        if (owed) {                              // the warpgroup has seen the bare commit, so s_full may be used again
          if (!warp_mbar_wait(&p_ready[w], n_p & 1u, abort_flag)) { ok = false; break; }
          ++n_p;
        }
        load_q(u);
        if (!hand_back(base, base + st) || !q_landed() || !k_landed(base + st)) { ok = false; break; }
        if (OWN_P && n_s > 0 && !warp_mbar_wait(&s_free[w], (n_s - 1u) & 1u, abort_flag)) { ok = false; break; }
        tc_fence_after_sync();
        if (elect_one()) mma_s(base + st);
        __syncwarp();
        ++n_s;
      }
      // two Q buffers: the last scores against the other one are read (s_free was waited for before this tile's first)
      if (OWN_P && chain) load_q(un);
      for (int j = 0; j < u.n_kv; ++j) {
        const bool last = j + 1 == u.n_kv;
        const bool more = !last || chain;
        const uint32_t row = base + static_cast<uint32_t>(j) * ns, g = row + st;
        const uint32_t gn = last ? next_base + st_next : g + ns;      // the K tile of the scores to come
        if (!OWN_P && last && chain) {
          // one Q buffer: free when the last scores are complete
          if (!warp_mbar_wait(&s_full[w], (n_s - 1u) & 1u, abort_flag)) { ok = false; break; }
          load_q(un);
        }
        if (!hand_back(g + 1, row + ns)) { ok = false; break; }
        if (!OWN_P && !warp_mbar_wait(&v_full[g % NST], (g / NST) & 1u, abort_flag)) { ok = false; break; }
        if (!OWN_P && last && u.S % KEYS != 0) clear_behind(g, u.S - j * KEYS);
        if (more && (!hand_back(last ? next_base : row + ns, gn) || !k_landed(gn))) { ok = false; break; }
        if (last && chain && !q_landed()) { ok = false; break; }
        if (OWN_P && more) {
          if (!warp_mbar_wait(&s_free[w], (n_s - 1u) & 1u, abort_flag)) { ok = false; break; }
          tc_fence_after_sync();
          if (elect_one()) mma_s(gn);
          __syncwarp();
          ++n_s;
        }
        if (OWN_P && !warp_mbar_wait(&v_full[g % NST], (g / NST) & 1u, abort_flag)) { ok = false; break; }
        if (OWN_P && last && u.S % KEYS != 0) clear_behind(g, u.S - j * KEYS);
        if (!warp_mbar_wait(&p_ready[w], n_p & 1u, abort_flag)) { ok = false; break; }
        ++n_p;
        tc_fence_after_sync();
        // 64-column swizzle atoms kAtomBytes apart (leading byte offset; head_dim 64 has one), 8-key groups 1 KB apart
        const uint64_t bd = make_smem_desc(smem_u32(v_tile(g % NST)), L::kAtomBytes, 1024, kSwizzle128B);
        if (elect_one()) {
#pragma unroll
          for (int ks = 0; ks < KEYS / 16; ++ks)                 // 16 keys: 8 columns of P, 2 KB of V
            umma_bf16_ts(tm + L::kOCol, tm + L::kPCol + ks * 8, bd + ks * (2048 >> 4), idesc_o, (j != 0 || ks != 0) ? 1u : 0u);
          if (OWN_P) umma_commit(&pv_done[w]);
          else if (more) mma_s(gn);
          else umma_commit(&s_full[w]);                          // bare: tells the warpgroup that its O is final
          umma_commit(&kv_empty[g % NST]);
        }
        __syncwarp();
        if (!OWN_P) ++n_s;
      }
      started = chain;
      owed = !OWN_P && !chain;
      base = next_base;
    }
  } else if (warp < 4) {
    setmaxnreg_dec<L::kRegsLight>();
  } else {
    // ------------------------------------------------------------------ softmax warpgroups
    setmaxnreg_inc<L::kRegsSoftmax>();
    const int w = (warp - 4) >> 2;
    const int quarter = warp & 3;                  // TMEM lane quarter of this warp
    const uint32_t s_addr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + w * L::kColStride;
    const uint32_t p_addr = s_addr + L::kPCol, o_addr = s_addr + L::kOCol;
    const uint64_t scale2 = pack2(p.scale_log2, p.scale_log2);
    uint32_t n = 0;                                // s_full phases waited for (own P: steps done)
    bool ok = true;
    // the finished tile whose output is still in tensor memory
    bool pend = false;
    bf16* pend_dst = nullptr;                      // nullptr: the row is past the item's end
    float pend_l = 1.f;
    auto flush_output = [&]() {
      const float inv = 1.0f / pend_l;
      uint4* dst = reinterpret_cast<uint4*>(pend_dst);
#pragma unroll 1
      for (int c = 0; c < HD / 16; ++c) {
        uint32_t o[16];
        __syncwarp();
        tmem_ld_32x16(o_addr + c * 16, o);
        tmem_ld_wait_16<0>(o);
        uint32_t pkd[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) pkd[i] = pack_bf16x2(__uint_as_float(o[2 * i]) * inv, __uint_as_float(o[2 * i + 1]) * inv);
        if (dst != nullptr) {
          dst[2 * c] = make_uint4(pkd[0], pkd[1], pkd[2], pkd[3]);
          dst[2 * c + 1] = make_uint4(pkd[4], pkd[5], pkd[6], pkd[7]);
        }
      }
      __syncwarp();
      pend = false;
    };

    int cursor = 0;
    uint32_t round = 0;
    for (int unit = unit_at(0); unit < p.total_units && ok; unit = unit_at(++round)) {
      const RrUnit u = decode(unit, cursor);
      if (w >= u.n_q) {                             // no tile in this unit
        if (pend) {
          if (!warp_mbar_wait(OWN_P ? &pv_done[w] : &s_full[w], (OWN_P ? n - 1u : n) & 1u, abort_flag)) { ok = false; break; }
          tc_fence_after_sync();
          flush_output();
          if (!OWN_P) {
            ++n;
            tc_fence_before_sync();
            __syncwarp();
            mbar_arrive_if(&p_ready[w], lane == 0);        // the issuer may use s_full[w] again
          }
        }
        continue;
      }
      float m_used = 0.f;
      uint64_t l2[2] = {0, 0};                      // row sum, two packed accumulators
      int left = u.S;                               // keys from this step on
#pragma unroll 1
      for (int j = 0; j < u.n_kv; ++j, left -= KEYS) {
        if (!warp_mbar_wait(&s_full[w], n & 1u, abort_flag)) { ok = false; break; }
        ++n;
        tc_fence_after_sync();
        if (!OWN_P && __builtin_expect(pend, 0)) flush_output();       // the previous tile's P V is complete
        uint32_t s[KEYS];
        tmem_ld_32x32_at<0>(s_addr, s);
        tmem_ld_32x32_at<32>(s_addr, s);
        tmem_ld_32x16_at<64>(s_addr, s);
        tmem_ld_wait_16<0>(s); tmem_ld_tie_16<16>(s); tmem_ld_tie_16<32>(s); tmem_ld_tie_16<48>(s); tmem_ld_tie_16<64>(s);
        if (OWN_P) {
          tc_fence_before_sync();
          __syncwarp();
          mbar_arrive_if(&s_free[w], lane == 0);
        }
        if (__builtin_expect(left < KEYS, 0)) {              // keys past the item's end
#pragma unroll
          for (int i = 0; i < KEYS; ++i) if (i >= left) s[i] = 0xff800000u;   // -inf
        }
        float mx;
        {
          float c0 = -INFINITY, c1 = -INFINITY, c2 = -INFINITY, c3 = -INFINITY;
#pragma unroll
          for (int i = 0; i < KEYS; i += 8) {
            c0 = fmax3(c0, __uint_as_float(s[i]), __uint_as_float(s[i + 1]));
            c1 = fmax3(c1, __uint_as_float(s[i + 2]), __uint_as_float(s[i + 3]));
            c2 = fmax3(c2, __uint_as_float(s[i + 4]), __uint_as_float(s[i + 5]));
            c3 = fmax3(c3, __uint_as_float(s[i + 6]), __uint_as_float(s[i + 7]));
          }
          mx = fmax3(fmaxf(c0, c1), c2, c3);
        }
        // the reference maximum moves only when the row maximum grew by more than the threshold (the first step: always)
        const float m_old = m_used;
        const bool moved = j == 0 || (mx - m_used) * p.scale_log2 > kRescaleThreshold;
        m_used = moved ? mx : m_used;
        const uint32_t rescale = __ballot_sync(0xffffffffu, moved && j != 0);
        const float mb = m_used * p.scale_log2;
        const uint64_t nmb2 = pack2(-mb, -mb);
        const uint64_t l_old[2] = {l2[0], l2[1]};
        l2[0] = l2[1] = 0;
        const uint32_t pv_ok = OWN_P ? mbar_try_wait(&pv_done[w], n & 1u) : 1u;      // the previous step's, tested ahead
        uint32_t pk[KEYS / 2];
#pragma unroll
        for (int i = 0; i < KEYS / 2; ++i) {
          const uint64_t t = ffma2(pack2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), scale2, nmb2);
          float p0, p1;
          unpack2(t, p0, p1);
          p0 = fast_ex2(p0);
          p1 = fast_ex2(p1);
          l2[i & 1] = fadd2(l2[i & 1], pack2(p0, p1));
          pk[i] = pack_bf16x2(p0, p1);
        }
        if (OWN_P) {
          // P goes where the previous step's was, and O may change: that step's P V has to be complete
          if (n > 1u && !warp_mbar_wait_tested(pv_ok, &pv_done[w], n & 1u, abort_flag)) { ok = false; break; }
          tc_fence_after_sync();
          if (__builtin_expect(pend, 0)) flush_output();
        }
        if (__builtin_expect(rescale != 0u, 0)) {
          // (the sum of this step is in l2 already and was taken against the new reference: the correction is applied to
          // what was there before, kept in l_old)
          const float corr = moved ? fast_ex2((m_old - m_used) * p.scale_log2) : 1.0f;
          const uint64_t corr2 = pack2(corr, corr);
          l2[0] = fadd2(fmul2(l_old[0], corr2), l2[0]);
          l2[1] = fadd2(fmul2(l_old[1], corr2), l2[1]);
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
        } else {
          l2[0] = fadd2(l_old[0], l2[0]);
          l2[1] = fadd2(l_old[1], l2[1]);
        }
        // P row: two bf16 per column of this thread's lane
        __syncwarp();
        tmem_st_32x32_from(p_addr, pk);
        tmem_st_32x8_from(p_addr + 32, pk + 32);
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        mbar_arrive_if(&p_ready[w], lane == 0);
      }
      if (!ok) break;
      pend = true;
      float l0, l1, l3, l4;
      unpack2(l2[0], l0, l1);
      unpack2(l2[1], l3, l4);
      pend_l = (l0 + l1) + (l3 + l4);
      const int head = (u.r0 + w) / u.nt, qrow = ((u.r0 + w) - head * u.nt) * kTcTile + quarter * 32 + lane;
      pend_dst = qrow < u.S ? p.out + static_cast<long long>(u.row0 + qrow) * p.ldo + head * HD : nullptr;
    }
    if (ok && pend) {
      if (warp_mbar_wait(OWN_P ? &pv_done[w] : &s_full[w], (OWN_P ? n - 1u : n) & 1u, abort_flag)) {
        tc_fence_after_sync();
        flush_output();
      }
    }
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
