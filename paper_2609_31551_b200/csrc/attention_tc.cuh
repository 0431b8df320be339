// Block-diagonal (variable-length) softmax attention on tcgen05 tensor cores with the probabilities staged in shared memory:
// a cross-check of the default kernel (attention_rr.cuh), selected with attention variant 2.
//
// One work unit = (item, head, 256 query rows) = two 128-row query tiles A and B that share every
// K/V tile.  Keys and values come from the same item only: the key loop stops at the item's last
// 128-key tile, the keys past the item's end are masked to -inf (probability exactly 0) and their value rows are cleared or
// left out of P V (0 x Inf or NaN is not 0).
//
//   warp 0       TMA producer: Q tiles (double buffered across units), K/V tiles through a ring
//   warp 1       UMMA issuer:  S = Q K^T (128 x 128 x {64|80}) into TMEM, O += P V (128 x {64|80} x 128) in TMEM
//   warps 2, 3   idle (they complete the first warpgroup, whose registers are handed to the softmax warps)
//   warps 4..7   softmax warpgroup of tile A: one thread per query row
//   warps 8..11  softmax warpgroup of tile B
//
// A softmax thread reads its row of S from TMEM, keeps a running reference maximum m and sum l, and writes
// P = exp2((s - m) * scale) as bf16 to shared memory, K-major with 128-byte swizzle.  The reference maximum only moves when
// the row maximum grows by more than 2^8 in the exponent; then the thread rescales its O row in TMEM.  Final O / l is
// written as bf16.
// Persistent: gridDim.x = sm_budget CTAs; the units are dealt to them in rounds of gridDim.x, alternate rounds in
// opposite directions (the host sorts the units by decreasing cost).
#pragma once
#include "attention_rr.cuh"
#include "ptx.cuh"

namespace eas {

constexpr int kTcThreads = 384;

struct AttnTcParams {
  CUtensorMap map_lo;   // qkv [T, 3d], box {64 columns, 128 rows}, 128-byte swizzle
  CUtensorMap map_hi;   // box {16 columns, 128 rows}, 32-byte swizzle (head_dim 80: columns 64..79)
  bf16* out;
  long long ldo;
  int d_model, n_heads;
  float scale_log2;     // log2(e) / sqrt(head_dim)
  int n_items, total_units;
  int item_start[128];
  int item_len[128];
  int unit_prefix[129];
  uint32_t* status;
  int early_launch;       // see pdl_launch_dependents
};

template <int HD>
struct AttnTcSmem {
  static constexpr int HI = HD - 64;                       // 0 or 16 extra columns
  static constexpr int kLoBytes = kTcTile * 128;           // 128 rows x 64 bf16
  static constexpr int kHiBytes = kTcTile * HI * 2;        // 128 rows x 16 bf16
  static constexpr int kTileBytes = kLoBytes + kHiBytes;   // a Q, K or V tile
  static constexpr int kStages = HD == 64 ? 3 : 2;
  static constexpr int kKvOff = 4 * kTileBytes;            // Q: [2 buffers][2 tiles]; K/V: [stages][K, V]
  static constexpr int kPOff = kKvOff + kStages * 2 * kTileBytes;   // [2 tiles][2 k-blocks of 16 KB]
  static constexpr int kBarOff = kPOff + 2 * 32768;
  static constexpr int kBytes = kBarOff + 512 + 1024;      // barriers + alignment slack
  static_assert(kBytes <= 232448, "exceeds the shared memory of an SM");
  // TMEM columns: S_A, S_B (128 each), O_A, O_B (64, or 128 of which 80 are used)
  static constexpr int kOCol0 = 2 * kTcTile, kOStride = HD == 64 ? 64 : 128;
  static_assert(kOCol0 + 2 * kOStride <= 512, "tensor memory columns");
};

// Register re-balancing between warpgroups.  The pool is the CTA's launch allocation (168 x 384 registers): the
// sum over warpgroups of 128 x their limit must stay BELOW it, or setmaxnreg.inc waits forever.
constexpr int kRegsLight = 112, kRegsSoftmax = 192;
static_assert(128 * kRegsLight + 256 * kRegsSoftmax < 168 * 384, "setmaxnreg budget exceeds the CTA's register allocation");

struct UnitInfo {
  int head, q0, S, n_kv, n_q;
  long long row0;
};
// `cursor` is the caller's item index of its previous unit: units are visited in increasing order, so the item is
// found by stepping forward (usually zero or one step) instead of searching.
__device__ __forceinline__ UnitInfo decode_unit(const AttnTcParams& p, int unit, int& cursor) {
  int lo = cursor;
  while (lo + 1 < p.n_items && p.unit_prefix[lo + 1] <= unit) ++lo;
  cursor = lo;
  UnitInfo u;
  u.S = p.item_len[lo];
  u.row0 = p.item_start[lo];
  u.n_kv = (u.S + kTcTile - 1) / kTcTile;
  const int r = unit - p.unit_prefix[lo];
  const int pairs = (u.S + 2 * kTcTile - 1) / (2 * kTcTile);
  u.head = r / pairs;
  u.q0 = (r - u.head * pairs) * 2 * kTcTile;       // pair index varies fastest: neighbours share K and V in L2
  u.n_q = (u.q0 + kTcTile < u.S) ? 2 : 1;
  return u;
}

template <int HD>
__global__ void __launch_bounds__(kTcThreads, 1) attn_tc_kernel(const __grid_constant__ AttnTcParams p) {
  using L = AttnTcSmem<HD>;
  constexpr int HI = L::HI;
  constexpr int NST = L::kStages;
  extern __shared__ uint8_t smem_raw_attn[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw_attn) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
  uint64_t* q_full = bars;                 // [2]
  uint64_t* q_empty = bars + 2;            // [2]
  uint64_t* k_full = bars + 4;             // [NST]
  uint64_t* v_full = bars + 4 + NST;       // [NST]
  uint64_t* kv_empty = bars + 4 + 2 * NST; // [NST]
  uint64_t* s_full = bars + 4 + 3 * NST;   // [2]
  uint64_t* p_ready = s_full + 2;          // [2]
  uint64_t* pv_done = s_full + 4;          // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_full + 6);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1);
      mbar_init(&s_full[i], 1); mbar_init(&p_ready[i], 4); mbar_init(&pv_done[i], 1);
    }
    for (int i = 0; i < NST; ++i) { mbar_init(&k_full[i], 1); mbar_init(&v_full[i], 1); mbar_init(&kv_empty[i], 1); }
    *abort_flag = 0;
    mbar_fence_init();
    tma_prefetch_desc(&p.map_lo);
    if (HI) tma_prefetch_desc(&p.map_hi);
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
  pdl_wait();

  // this CTA's unit of a round; increasing in `round`
  auto unit_at = [&](uint32_t round) -> int {
    const int g = static_cast<int>(gridDim.x), b = static_cast<int>(blockIdx.x);
    return static_cast<int>(round) * g + ((round & 1u) ? g - 1 - b : b);
  };
  auto q_tile = [&](int buf, int t) { return smem + (buf * 2 + t) * L::kTileBytes; };
  auto k_tile = [&](int s) { return smem + L::kKvOff + s * 2 * L::kTileBytes; };
  auto v_tile = [&](int s) { return smem + L::kKvOff + s * 2 * L::kTileBytes + L::kTileBytes; };
  auto p_tile = [&](int w) { return smem + L::kPOff + w * 32768; };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    setmaxnreg_dec<kRegsLight>();
    if (lane == 0) {
      uint32_t kv_it = 0, u_cnt = 0;
      bool ok = true;
      int cursor = 0;
      for (int unit = unit_at(0); unit < p.total_units && ok; unit = unit_at(++u_cnt)) {
        const UnitInfo u = decode_unit(p, unit, cursor);
        const int qb = u_cnt & 1;
        if (!mbar_wait(&q_empty[qb], ((u_cnt >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
        mbar_expect_tx(&q_full[qb], u.n_q * L::kTileBytes);
        for (int t = 0; t < u.n_q; ++t) {
          const int xq = u.head * HD, y = static_cast<int>(u.row0) + u.q0 + t * kTcTile;
          tma_load_2d(q_tile(qb, t), &p.map_lo, &q_full[qb], xq, y);
          if (HI) tma_load_2d(q_tile(qb, t) + L::kLoBytes, &p.map_hi, &q_full[qb], xq + 64, y);
        }
        for (int j = 0; j < u.n_kv; ++j, ++kv_it) {
          const int s = kv_it % NST;
          if (!mbar_wait(&kv_empty[s], ((kv_it / NST) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
          const int x = p.d_model + u.head * HD, y = static_cast<int>(u.row0) + j * kTcTile;
          mbar_expect_tx(&k_full[s], L::kTileBytes);
          tma_load_2d(k_tile(s), &p.map_lo, &k_full[s], x, y);
          if (HI) tma_load_2d(k_tile(s) + L::kLoBytes, &p.map_hi, &k_full[s], x + 64, y);
          mbar_expect_tx(&v_full[s], L::kTileBytes);
          tma_load_2d(v_tile(s), &p.map_lo, &v_full[s], x + p.d_model, y);
          if (HI) tma_load_2d(v_tile(s) + L::kLoBytes, &p.map_hi, &v_full[s], x + p.d_model + 64, y);
        }
      }
      // the last hand-backs of the K/V stages and Q buffers: asynchronous arrivals, in before the CTA's shared memory passes on
      for (uint32_t e = kv_it; e < kv_it + NST && ok; ++e) ok = mbar_wait(&kv_empty[e % NST], ((e / NST) & 1u) ^ 1u, abort_flag);
      for (uint32_t e = u_cnt; e < u_cnt + 2 && ok; ++e) ok = mbar_wait(&q_empty[e & 1], ((e >> 1) & 1u) ^ 1u, abort_flag);
      if (!ok) {
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000) {}     // let loads in flight land before the CTA retires
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ UMMA issuer
    setmaxnreg_dec<kRegsLight>();
    if (lane == 0) {
      constexpr uint32_t idesc_s = make_idesc_bf16(128, kTcTile, 0, 0);     // S = Q K^T, both K-major
      constexpr uint32_t idesc_o_lo = make_idesc_bf16(128, 64, 0, 1);   // O[:, 0:64] += P V, V is MN-major
      constexpr uint32_t idesc_o_hi = make_idesc_bf16(128, 16, 0, 1);   // O[:, 64:80]
      uint32_t kv_it = 0, u_cnt = 0;
      uint32_t n_pv[2] = {0, 0};
      bool ok = true;
      auto issue_s = [&](int w, int qb, int s) {
        const uint32_t qa = smem_u32(q_tile(qb, w));
        const uint32_t ka = smem_u32(k_tile(s));
        const uint64_t ad = make_smem_desc(qa, 16, 1024, kSwizzle128B);
        const uint64_t bd = make_smem_desc(ka, 16, 1024, kSwizzle128B);
        const uint32_t d = tmem_base + w * kTcTile;
#pragma unroll
        for (int k = 0; k < 4; ++k) umma_bf16_ss(d, ad + 2 * k, bd + 2 * k, idesc_s, k != 0);
        if (HI) {
          const uint64_t ah = make_smem_desc(qa + L::kLoBytes, 16, 256, kSwizzle32B);
          const uint64_t bh = make_smem_desc(ka + L::kLoBytes, 16, 256, kSwizzle32B);
          umma_bf16_ss(d, ah, bh, idesc_s, 1);
        }
        umma_commit(&s_full[w]);
      };
      // rows of the V tile that belong to the item; the rest of the last 16 that P V multiplies in is cleared (by this thread,
      // once a tile: before tile A's P V)
      auto clear_behind = [&](int s, int rows) {
        for (int c = rows * 8; c < (rows + 15) / 16 * 16 * 8; ++c) *reinterpret_cast<uint4*>(v_tile(s) + c * 16) = make_uint4(0u, 0u, 0u, 0u);
        if (HI)
          for (int c = rows * 2; c < (rows + 15) / 16 * 16 * 2; ++c) *reinterpret_cast<uint4*>(v_tile(s) + L::kLoBytes + c * 16) = make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async_smem();
      };
      auto issue_pv = [&](int w, int s, bool accumulate, int rows) {
        const uint32_t va = smem_u32(v_tile(s));
        const uint32_t d = tmem_base + L::kOCol0 + w * L::kOStride;
#pragma unroll
        for (int ks = 0; ks < kTcTile / 16; ++ks) {        // 16 keys per step
          if (ks * 16 >= rows) break;
          const uint64_t bd = make_smem_desc(va + ks * 2048, 1024, 1024, kSwizzle128B);
          const uint32_t acc = (accumulate || ks != 0) ? 1u : 0u;
          const uint32_t pa = smem_u32(p_tile(w));
          const uint64_t ad = make_smem_desc(pa + (ks >> 2) * 16384 + (ks & 3) * 32, 16, 1024, kSwizzle128B);
          umma_bf16_ss(d, ad, bd, idesc_o_lo, acc);
          if (HI) {
            const uint64_t bh = make_smem_desc(va + L::kLoBytes + ks * 512, 256, 256, kSwizzle32B);
            umma_bf16_ss(d + 64, ad, bh, idesc_o_hi, acc);
          }
        }
        umma_commit(&pv_done[w]);
        ++n_pv[w];
      };
      int cursor = 0;
      for (int unit = unit_at(0); unit < p.total_units && ok; unit = unit_at(++u_cnt)) {
        const UnitInfo u = decode_unit(p, unit, cursor);
        const int qb = u_cnt & 1;
        if (!mbar_wait(&q_full[qb], (u_cnt >> 1) & 1u, abort_flag)) { ok = false; break; }
        if (!mbar_wait(&k_full[kv_it % NST], (kv_it / NST) & 1u, abort_flag)) { ok = false; break; }
        tc_fence_after_sync();
        for (int w = 0; w < u.n_q; ++w) issue_s(w, qb, kv_it % NST);
        for (int j = 0; j < u.n_kv && ok; ++j, ++kv_it) {
          const bool last = j + 1 == u.n_kv;
          const int s = kv_it % NST, sn = (kv_it + 1) % NST;
          for (int w = 0; w < u.n_q; ++w) {
            // P(w, j) is in shared memory, S(w) has been read, O(w) has been rescaled if it had to be
            if (!mbar_wait(&p_ready[w], n_pv[w] & 1u, abort_flag)) { ok = false; break; }
            // the next scores first: the softmax of the next tile overlaps P V of this one
            if (!last) {
              if (!mbar_wait(&k_full[sn], ((kv_it + 1) / NST) & 1u, abort_flag)) { ok = false; break; }
              tc_fence_after_sync();
              issue_s(w, qb, sn);
            }
            if (!mbar_wait(&v_full[s], (kv_it / NST) & 1u, abort_flag)) { ok = false; break; }
            tc_fence_after_sync();
            const int rows = min(kTcTile, u.S - j * kTcTile);
            if (w == 0 && rows % 16 != 0) clear_behind(s, rows);
            issue_pv(w, s, j != 0, rows);
          }
          if (ok) umma_commit(&kv_empty[s]);
        }
        if (ok) umma_commit(&q_empty[qb]);
      }
    }
  } else if (warp < 4) {
    setmaxnreg_dec<kRegsLight>();
  } else {
    // ------------------------------------------------------------------ softmax warpgroups
    setmaxnreg_inc<kRegsSoftmax>();
    const int w = (warp - 4) >> 2;                 // 0: tile A, 1: tile B
    const int quarter = warp & 3;                  // TMEM lane quarter of this warp
    const int row = quarter * 32 + lane;           // query row inside the tile == TMEM lane
    const uint32_t lane_addr = static_cast<uint32_t>(quarter * 32) << 16;
    const uint32_t s_addr = tmem_base + lane_addr + w * kTcTile;
    const uint32_t o_addr = tmem_base + lane_addr + L::kOCol0 + w * L::kOStride;
    uint8_t* p_row = p_tile(w) + row * 128;
    const int sw = row & 7;
    uint32_t n = 0;                                // tiles processed by this warpgroup
    bool ok = true;
    int cursor = 0;
    uint32_t round = 0;
    for (int unit = unit_at(0); unit < p.total_units && ok; unit = unit_at(++round)) {
      const UnitInfo u = decode_unit(p, unit, cursor);
      if (w >= u.n_q) continue;                     // this warpgroup has no tile in the unit
      float m_used = -INFINITY, l = 0.f;
      for (int j = 0; j < u.n_kv; ++j, ++n) {
        if (!mbar_wait(&s_full[w], n & 1u, abort_flag)) { ok = false; break; }
        tc_fence_after_sync();
        const int valid = min(kTcTile, u.S - j * kTcTile);     // keys of this tile that belong to the item
        uint32_t sr[kTcTile];                                  // the whole score row
        __syncwarp();
        tmem_ld_32x32_at<0>(s_addr, sr);
        tmem_ld_32x32_at<32>(s_addr, sr);
        tmem_ld_32x32_at<64>(s_addr, sr);
        tmem_ld_32x32_at<96>(s_addr, sr);
        tmem_ld_wait();
        if (valid < kTcTile) {                                 // last tile of the item: keys past its end
#pragma unroll
          for (int i = 0; i < kTcTile; ++i) if (i >= valid) sr[i] = 0xff800000u;   // -inf
        }
        float mx = -INFINITY;
#pragma unroll
        for (int i = 0; i < kTcTile; i += 2) mx = fmax3(mx, __uint_as_float(sr[i]), __uint_as_float(sr[i + 1]));
        // reference maximum: moves only when the row maximum grew by more than the threshold
        float corr = 1.0f;
        bool rescale = false;
        if (j == 0) {
          m_used = mx;
        } else if ((mx - m_used) * p.scale_log2 > kRescaleThreshold) {
          corr = fast_ex2((m_used - mx) * p.scale_log2);
          m_used = mx;
          rescale = true;
        }
        l *= corr;
        const float mb = m_used * p.scale_log2;
        uint32_t pk[kTcTile / 2];
#pragma unroll
        for (int i = 0; i < kTcTile / 2; ++i) {
          const float p0 = fast_ex2(fmaf(__uint_as_float(sr[2 * i]), p.scale_log2, -mb));
          const float p1 = fast_ex2(fmaf(__uint_as_float(sr[2 * i + 1]), p.scale_log2, -mb));
          l += p0 + p1;
          pk[i] = pack_bf16x2(p0, p1);
        }
        // The previous P V must be complete before P is overwritten or O is touched.
        if (n > 0 && !mbar_wait(&pv_done[w], (n - 1) & 1u, abort_flag)) { ok = false; break; }
        tc_fence_after_sync();
        if (__any_sync(0xffffffffu, rescale)) {
#pragma unroll 1
          for (int c = 0; c < HD / 16; ++c) {
            uint32_t o[16];
            __syncwarp();
            tmem_ld_32x16(o_addr + c * 16, o);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * corr);
            tmem_st_32x8_from(o_addr + c * 16, o);
            tmem_st_32x8_from(o_addr + c * 16 + 8, o + 8);
          }
          tmem_st_wait();
        }
        // P row: 2 k-blocks of 64 keys, each row 128 bytes, 16-byte chunks XOR-swizzled by (row & 7)
#pragma unroll
        for (int cc = 0; cc < 16; ++cc) {
          const int kblk = cc >> 3, ch = cc & 7;
          *reinterpret_cast<uint4*>(p_row + kblk * 16384 + ((ch ^ sw) << 4)) = make_uint4(pk[cc * 4], pk[cc * 4 + 1], pk[cc * 4 + 2], pk[cc * 4 + 3]);
        }
        fence_proxy_async_smem();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_ready[w]);
      }
      if (!ok) break;
      // the unit's last P V
      if (!mbar_wait(&pv_done[w], (n - 1) & 1u, abort_flag)) { ok = false; break; }
      tc_fence_after_sync();
      const float inv = 1.0f / l;
      const int qrow = u.q0 + w * kTcTile + row;
      uint4* dst = reinterpret_cast<uint4*>(p.out + (u.row0 + qrow) * p.ldo + u.head * HD);
#pragma unroll
      for (int c = 0; c < HD / 16; ++c) {
        uint32_t o[16], pkd[8];
        __syncwarp();
        tmem_ld_32x16(o_addr + c * 16, o);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 8; ++i) pkd[i] = pack_bf16x2(__uint_as_float(o[2 * i]) * inv, __uint_as_float(o[2 * i + 1]) * inv);
        if (qrow < u.S) {
          dst[2 * c] = make_uint4(pkd[0], pkd[1], pkd[2], pkd[3]);
          dst[2 * c + 1] = make_uint4(pkd[4], pkd[5], pkd[6], pkd[7]);
        }
      }
      tc_fence_before_sync();                       // the O reads are complete before the next p_ready lets P V overwrite O
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
