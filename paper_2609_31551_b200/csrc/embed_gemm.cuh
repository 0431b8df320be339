// Patch embedding as an im2col-fused GEMM for sm_100a (two kernels: embed_resident_kernel for patch vectors of up to 1216 elements, at
// the end, and embed_gemm_kernel for longer ones and many short ones, described here):
//
//     x[row(m), :] = patch(m) * W_emb^T + b (+ pos[posrow(m), :])        m = patch index over the micro-batch
//
// The A operand (one row per patch: its pixels in the order channel, frame-in-patch, row, column) is never
// materialised in global memory.  Gather warps read the pixel runs of 128 patches straight from the packed images /
// clips and write them into shared memory in the layout a 128-byte-swizzled TMA tile would have, so the tensor core
// reads them through the same UMMA descriptors as any other A tile.  (TMA itself cannot fetch them: a run of a
// 14-pixel patch row is 28 bytes long and starts on a 28-byte grid, neither a multiple of 16.)
//
// Gathering is the expensive part (small scattered loads): a CTA takes a block of R patches, keeps up to kEgMaxResident
// 64-wide k-blocks of their rows resident in shared memory and runs a group of column blocks of the output against them
// while the weight tiles stream through a small TMA ring.  With many patches R is 128 and the group is all columns, so every
// patch is gathered once.  With few patches that leaves most SMs idle and one CTA's gather and column loop is the kernel's
// time (38-76 us for one image): the columns are dealt to several CTAs, which gather the same patches again, and R shrinks
// to 64 or 32 (the other rows of the 128-row UMMA tile are whatever lies in shared memory; their results are not stored), so
// that a row has 4 or 8 gather threads.  The host picks both by estimated time.
// A patch vector longer than the resident part is processed in passes over K: the first pass stores bias + position +
// partial sum, every later pass adds its partial sum to the stored row.  The passes do not depend on R or the column groups,
// so the result does not either.
//
//   warp 0        TMA producer of the weight tiles (256 rows x 64 columns per stage), lane 0
//   warp 1        UMMA issuer (128 x 256 x 16, fp32 accumulators in TMEM, two accumulator buffers), lane 0
//   warps 2..9    gather: 256 / R threads per patch row, each loads pixel pairs of a k-block (4-byte loads; a pair never
//                 straddles a run because patch edges are even) and stores swizzled 16-byte chunks; the loads of several
//                 k-blocks are in flight
//   warps 10..17  epilogue, two warps per TMEM lane quarter (half of the columns each): tcgen05.ld -> + bias (+ position row)
//                 or + stored row -> fp32 rows of the residual stream, scattered by the row map (CLS rows and item boundaries
//                 make output rows differ from patch rows)
//
// The grid is at most `sm_budget` CTAs, one per SM, walking the units (patch block, column group) blockIdx.x, + gridDim.x, ...; every output
// element is accumulated over K in one fixed order, so results do not depend on the budget.
#pragma once
#include "elementwise.cuh"
#include "ptx.cuh"

namespace eas {

constexpr int kEgThreads = 18 * 32;
constexpr int kEgGatherWarps = 8;
constexpr int kEgMaxResident = 10;                      // k-blocks of the A rows kept in shared memory per pass, at most
constexpr int kEgWStages = 2;
constexpr int kEgABytes = 128 * 64 * 2;                 // 16 KB: 128 patch rows x 64 elements
constexpr int kEgBBytes = 256 * 64 * 2;                 // 32 KB: 256 weight rows x 64 elements
// shared memory: [resident A: 10 x 16 KB, or 10 x R x 128 bytes][weight ring: 2 x 32 KB][barriers]: fills an SM's 227 KB at R = 128
// (smaller R: the last slot's tile reads past the slots, into the ring: rows of no patch)
constexpr int kEgSmemBytes = kEgMaxResident * kEgABytes + kEgWStages * kEgBBytes + 512 + 1024;   // + barriers + alignment slack
static_assert(kEgSmemBytes <= 232448, "exceeds the shared memory of an SM");

struct EmbedGemmParams {
  CUtensorMap tma_w;       // W_emb [N, K_pad] (K zero-padded to a multiple of 64), box {64, 256}, 128-byte swizzle
  const bf16* data;        // packed items: image [C, H, W]; clip [F, C, H, W]
  const bf16* bias;        // [N]
  float* x;                // residual stream [*, N]
  const int* row_map;      // [n_patches] -> row of x
  const int* pos_idx;      // [n_patches] -> row of the position table (with pos)
  const bf16* pos;         // optional position table [*, N]
  int n_patches, N;
  int k, k_pad;            // patch elements C * pt * P * P, and the same padded to a multiple of 64
  int channels, patch, tpatch;
  int merge_order;         // 0: patches in raster order; 1: merge-group-major (the four patches of a 2x2 group adjacent)
  int col_groups;          // the column blocks are dealt to this many units per patch block
  int pairs_ok;            // 1: patch edge, image widths and item offsets are even, so pixel pairs are 4-byte aligned
  int chunks_ok;           // 1: patch edge, image widths and item offsets are multiples of 8, so eight elements of a run are 16-byte aligned
  const uint32_t* table;   // [k_pad / 2] where each pixel pair of the patch vector comes from (built once per encoder)
  uint32_t* status;
  ItemTable items;         // aux_start = patch-row prefix per item
  int early_launch;       // see pdl_launch_dependents
};

// Table entry of a pixel pair (elements k, k + 1 of the patch vector): channel << 24 | frame-in-patch << 16 | py << 8 | px.
// 0xFFFFFFFF: padding behind the patch vector (zeros).
constexpr uint32_t kEgPad = 0xFFFFFFFFu;

// Fills the pair table of an architecture (create time).
__global__ void embed_table_kernel(uint32_t* table, int k, int k_pad, int patch, int tpatch) {
  const int PP = patch * patch;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < k_pad / 2; j += gridDim.x * blockDim.x) {
    const int kk = 2 * j;
    uint32_t e = kEgPad;
    if (kk < k) {
      const int plane = kk / PP, rem = kk - plane * PP;          // plane = channel * pt + frame-in-patch
      const int py = rem / patch, px = rem - py * patch;
      const int ch = plane / tpatch, f = plane - ch * tpatch;
      e = (static_cast<uint32_t>(ch) << 24) | (static_cast<uint32_t>(f) << 16) | (static_cast<uint32_t>(py) << 8) | static_cast<uint32_t>(px);
    }
    table[j] = e;
  }
}

// Where patch m lies: its first pixel in frame-in-patch 0 of channel 0, the elements between channels and between the frames of a
// clip (an item has fewer than 2^31 elements: checked by the host), and the image width.
struct EgPatch { const bf16* base; int plane_stride, frame_stride, width; };
__device__ __forceinline__ EgPatch eg_locate(const EmbedGemmParams& p, int m) {
  const int item = find_item(p.items.aux_start, p.items.n_items, m);
  const int local = m - p.items.aux_start[item];
  const int H = p.items.height[item], W = p.items.width[item];
  const int gh = H / p.patch, gw = W / p.patch;
  const int tt = local / (gh * gw);
  const int rem = local - tt * gh * gw;
  int r, c;
  if (p.merge_order) {
    const int grp = rem >> 2, within = rem & 3;
    const int hb = grp / (gw >> 1), wb = grp - hb * (gw >> 1);
    r = 2 * hb + (within >> 1);
    c = 2 * wb + (within & 1);
  } else {
    r = rem / gw;
    c = rem - r * gw;
  }
  EgPatch e;
  e.width = W;
  e.plane_stride = H * W;
  const bool clip = p.tpatch > 1 || p.items.frames[item] > 1;
  e.frame_stride = clip ? e.plane_stride * p.channels : 0;
  e.base = p.data + p.items.offset[item] + static_cast<long long>(tt) * p.tpatch * e.frame_stride +
           static_cast<long long>(r) * p.patch * W + c * p.patch;
  return e;
}
__device__ __forceinline__ int eg_offset(uint32_t e, int plane_stride, int frame_stride, int W) {
  return static_cast<int>((e >> 16) & 0xFFu) * frame_stride + static_cast<int>(e >> 24) * plane_stride + static_cast<int>((e >> 8) & 0xFFu) * W +
         static_cast<int>(e & 0xFFu);
}
// the pixel pair `pair` of the patch vector, whose table entry is e
__device__ __forceinline__ uint32_t eg_load_pair(const EmbedGemmParams& p, const bf16* base, int plane_stride, int frame_stride, int W,
                                                 uint32_t e, int pair) {
  if (e == kEgPad) return 0u;
  const bf16* src = base + eg_offset(e, plane_stride, frame_stride, W);
  if (p.pairs_ok) return *reinterpret_cast<const uint32_t*>(src);
  // odd geometry (odd patch edge, width or item offset): element loads; the second element of the pair
  // may belong to the next run
  const unsigned short lo = *reinterpret_cast<const unsigned short*>(src);
  int px1 = static_cast<int>(e & 0xFFu) + 1, py1 = static_cast<int>((e >> 8) & 0xFFu), f1 = static_cast<int>((e >> 16) & 0xFFu), ch1 = static_cast<int>(e >> 24);
  if (px1 == p.patch) { px1 = 0; if (++py1 == p.patch) { py1 = 0; if (++f1 == p.tpatch) { f1 = 0; ++ch1; } } }
  unsigned short hi = 0;
  if (2 * pair + 1 < p.k) hi = *reinterpret_cast<const unsigned short*>(base + (f1 * frame_stride + ch1 * plane_stride + py1 * W + px1));
  return static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 16);
}

template <int R>
__global__ void __launch_bounds__(kEgThreads, 1) embed_gemm_kernel(const __grid_constant__ EmbedGemmParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw_eg[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw_eg) + 1023) & ~uintptr_t(1023));
  const int k_blocks = p.k_pad / 64;
  const int resident = min(k_blocks, kEgMaxResident);
  constexpr int kSlot = R * 128;                       // R patch rows x 64 elements
  static_assert(R == 32 || R == 64 || R == 128, "rows of a patch block");
  uint8_t* wring = smem + kEgMaxResident * kSlot;
  uint64_t* bars = reinterpret_cast<uint64_t*>(wring + kEgWStages * kEgBBytes);
  uint64_t* a_full = bars;                             // [resident] the gather warps have written the slot
  uint64_t* a_free = bars + kEgMaxResident;            // [resident] the last UMMA that reads the slot has completed
  uint64_t* w_full = bars + 2 * kEgMaxResident;        // [kEgWStages]
  uint64_t* w_empty = w_full + kEgWStages;             // [kEgWStages]
  uint64_t* acc_full = w_empty + kEgWStages;           // [2]
  uint64_t* acc_empty = acc_full + 2;                  // [2] 8 epilogue warps
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m_blocks = (p.n_patches + R - 1) / R;
  const int n_blocks = (p.N + 255) / 256;
  const int n_units = m_blocks * p.col_groups;         // unit: patch block unit / col_groups, column group unit % col_groups
  auto first_col = [&](int group) { return group * n_blocks / p.col_groups; };     // a group's column blocks, as even as possible
  const int passes = (k_blocks + resident - 1) / resident;

  if (threadIdx.x == 0) {
    for (int s = 0; s < resident; ++s) { mbar_init(&a_full[s], kEgGatherWarps); mbar_init(&a_free[s], 1); }
    for (int s = 0; s < kEgWStages; ++s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(&acc_full[a], 1); mbar_init(&acc_empty[a], 8); }
    *abort_flag = 0;
    mbar_fence_init();
    tma_prefetch_desc(&p.tma_w);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  if (p.early_launch) pdl_launch_dependents();
  if (warp != 0) pdl_wait();     // the weights are constant: their loads need not wait for the stream's earlier work

  // a whole warp waits on a barrier: lane 0 polls, the outcome is the same for all lanes (so the warp leaves a loop together)
  auto warp_wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    uint32_t got = 1u;
    if (lane == 0) got = mbar_wait(bar, parity, abort_flag) ? 1u : 0u;
    return __shfl_sync(0xffffffffu, got, 0) != 0u;
  };
  // the k-blocks are dealt to the passes as evenly as possible: pass p covers [pass_first(p), pass_first(p) + pass_blocks(p))
  const int per_pass = k_blocks / passes, extra = k_blocks - per_pass * passes;
  auto pass_blocks = [&](int pass) { return per_pass + (pass < extra ? 1 : 0); };
  auto pass_first = [&](int pass) { return pass * per_pass + min(pass, extra); };

  if (warp == 0) {
    // ------------------------------------------------------------------ W producer
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int unit = blockIdx.x; unit < n_units && ok; unit += gridDim.x)
        for (int pass = 0; pass < passes && ok; ++pass)
          for (int nb = first_col(unit % p.col_groups); nb < first_col(unit % p.col_groups + 1) && ok; ++nb)
            for (int j = 0; j < pass_blocks(pass); ++j, ++it) {
              const int s = it % kEgWStages;
              if (it == kEgWStages) pdl_wait();      // the next wait needs the consumer, hence the earlier kernels
              if (!mbar_wait(&w_empty[s], ((it / kEgWStages) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
              mbar_expect_tx(&w_full[s], kEgBBytes);
              tma_load_2d(wring + s * kEgBBytes, &p.tma_w, &w_full[s], (pass_first(pass) + j) * 64, nb * 256);
            }
      if (!ok) {
        const long long t0 = clock64();
        while (clock64() - t0 < 4000000) {}          // let loads in flight land before the CTA retires
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ UMMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc_bf16(128, 256, 0, 0);
      uint32_t it = 0, tcount = 0;                   // weight stages used, accumulators used
      uint32_t full_par = 0;                         // bit j: parity of slot j's next fill (slots are not all used in every pass)
      bool ok = true;
      for (int unit = blockIdx.x; unit < n_units && ok; unit += gridDim.x)
        for (int pass = 0; pass < passes && ok; ++pass) {
          const int nj = pass_blocks(pass);
          const int nb0 = first_col(unit % p.col_groups), nb1 = first_col(unit % p.col_groups + 1);
          for (int nb = nb0; nb < nb1 && ok; ++nb, ++tcount) {
            const uint32_t acc = tcount & 1u;
            if (!mbar_wait(&acc_empty[acc], ((tcount >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t tmem_d = tmem_base + acc * 256;
            for (int j = 0; j < nj; ++j, ++it) {
              const int s = it % kEgWStages;
              // the first column block runs behind the gather; the others find every slot filled
              if (nb == nb0) {
                if (!mbar_wait(&a_full[j], (full_par >> j) & 1u, abort_flag)) { ok = false; break; }
                full_par ^= 1u << j;
              }
              if (!mbar_wait(&w_full[s], (it / kEgWStages) & 1u, abort_flag)) { ok = false; break; }
              tc_fence_after_sync();
              const uint64_t adesc = make_smem_desc(smem_u32(smem + j * kSlot), 16, 1024, kSwizzle128B);
              const uint64_t bdesc = make_smem_desc(smem_u32(wring + s * kEgBBytes), 16, 1024, kSwizzle128B);
#pragma unroll
              for (int k = 0; k < 4; ++k) umma_bf16_ss(tmem_d, adesc + 2 * k, bdesc + 2 * k, idesc, (j | k) != 0);
              umma_commit(&w_empty[s]);
              if (nb == nb1 - 1) umma_commit(&a_free[j]);   // the slot's last reader: the gather may refill it
            }
            if (ok) umma_commit(&acc_full[acc]);
          }
        }
    }
  } else if (warp < 2 + kEgGatherWarps) {
    // ------------------------------------------------------------------ gather: kThreadsPerRow threads per patch row
    constexpr int kThreadsPerRow = 32 * kEgGatherWarps / R, kChunks = 8 / kThreadsPerRow;   // 16-byte chunks per thread and k-block
    constexpr int kDepth = R == 128 ? 3 : 6;        // k-blocks whose loads are in flight
    const int t = threadIdx.x - 64;                 // 0..255
    const int row = t / kThreadsPerRow, sub = t % kThreadsPerRow;   // this thread writes chunks kChunks * sub ... of the row
    const int sw = row & 7;
    uint32_t used = 0, free_par = 0;                // bit j: slot j has been filled before; parity of its next hand-back
    bool ok = true;
    for (int unit = blockIdx.x; unit < n_units && ok; unit += gridDim.x) {
      const int m = unit / p.col_groups * R + row;
      const bool row_ok = m < p.n_patches;
      EgPatch e{p.data, 0, 0, 0};
      if (row_ok) e = eg_locate(p, m);
      // the pairs of this thread in k-block kb (registers only)
      auto load_block = [&](int kb, uint32_t (&v)[4 * kChunks]) {
        const uint4* tab4 = reinterpret_cast<const uint4*>(p.table + kb * 32 + sub * (4 * kChunks));
#pragma unroll
        for (int q = 0; q < kChunks; ++q) {
          const uint4 e4 = __ldg(tab4 + q);
          const uint32_t ent[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            v[q * 4 + j] = row_ok ? eg_load_pair(p, e.base, e.plane_stride, e.frame_stride, e.width, ent[j], kb * 32 + (sub * kChunks + q) * 4 + j) : 0u;
        }
      };
      for (int pass = 0; pass < passes && ok; ++pass) {
        const int nj = pass_blocks(pass), kb0 = pass_first(pass);
        uint32_t buf[kDepth][4 * kChunks];
#pragma unroll
        for (int d = 0; d < kDepth; ++d)
          if (d < nj) load_block(kb0 + d, buf[d]);
        for (int j0 = 0; j0 < nj && ok; j0 += kDepth) {
#pragma unroll
          for (int d = 0; d < kDepth; ++d) {
            const int j = j0 + d;
            if (j >= nj) break;
            // the slot's previous contents (an earlier pass or unit) have been read by their last UMMA
            if ((used >> j) & 1u) {
              if (!warp_wait(&a_free[j], (free_par >> j) & 1u)) { ok = false; break; }
              free_par ^= 1u << j;
            }
            used |= 1u << j;
            uint8_t* srow = smem + j * kSlot + row * 128;
#pragma unroll
            for (int q = 0; q < kChunks; ++q)
              *reinterpret_cast<uint4*>(srow + (((sub * kChunks + q) ^ sw) << 4)) = make_uint4(buf[d][4 * q], buf[d][4 * q + 1], buf[d][4 * q + 2], buf[d][4 * q + 3]);
            fence_proxy_async_smem();               // generic-proxy stores -> visible to the tensor core's operand reads
            __syncwarp();
            if (lane == 0) mbar_arrive(&a_full[j]);
            if (j + kDepth < nj) load_block(kb0 + j + kDepth, buf[d]);
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    const int quarter = warp & 3;                 // TMEM lane quarter this warp may read (warps 10..17 -> 2, 3, 0, 1, 2, 3, 0, 1)
    const int half = (warp - 2 - kEgGatherWarps) >> 2;       // which 128 of the 256 columns
    uint32_t tcount = 0;
    bool ok = true;
    for (int unit = blockIdx.x; unit < n_units && ok; unit += gridDim.x) {
      const int m = unit / p.col_groups * R + quarter * 32 + lane;
      bool row_ok = quarter * 32 < R && m < p.n_patches;
      long long orow = 0;
      int posrow = 0;
      if (row_ok) {
        const int mapped = p.row_map[m];
        row_ok = mapped >= 0;
        orow = mapped;
        if (p.pos != nullptr) posrow = p.pos_idx[m];
      }
      for (int pass = 0; pass < passes && ok; ++pass)
        for (int nb = first_col(unit % p.col_groups); nb < first_col(unit % p.col_groups + 1) && ok; ++nb, ++tcount) {
          const uint32_t acc = tcount & 1u;
          if (!warp_wait(&acc_full[acc], (tcount >> 1) & 1u)) { ok = false; break; }
          tc_fence_after_sync();
#pragma unroll 1
          for (int c = half * 4; c < half * 4 + 4 && quarter * 32 < R; ++c) {
            const int col0 = nb * 256 + c * 32;
            uint32_t raw[32];
            __syncwarp();
            tmem_ld_32x32(tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + acc * 256 + c * 32, raw);
            tmem_ld_wait();
            if (!row_ok || col0 >= p.N) continue;
            float v[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(raw[i]);
            float4* o4 = reinterpret_cast<float4*>(p.x + orow * p.N + col0);
            if (pass == 0) {
              const uint4* bp = reinterpret_cast<const uint4*>(p.bias + col0);
              const uint4* pp = p.pos != nullptr ? reinterpret_cast<const uint4*>(p.pos + static_cast<long long>(posrow) * p.N + col0) : nullptr;
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const uint4 b = __ldg(bp + q);
                const uint32_t wb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) { v[q * 8 + 2 * j] += bf16_lo(wb[j]); v[q * 8 + 2 * j + 1] += bf16_hi(wb[j]); }
                if (pp != nullptr) {
                  const uint4 t4 = __ldg(pp + q);
                  const uint32_t wp[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                  for (int j = 0; j < 4; ++j) { v[q * 8 + 2 * j] += bf16_lo(wp[j]); v[q * 8 + 2 * j + 1] += bf16_hi(wp[j]); }
                }
              }
            } else {
              // a later pass over K: add to what the earlier passes stored (this thread wrote it: program order)
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const float4 r = o4[q];
                v[4 * q] += r.x; v[4 * q + 1] += r.y; v[4 * q + 2] += r.z; v[4 * q + 3] += r.w;
              }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) o4[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          }
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[acc]);
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

// ------------------------------------------------------------------------------- vectors that stay resident
// Patch vectors of up to kErMaxK k-blocks (1216 elements).  The same product with the operands exchanged: the UMMA's 128 rows are output
// columns (the weight tile) and its columns are R patches.  What bounds embed_gemm_kernel is a unit's chain of latencies with few
// patches and the second pass over K with longer vectors; here
//   - a unit (R = 32 or 64 patches, a group of 128-column blocks) is small, so that one image fills the chip;
//   - the whole patch vector stays in shared memory, 16 KB weight tiles run through a ring of eight or four;
//   - an epilogue thread owns one output column, so its stores are whole 128-byte lines, and it has loaded the position rows before the
//     accumulator is complete (one load behind each store cost a column block 8 us);
//   - where the patches' pixels are (item, row, column, table entries) is worked out before the grid dependency resolves;
//   - where eight elements of a pixel run lie on a 16-byte boundary (patch edges, widths and offsets that are multiples of 8) they are one load.
// A vector that embed_gemm_kernel walks in two passes has an accumulator per pass, added in that order: the same bits.
constexpr int kErMaxK = 19;
constexpr int kErWBytes = 128 * 64 * 2;                 // 16 KB: 128 weight rows x 64 elements
template <int R> struct EmbedResidentCfg {
  static constexpr int kSlot = R * 128;                 // R patch rows x 64 elements
  static constexpr int kWStages = R == 32 ? 8 : 4;
  static constexpr int kWOff = kErMaxK * kSlot, kBarOff = kWOff + kWStages * kErWBytes;
  static constexpr int kBytes = kBarOff + 512 + 1024;   // + barriers + alignment slack
  static_assert(kBytes <= 232448 && kBytes > 116224, "one CTA per SM");
  static_assert((2 * kErMaxK + 2 * kWStages + 4) * 8 + 8 <= 512, "barrier area");
};

template <int R>
__global__ void __launch_bounds__(kEgThreads, 1) embed_resident_kernel(const __grid_constant__ EmbedGemmParams p) {
  using Cfg = EmbedResidentCfg<R>;
  constexpr int kSlot = Cfg::kSlot, kWStages = Cfg::kWStages;
  extern __shared__ __align__(1024) uint8_t smem_raw_eg[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw_eg) + 1023) & ~uintptr_t(1023));
  uint8_t* wring = smem + Cfg::kWOff;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Cfg::kBarOff);
  uint64_t* a_full = bars;                              // [kErMaxK] the gather warps have written the slot
  uint64_t* a_free = a_full + kErMaxK;                  // [kErMaxK] the last UMMA that reads the slot has completed
  uint64_t* w_full = a_free + kErMaxK;                  // [kWStages]
  uint64_t* w_empty = w_full + kWStages;                // [kWStages]
  uint64_t* acc_full = w_empty + kWStages;              // [2]
  uint64_t* acc_empty = acc_full + 2;                   // [2] 8 epilogue warps
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int k_blocks = p.k_pad / 64;
  const int passes = (k_blocks + kEgMaxResident - 1) / kEgMaxResident;          // 1 or 2, dealt as in embed_gemm_kernel
  const int pass0 = k_blocks / passes + (k_blocks % passes != 0 ? 1 : 0);       // k-blocks of the first
  const int n_blocks = p.N / 128;
  const int n_units = (p.n_patches + R - 1) / R * p.col_groups;
  auto first_col = [&](int group) { return group * n_blocks / p.col_groups; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kErMaxK; ++s) { mbar_init(&a_full[s], kEgGatherWarps); mbar_init(&a_free[s], 1); }
    for (int s = 0; s < kWStages; ++s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(&acc_full[a], 1); mbar_init(&acc_empty[a], 8); }
    *abort_flag = 0;
    mbar_fence_init();
    tma_prefetch_desc(&p.tma_w);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 256); tmem_relinquish(); }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  if (p.early_launch) pdl_launch_dependents();

  if (warp == 0) {
    // ------------------------------------------------------------------ W producer (constant weights: no wait for earlier work yet)
    uint32_t it = 0;
    bool ok = true;
    for (int unit = blockIdx.x; unit < n_units && ok; unit += gridDim.x)
      for (int nb = first_col(unit % p.col_groups); nb < first_col(unit % p.col_groups + 1) && ok; ++nb)
        for (int j = 0; j < k_blocks; ++j, ++it) {
          const uint32_t s = it % kWStages;
          if (it == kWStages) pdl_wait();               // the next wait needs the consumer, hence the earlier kernels
          if (!warp_mbar_wait(&w_empty[s], ((it / kWStages) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
          if (elect_one()) {
            mbar_expect_tx(&w_full[s], kErWBytes);
            tma_load_2d(wring + s * kErWBytes, &p.tma_w, &w_full[s], j * 64, nb * 128);
          }
          __syncwarp();
        }
    if (!ok) {
      const long long t0 = clock64();
      while (clock64() - t0 < 4000000) {}               // let loads in flight land before the CTA retires
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ UMMA issuer
    pdl_wait();
    constexpr uint32_t idesc = make_idesc_bf16(128, R, 0, 0);
    uint32_t it = 0, tcount = 0, round = 0;
    bool ok = true;
    for (int unit = blockIdx.x; unit < n_units && ok; unit += gridDim.x, ++round) {
      const int nb0 = first_col(unit % p.col_groups), nb1 = first_col(unit % p.col_groups + 1);
      for (int nb = nb0; nb < nb1 && ok; ++nb, ++tcount) {
        const uint32_t acc = tcount & 1u;
        if (!warp_mbar_wait(&acc_empty[acc], ((tcount >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
        for (int j = 0; j < k_blocks; ++j, ++it) {
          const uint32_t s = it % kWStages;
          if (nb == nb0 && !warp_mbar_wait(&a_full[j], round & 1u, abort_flag)) { ok = false; break; }
          if (!warp_mbar_wait(&w_full[s], (it / kWStages) & 1u, abort_flag)) { ok = false; break; }
          tc_fence_after_sync();
          if (elect_one()) {
            const uint64_t wdesc = make_smem_desc(smem_u32(wring + s * kErWBytes), 16, 1024, kSwizzle128B);
            const uint64_t pdesc = make_smem_desc(smem_u32(smem + j * kSlot), 16, 1024, kSwizzle128B);
            const uint32_t d = tmem_base + acc * (2 * R) + (j < pass0 ? 0 : R);
#pragma unroll
            for (int k = 0; k < 4; ++k) umma_bf16_ss(d, wdesc + 2 * k, pdesc + 2 * k, idesc, (k != 0 || (j != 0 && j != pass0)) ? 1u : 0u);
            umma_commit(&w_empty[s]);
            if (nb == nb1 - 1) umma_commit(&a_free[j]);   // the slot's last reader: the gather may refill it
            if (j == k_blocks - 1) umma_commit(&acc_full[acc]);
          }
          __syncwarp();
        }
      }
    }
    // the last hand-backs are asynchronous arrivals that nothing else waits for: in before the shared memory passes on
    for (uint32_t e = it; e < it + kWStages && ok; ++e) ok = warp_mbar_wait(&w_empty[e % kWStages], ((e / kWStages) & 1u) ^ 1u, abort_flag);
    for (int j = 0; j < k_blocks && ok && round > 0; ++j) ok = warp_mbar_wait(&a_free[j], (round - 1) & 1u, abort_flag);
  } else if (warp < 2 + kEgGatherWarps) {
    // ------------------------------------------------------------------ gather: kThreadsPerRow threads per patch row
    constexpr int kThreadsPerRow = 32 * kEgGatherWarps / R, kChunks = 8 / kThreadsPerRow;   // 16-byte chunks per thread and k-block
    constexpr int kDepth = R == 32 ? 6 : 3;           // k-blocks whose loads are in flight
    const int t = threadIdx.x - 64;                   // 0..255
    const int row = t / kThreadsPerRow, sub = t % kThreadsPerRow;
    const int sw = row & 7;
    const bf16* base = p.data;                        // first pixel of the patch in frame-in-patch 0 of channel 0, and the strides
    int plane_stride = 0, frame_stride = 0, W = 0;
    bool row_ok = false;
    auto locate = [&](int unit) {
      const int m = unit / p.col_groups * R + row;
      row_ok = m < p.n_patches;
      if (!row_ok) return;
      const EgPatch e = eg_locate(p, m);
      base = e.base; plane_stride = e.plane_stride; frame_stride = e.frame_stride; W = e.width;
    };
    uint4 ent[kDepth][kChunks];                       // table entries of the next k-blocks
    auto load_table = [&](int kb, uint4 (&e)[kChunks]) {
#pragma unroll
      for (int q = 0; q < kChunks; ++q) e[q] = __ldg(reinterpret_cast<const uint4*>(p.table + kb * 32 + (sub * kChunks + q) * 4));
    };
    auto load_pixels = [&](int kb, const uint4 (&e4)[kChunks], uint4 (&v)[kChunks]) {
#pragma unroll
      for (int q = 0; q < kChunks; ++q) {
        if (p.chunks_ok) {                              // a chunk of eight elements lies inside a pixel run, on a 16-byte boundary
          v[q] = row_ok && e4[q].x != kEgPad ? *reinterpret_cast<const uint4*>(base + eg_offset(e4[q].x, plane_stride, frame_stride, W)) : make_uint4(0u, 0u, 0u, 0u);
          continue;
        }
        const uint32_t e[4] = {e4[q].x, e4[q].y, e4[q].z, e4[q].w};
        uint32_t o[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          o[j] = row_ok ? eg_load_pair(p, base, plane_stride, frame_stride, W, e[j], kb * 32 + (sub * kChunks + q) * 4 + j) : 0u;
        v[q] = make_uint4(o[0], o[1], o[2], o[3]);
      }
    };
    if (static_cast<int>(blockIdx.x) < n_units) locate(blockIdx.x);
#pragma unroll
    for (int d = 0; d < kDepth; ++d)
      if (d < k_blocks) load_table(d, ent[d]);
    pdl_wait();
    uint32_t round = 0;
    bool ok = true;
    for (int unit = blockIdx.x; unit < n_units && ok; unit += gridDim.x, ++round) {
      if (round != 0) {
        locate(unit);
#pragma unroll
        for (int d = 0; d < kDepth; ++d)
          if (d < k_blocks) load_table(d, ent[d]);
      }
      uint4 buf[kDepth][kChunks];
#pragma unroll
      for (int d = 0; d < kDepth; ++d)
        if (d < k_blocks) {
          load_pixels(d, ent[d], buf[d]);
          if (d + kDepth < k_blocks) load_table(d + kDepth, ent[d]);
        }
      for (int j0 = 0; j0 < k_blocks && ok; j0 += kDepth) {
#pragma unroll
        for (int d = 0; d < kDepth; ++d) {
          const int j = j0 + d;
          if (j >= k_blocks) break;
          if (round != 0 && !warp_mbar_wait(&a_free[j], (round - 1) & 1u, abort_flag)) { ok = false; break; }
          uint8_t* srow = smem + j * kSlot + row * 128;
#pragma unroll
          for (int q = 0; q < kChunks; ++q) *reinterpret_cast<uint4*>(srow + (((sub * kChunks + q) ^ sw) << 4)) = buf[d][q];
          fence_proxy_async_smem();                   // generic-proxy stores -> visible to the tensor core's operand reads
          __syncwarp();
          if (lane == 0) mbar_arrive(&a_full[j]);
          if (j + kDepth < k_blocks) {
            load_pixels(j + kDepth, ent[d], buf[d]);
            if (j + 2 * kDepth < k_blocks) load_table(j + 2 * kDepth, ent[d]);
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue: a thread per output column, half of the patches a warp
    const int quarter = warp & 3, half = (warp - 2 - kEgGatherWarps) >> 2;
    constexpr int kHalf = R / 2;
    pdl_wait();
    uint32_t tcount = 0;
    bool ok = true;
    for (int unit = blockIdx.x; unit < n_units && ok; unit += gridDim.x) {
      const int m0 = unit / p.col_groups * R + half * kHalf;
      int my_row = -1, my_pos = 0;                    // of patch m0 + lane
      if (lane < kHalf && m0 + lane < p.n_patches) {
        my_row = p.row_map[m0 + lane];
        if (p.pos != nullptr) my_pos = p.pos_idx[m0 + lane];
      }
      for (int nb = first_col(unit % p.col_groups); nb < first_col(unit % p.col_groups + 1) && ok; ++nb, ++tcount) {
        const uint32_t acc = tcount & 1u;
        const int col = nb * 128 + quarter * 32 + lane;
        const float bias = __bfloat162float(p.bias[col]);
        bf16 pos[kHalf];                              // all ahead of the stores (and of the accumulator): a load each costs an L2 round trip
#pragma unroll
        for (int i = 0; i < kHalf; ++i)
          if (p.pos != nullptr) pos[i] = p.pos[static_cast<long long>(__shfl_sync(0xffffffffu, my_pos, i)) * p.N + col];
        if (!warp_mbar_wait(&acc_full[acc], (tcount >> 1) & 1u, abort_flag)) { ok = false; break; }
        tc_fence_after_sync();
        const uint32_t d = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + acc * (2 * R) + half * kHalf;
#pragma unroll
        for (int c = 0; c < kHalf; c += 16) {
          uint32_t v0[16], v1[16];
          __syncwarp();
          tmem_ld_32x16(d + c, v0);
          if (passes > 1) tmem_ld_32x16(d + R + c, v1);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int orow = __shfl_sync(0xffffffffu, my_row, c + i);
            float v = __uint_as_float(v0[i]) + bias;
            if (p.pos != nullptr) v += __bfloat162float(pos[c + i]);
            if (passes > 1) v = __uint_as_float(v1[i]) + v;
            if (orow >= 0) p.x[static_cast<long long>(orow) * p.N + col] = v;
          }
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[acc]);
      }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem_base, 256);
  }
  if (threadIdx.x == 0 && *abort_flag) atomicCAS(p.status, DEV_OK, DEV_ERR_WAIT_TIMEOUT);
}

}  // namespace eas
