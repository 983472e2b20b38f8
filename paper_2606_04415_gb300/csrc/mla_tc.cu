// Absorbed multi-head latent attention (MLA, the DeepSeek-R1 shape) on the
// fifth-generation tensor cores: every query head reads one shared latent
// cache row of d_qk = 576 values per key, and V is its first d_v = 512 values
// (Eq. 1 with K = latent, V = latent[:, :512]). Prefill and decode rows share
// the kernel: the 128 heads of one query token are the 128 rows of a tile, so
// the phase only changes how many keys a token sees.
//
// The fp32 accumulator of 128 rows x 512 columns would fill all of tensor
// memory, so one work item is (token, half of d_v, key range) and two CTAs
// take the two halves of a token; both compute the same S = Q K^T (the
// product is 1.5x the minimum, against none of the accumulator fitting
// otherwise) and each keeps O for its 256 columns. Both halves read the same
// latent tiles at about the same time (they are neighbours in the work list),
// so the second read is served by L2.
//
// Tensor memory (512 columns): O half [0, 256), S [256, 320), P (bf16) [320,
// 352), and the Q columns of this half's V columns and the rotary ones as packed
// bf16 pairs [352, 512), the A operand of 20 of the 36 k-steps of S. The other
// 256 Q columns sit in shared memory for the other 16 (a product with both
// operands there takes 46 cycles instead of 32, so these are the ones that run
// beside the softmax). S and P do not share columns: S(j + 1) may overwrite S(j) as soon
// as the softmax has read it into registers, so that its product runs beside
// the exponentials of tile j.
//
// A 64-key latent tile comes in two parts with a ring each: the five
// 64-column chunks that only S reads (the other half's value columns and the
// rotary ones; two slots of 40 KB, free once S is done) and the four chunks
// that are also this half's V operand (two slots of 32 KB, free after P V).
// MMAs are issued in the order S(j + 1) over the first part, P V(j), S(j + 1)
// over the V part: P V(j) frees its slot as soon as P is there, and the first
// part of S covers the exponentials.
//
// One persistent CTA per SM (320 threads) takes items, longest first, from an
// atomic queue (the last CTA out resets it):
//   warps 0-3  softmax, one row each (TMEM lane = head), with a lazy O rescale
//              (only when the row maximum grows by more than 2^8), while no
//              product is writing O: when S(j) is complete so is P V(j - 1);
//   warp 4     scheduler and TMA producer (each lane issues one box of a part,
//              so that a tile of four 16-slot blocks is no slower): the next
//              item's first tiles load while the current one ends;
//   warp 5     MMA issuer;
//   warps 6-9  the next item's tensor-memory part of Q (held in registers
//              until the last S of the current item is done) and the epilogue
//              of the last item, beside the next item's first S and softmax.
// Measured, one 1024-token prompt and 256 decodes of 1024..16384 keys: 974 us a
// step with one CTA per item and P over S's columns, 904 with this kernel in a
// loop that lasts (at the power limit, SM clock 1785 of 2070 MHz), 839 in a
// short one; the prompt alone 281 us and 208.
// Every mbarrier wait is bounded; a timeout raises the plan's error flag and
// the CTA drains its copies and tensor-core work, frees its tensor memory and
// exits.
#include <math.h>

#include "common.cuh"
#include "tc.cuh"

namespace fnpu {
namespace {

constexpr int kDq = 576, kDv = 512, kDvHalf = 256;
constexpr int kRows = 128;                    // heads of one token = TMEM lanes
constexpr int kKeysT = 64;                    // keys per latent tile
constexpr int kQsChunks = 4;                  // Q chunks in shared memory (the other half's V columns)
constexpr int kQtChunks = 5;                  // Q chunks in tensor memory (this half's V columns, the rotary ones)
constexpr int kNChunks = 5;                   // chunks of a tile read by S only
constexpr int kVChunks = 4;                   // chunks of a tile that are V as well
constexpr int kStages = 2;
constexpr int kItemSlots = 4;
constexpr int kThreads = 320;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColO = 0, kColS = 256, kColP = 320, kColQ = 352;
constexpr float kRescaleThreshold = 8.0f;     // log2 units

constexpr int kChunkBytes = kKeysT * 128;             // 8 KB
constexpr int kQChunkBytes = kRows * 128;             // 16 KB
constexpr int kNBytes = kNChunks * kChunkBytes;       // 40 KB
constexpr int kVBytes = kVChunks * kChunkBytes;       // 32 KB
constexpr int kOffN = kQsChunks * kQChunkBytes;
constexpr int kOffV = kOffN + kStages * kNBytes;
constexpr int kOffStage = kOffV + kStages * kVBytes;  // a 32-row x 64-column box per epilogue warp (Q in, O out)
constexpr int kOffL = kOffStage + kQChunkBytes;       // [2 items][128 rows] (log2 max, sum)
constexpr int kOffBar = kOffL + 2 * kRows * 8;
// nfull[2] nempty[2] vfull[2] vempty[2] itemfull[4] itemempty[4] and
// sfull sfree pready odone ofree lready[2] qfull qready qfree drain stage[4]
constexpr int kNumBars = 4 * kStages + 2 * kItemSlots + 15;
constexpr int kOffMisc = kOffBar + 8 * kNumBars;      // tmem address, abort flag, item ring
constexpr int kSmemBytes = kOffMisc + 8 + 4 * kItemSlots;
static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
static_assert(kColQ + kQtChunks * 32 == kTmemCols, "tensor memory budget");
static_assert((kQsChunks + kQtChunks) * 64 == kDq, "Q chunks");

struct MlaMaps {
    CUtensorMap kv, q, q32, out32;  // (32 rows a box: one warp's)
};

__global__ void __launch_bounds__(kThreads, 1) mla_tc_kernel(const AttnParams p, const __grid_constant__ MlaMaps maps) {
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t s_base = smem_u32(smem);
    const uint32_t bars = s_base + kOffBar;
    auto NFULL = [&](int s) { return bars + 8 * s; };
    auto NEMPTY = [&](int s) { return bars + 8 * (kStages + s); };
    auto VFULL = [&](int s) { return bars + 8 * (2 * kStages + s); };
    auto VEMPTY = [&](int s) { return bars + 8 * (3 * kStages + s); };
    const uint32_t b1 = bars + 8 * (4 * kStages);
    auto ITEMFULL = [&](int s) { return b1 + 8 * s; };
    auto ITEMEMPTY = [&](int s) { return b1 + 8 * (kItemSlots + s); };
    const uint32_t b2 = b1 + 16 * kItemSlots;
    const uint32_t SFULL = b2, SFREE = b2 + 8, PREADY = b2 + 16, ODONE = b2 + 24, OFREE = b2 + 32,
                   QFULL = b2 + 56, QREADY = b2 + 64, QFREE = b2 + 72, DRAIN = b2 + 80;
    // (one for even and one for odd items: an item of one tile may end before an
    // epilogue warp has looked at the end of the one before; the next of the same
    // parity cannot, as its Q comes from that warp)
    auto LREADY = [&](int k) { return b2 + 40 + 8 * (k & 1); };
    auto STAGE = [&](int w) { return b2 + 88 + 8 * w; };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + kOffMisc);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + kOffMisc + 4);
    volatile int *item_slot = reinterpret_cast<volatile int *>(smem + kOffMisc + 8);  // [kItemSlots]
    float2 *l_buf = reinterpret_cast<float2 *>(smem + kOffL);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_trigger();  // the merge grid may be placed once these CTAs are; it waits for them to finish
    if ((s_base & 1023u) != 0) {  // the swizzled tiles need 1024-byte alignment
        pdl_wait();
        if (tid == 0) atomicOr(p.err, 2);
        return;
    }
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(NFULL(s), 1);
            tc::mbar_init(NEMPTY(s), 1);
            tc::mbar_init(VFULL(s), 1);
            tc::mbar_init(VEMPTY(s), 1);
        }
        for (int s = 0; s < kItemSlots; ++s) {
            tc::mbar_init(ITEMFULL(s), 1);
            tc::mbar_init(ITEMEMPTY(s), 9);  // MMA issuer, four softmax and four epilogue warps
        }
        tc::mbar_init(SFULL, 1);
        tc::mbar_init(SFREE, 4);
        tc::mbar_init(PREADY, 4);
        tc::mbar_init(ODONE, 1);
        tc::mbar_init(OFREE, 4);
        tc::mbar_init(LREADY(0), 4);
        tc::mbar_init(LREADY(1), 4);
        tc::mbar_init(QFULL, 1);
        tc::mbar_init(QREADY, 4);
        tc::mbar_init(QFREE, 1);
        for (int w = 0; w < 4; ++w) tc::mbar_init(STAGE(w), 1);
        tc::mbar_init(DRAIN, 1);
        *abort_flag = 0;
        tc::fence_mbar_init();
    }
    if (warp == 0) {
        tc::tmem_alloc(smem_u32(const_cast<uint32_t *>(tmem_slot)), kTmemCols);
        tc::tmem_relinquish();
    }
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();  // the cache writes of the kernel before (the step's append)

    auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
        if (tc::mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (tc::mbar_wait(bar, parity)) return true;
        *abort_flag = 1;
        atomicOr(p.err, 1);
        return false;
    };
    // item k of this CTA: its index from the ring (-1: no more)
    auto next_item = [&](int k, int &idx) -> bool {
        if (!wait(ITEMFULL(k % kItemSlots), (k / kItemSlots) & 1)) return false;
        idx = item_slot[k % kItemSlots];
        return true;
    };
    auto tiles_of = [](const MlaItem &it) { return (it.key_end - it.key_begin + kKeysT - 1) / kKeysT; };

    if (warp == 4) {
        // ----------------------------------------- scheduler and TMA producer
        if (lane == 0) {
            tc::prefetch_tmap(&maps.kv);
            tc::prefetch_tmap(&maps.q);
        }
        const int bs = p.block_size;
        const int per_tile = kKeysT / bs;  // blocks per tile (1, 2 or 4)
        int gt = 0, gv = 0;                // tiles issued so far, first part and V part
        // the first item of CTA b is item b; later ones come from the queue
        int idx = static_cast<int>(blockIdx.x);  // (grid <= items)
        if (lane == 0) {
            item_slot[0] = idx;
            tc::mbar_arrive(ITEMFULL(0));
        }
        bool ok = true;
        for (int k = 0; ok && idx < p.num_mitems; ++k) {
            const MlaItem it = p.mitems[idx];
            const int n = __shfl_sync(0xffffffffu, tiles_of(it), 0);
            const int half = __shfl_sync(0xffffffffu, it.hb, 0);
            const int tok = __shfl_sync(0xffffffffu, it.token, 0);
            const int32_t *bt = p.block_table + static_cast<int64_t>(it.bt_row) * p.bt_stride;
            const int nblk_seq = (it.ctx_len + bs - 1) / bs;
            const int b00 = it.key_begin / bs;  // key_begin is a multiple of 64
            // block ids of the next tile, one per lane, loaded a tile ahead
            int blk_next = (lane < per_tile && b00 + lane < nblk_seq) ? __ldg(bt + b00 + lane) : 0;
            // the next item is taken some tiles before this one ends and
            // published two tiles later, in time for its Q to be fetched
            const int jf = n > 8 ? n - 8 : 0, jp = n > 6 ? n - 6 : 0;
            int a = 0, idx_n = 0;
            for (int j = 0; j < n; ++j) {
                if (j == jf && lane == 0) a = static_cast<int>(gridDim.x) + atomicAdd(p.sched, 1);
                const int blk_cur = blk_next;
                const int b0 = b00 + j * per_tile;
                blk_next = (j + 1 < n && lane < per_tile && b0 + per_tile + lane < nblk_seq) ? __ldg(bt + b0 + per_tile + lane) : 0;
                int nvalid = nblk_seq - b0;
                nvalid = __shfl_sync(0xffffffffu, nvalid > per_tile ? per_tile : nvalid, 0);
                const int st = gt % kStages;
                if (gt >= kStages && !wait(NEMPTY(st), ((gt / kStages) - 1) & 1)) { ok = false; break; }
                tc::mbar_arrive_expect_tx_warp(NFULL(st), static_cast<uint32_t>(nvalid * bs * 128 * kNChunks));
                __syncwarp();
                {  // the chunks that only S reads, one copy (block, chunk) a lane
                    const int b = lane / kNChunks, c = lane % kNChunks;
                    const int blk = __shfl_sync(0xffffffffu, blk_cur, b);
                    if (b < nvalid)
                        tc::tma_load_3d(s_base + kOffN + st * kNBytes + c * kChunkBytes + b * bs * 128, &maps.kv, NFULL(st),
                                        64 * (c < 4 ? 4 * (1 - half) + c : 8), 0, blk);
                    __syncwarp();
                }
                ++gt;
                if (gv >= kStages && !wait(VEMPTY(st), ((gv / kStages) - 1) & 1)) { ok = false; break; }
                tc::mbar_arrive_expect_tx_warp(VFULL(st), static_cast<uint32_t>(nvalid * bs * 128 * kVChunks));
                __syncwarp();
                {  // the chunks of this half's V
                    const int b = lane / kVChunks, c = lane % kVChunks;
                    const int blk = __shfl_sync(0xffffffffu, blk_cur, b);
                    if (b < nvalid)
                        tc::tma_load_3d(s_base + kOffV + st * kVBytes + c * kChunkBytes + b * bs * 128, &maps.kv, VFULL(st),
                                        64 * (4 * half + c), 0, blk);
                    __syncwarp();
                }
                ++gv;
                if (j == 0) {  // the other half's Q columns, once the previous item's last S is done
                    if (k >= 1 && !wait(QFREE, (k - 1) & 1)) { ok = false; break; }
                    tc::mbar_arrive_expect_tx_warp(QFULL, kQsChunks * kQChunkBytes);
#pragma unroll
                    for (int c = 0; c < kQsChunks; ++c)
                        tc::tma_load_3d_warp(s_base + c * kQChunkBytes, &maps.q, QFULL, 64 * (4 * (1 - half) + c), 0, tok);
                }
                if (j == jp) {  // publish the next item
                    idx_n = __shfl_sync(0xffffffffu, a, 0);
                    const int sl = (k + 1) % kItemSlots;
                    if (k + 1 >= kItemSlots && !wait(ITEMEMPTY(sl), (((k + 1) / kItemSlots) - 1) & 1)) { ok = false; break; }
                    if (lane == 0) {
                        item_slot[sl] = idx_n < p.num_mitems ? idx_n : -1;
                        tc::mbar_arrive(ITEMFULL(sl));
                    }
                    __syncwarp();
                }
            }
            idx = idx_n;
        }
    } else if (warp == 5) {
        // -------------------------------------------------------- MMA issuer
        constexpr uint32_t idS = tc::idesc_bf16(kRows, kKeysT, false);
        constexpr uint32_t idO = tc::idesc_bf16(kRows, kDvHalf, true);
        const uint32_t utmem = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t us = __shfl_sync(0xffffffffu, s_base, 0);
        const uint32_t tS = utmem + kColS, tO = utmem + kColO, tQ = utmem + kColQ, tP = utmem + kColP;
        const uint64_t qd = tc::sdesc_sw128(us, 16, 1024);
        int gt = 0;  // S tiles issued
        bool ok = true, issued = false;
        // Every MMA of a tile has one place in the code, whichever half: the
        // warps run different code side by side, and an issuer with a copy
        // per half and for the first tile (150 unrolled MMAs) and the softmax
        // evicted each other from the instruction cache (2.7 us a tile; rolled
        // loops over the chunks took 2.0 us by their address arithmetic). One
        // elected lane issues a burst (electing one for each product cost 3%). A
        // wait costs this warp 100 to 170 cycles and a commit 80 to 120 with
        // the tensor pipe idle, so the softmax warps wait for the next tile's
        // V part (before they signal P) and free the first part's slots.
        for (int k = 0; ok; ++k) {
            int idx;
            if (!next_item(k, idx)) { ok = false; break; }
            if (idx < 0) break;
            const int n = __shfl_sync(0xffffffffu, tiles_of(p.mitems[idx]), 0);
            if (!wait(QFULL, k & 1) || !wait(QREADY, k & 1)) { ok = false; break; }
#pragma unroll 1
            for (int u = 0; u <= n; ++u) {
                const int st = __shfl_sync(0xffffffffu, gt % kStages, 0);
                const uint64_t nd = tc::sdesc_sw128(us + kOffN + st * kNBytes, 16, 1024);
                const uint64_t kd = tc::sdesc_sw128(us + kOffV + st * kVBytes, 16, 1024);
                const uint64_t vd = tc::sdesc_sw128(us + kOffV + (st ^ 1) * kVBytes, kChunkBytes, 1024);
                const uint32_t acc = __shfl_sync(0xffffffffu, u > 1 ? 1u : 0u, 0);
                if (u < n) {  // S(u) over the chunks that only S reads
                    if (!wait(NFULL(st), (gt / kStages) & 1)) { ok = false; break; }
                    if (u == 0 && !wait(VFULL(st), (gt / kStages) & 1)) { ok = false; break; }
                    if (gt > 0 && !wait(SFREE, (gt - 1) & 1)) { ok = false; break; }  // the tile before is in registers
                    tc::fence_after_sync();
                    if (tc::elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < 4 * kQsChunks; ++kk)
                            tc::mma_ss(tS, qd + ((kk / 4) * kQChunkBytes + (kk % 4) * 32) / 16,
                                       nd + ((kk / 4) * kChunkBytes + (kk % 4) * 32) / 16, idS, kk > 0 ? 1u : 0u);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)  // the rotary columns
                            tc::mma_ts(tS, tQ + 128 + kk * 8, nd + (4 * kChunkBytes + kk * 32) / 16, idS, 1u);
                    }
                    __syncwarp();
                    issued = true;
                }
                if (u > 0) {  // O += P(u - 1) V(u - 1)
                    if (!wait(PREADY, (gt - 1) & 1)) { ok = false; break; }
                    if (u == 1 && k >= 1 && !wait(OFREE, (k - 1) & 1)) { ok = false; break; }
                    tc::fence_after_sync();
                    if (tc::elect_one()) {
                        tc::mma_ts(tO, tP, vd, idO, acc);
#pragma unroll
                        for (int kk = 1; kk < kKeysT / 16; ++kk) tc::mma_ts(tO, tP + kk * 8, vd + (kk * 2048) / 16, idO, 1u);
                        tc::commit(VEMPTY(st ^ 1));
                        if (u == n) tc::commit(ODONE);
                    }
                    __syncwarp();
                }
                if (u < n) {  // S(u) over the chunks of this half's V
                    if (tc::elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < 4 * kVChunks; ++kk)
                            tc::mma_ts(tS, tQ + kk * 8, kd + ((kk / 4) * kChunkBytes + (kk % 4) * 32) / 16, idS, 1u);
                        tc::commit(SFULL);
                        if (u == n - 1) tc::commit(QFREE);  // the last S of this item
                    }
                    __syncwarp();
                    ++gt;
                }
            }
            if (!ok) break;
            tc::mbar_arrive_warp(ITEMEMPTY(k % kItemSlots));
        }
        if (!ok && issued) {  // drain whatever is still in flight
            tc::commit_warp(DRAIN);
            tc::mbar_wait(DRAIN, 0, 200000000ull);
        }
    } else if (warp < 4) {
        // ------------------------------------------------------ softmax rows
        const int r = tid;  // head = TMEM lane
        const uint32_t lane_addr = tmem + (static_cast<uint32_t>(warp * 32) << 16);
        const float sc = p.scale_log2;
        int T = 0;
        for (int k = 0;; ++k) {
            int idx;
            if (!next_item(k, idx) || idx < 0) break;
            const MlaItem it = p.mitems[idx];
            const int n = tiles_of(it);
            float m_run = -INFINITY, l = 0.f;
            bool ok = true;
            for (int j = 0; j < n; ++j, ++T) {
                if (!wait(SFULL, T & 1)) { ok = false; break; }
                tc::fence_after_sync();
                uint32_t s[kKeysT];
                tc::tmem_ld32(lane_addr + kColS, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
                tc::tmem_ld32(lane_addr + kColS + 32, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
                tc::tmem_wait_ld();
                tc::fence_before_sync();
                __syncwarp();
                tc::mbar_arrive_warp(SFREE);  // the next S may overwrite these columns
                if (warp == 0) tc::mbar_arrive_warp(NEMPTY(T % kStages));  // S(j) has read its first part
                const int nv = it.key_end - (it.key_begin + j * kKeysT);  // keys of this tile inside the item (>= 1)
                if (nv < kKeysT) {
#pragma unroll
                    for (int x = 0; x < kKeysT; ++x)
                        if (x >= nv) s[x] = __float_as_uint(-INFINITY);
                }
                float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
                for (int x = 0; x < kKeysT; x += 4) {
                    mx0 = fmax3(mx0, __uint_as_float(s[x]), __uint_as_float(s[x + 1]));
                    mx1 = fmax3(mx1, __uint_as_float(s[x + 2]), __uint_as_float(s[x + 3]));
                }
                const float tmax = fmaxf(mx0, mx1) * sc;  // finite: the tile has a visible key
                const bool need = m_run == -INFINITY || tmax > m_run + kRescaleThreshold;
                // tensor-memory loads and stores are warp-wide: the warp rescales
                // together, lanes that need none with alpha = 1
                if (__any_sync(0xffffffffu, need)) {
                    const float m_new = need ? fmaxf(m_run, tmax) : m_run;
                    if (j > 0) {
                        // P V(j - 1) is complete: it was issued before the end of S(j)
                        const float alpha = need ? fast_exp2(m_run - m_new) : 1.f;
#pragma unroll 1
                        for (int c = 0; c < kDvHalf / 32; ++c) {
                            uint32_t o[32];
                            tc::tmem_ld32(lane_addr + kColO + 32 * c, o);
                            tc::tmem_wait_ld();
#pragma unroll
                            for (int x = 0; x < 32; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * alpha);
                            tc::tmem_st32(lane_addr + kColO + 32 * c, o);
                        }
                        l *= alpha;
                    }
                    m_run = m_new;
                }
                const uint64_t sc2 = f2_pack(sc, sc), nb2 = f2_pack(-m_run, -m_run);
                uint64_t lacc0 = f2_pack(0.f, 0.f), lacc1 = lacc0;
#pragma unroll
                for (int q4 = 0; q4 < kKeysT / 32; ++q4) {
                    uint32_t pk[16];
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        const uint64_t x2 = f2_fma(
                            f2_pack(__uint_as_float(s[32 * q4 + 2 * x]), __uint_as_float(s[32 * q4 + 2 * x + 1])), sc2, nb2);
                        float x0, x1;
                        f2_unpack(x2, x0, x1);
                        const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                        if (x & 1) lacc1 = f2_add(lacc1, f2_pack(p0, p1));
                        else lacc0 = f2_add(lacc0, f2_pack(p0, p1));
                        pk[x] = pack_bf16x2(p0, p1);
                    }
                    tc::tmem_st16(lane_addr + kColP + 16 * q4, pk);
                }
                {
                    float a0, a1;
                    f2_unpack(f2_add(lacc0, lacc1), a0, a1);
                    l += a0 + a1;
                }
                if (nv < kKeysT) {
                    // rows past the item hold keys of the next piece or stale slots:
                    // zero this half's V columns there (their P is 0, but 0 * NaN is not)
                    for (int e = r; e < (kKeysT - nv) * 4 * 8; e += kRows) {
                        const int row = nv + e / 32, rem = e % 32;
                        *reinterpret_cast<uint4 *>(smem + kOffV + (T % kStages) * kVBytes + (rem / 8) * kChunkBytes + row * 128 +
                                                   (rem % 8) * 16) = make_uint4(0u, 0u, 0u, 0u);
                    }
                    tc::fence_proxy_async_smem();
                }
                tc::tmem_wait_st();
                tc::fence_before_sync();
                // for the issuer: P, and the next tile's V part
                if (j + 1 < n && !wait(VFULL((T + 1) % kStages), ((T + 1) / kStages) & 1)) { ok = false; break; }
                __syncwarp();
                tc::mbar_arrive_warp(PREADY);
            }
            if (!ok) break;
            l_buf[(k & 1) * kRows + r] = make_float2(m_run, l);
            __syncwarp();
            tc::mbar_arrive_warp(LREADY(k));
            tc::mbar_arrive_warp(ITEMEMPTY(k % kItemSlots));
        }
    } else {
        // --------------------------- Q into tensor memory, and the epilogue
        const int quarter = warp & 3;  // the TMEM lanes this warp may read
        const int r = 32 * quarter + lane;
        const uint32_t lane_addr = tmem + (static_cast<uint32_t>(32 * quarter) << 16);
        // Both go by TMA through a 4 KB box of this warp in shared memory: a
        // lane owns a row, and its own global loads and stores (32 lines an
        // instruction) took 3 us each and slowed the products beside them.
        uint8_t *box = smem + kOffStage + quarter * (kQChunkBytes / 4);
        const uint32_t box_addr = s_base + kOffStage + quarter * (kQChunkBytes / 4), bar = STAGE(quarter);
        uint32_t qv[kQtChunks][32];
        uint32_t parity = 0;
        auto load_q = [&](const MlaItem &it) -> bool {
            const int tok = __shfl_sync(0xffffffffu, it.token, 0), half = __shfl_sync(0xffffffffu, it.hb, 0);
#pragma unroll
            for (int c = 0; c < kQtChunks; ++c) {
                tc::mbar_arrive_expect_tx_warp(bar, kQChunkBytes / 4);
                tc::tma_load_3d_warp(box_addr, &maps.q32, bar, 64 * (c < 4 ? 4 * half + c : 8), 32 * quarter, tok);
                const bool ok = wait(bar, parity);
                parity ^= 1;
                if (!ok) return false;
#pragma unroll
                for (int j = 0; j < 8; ++j) {  // 16-byte chunk j of the row at position j ^ (r mod 8)
                    const uint4 x = *reinterpret_cast<const uint4 *>(box + lane * 128 + ((j ^ (lane & 7)) << 4));
                    qv[c][4 * j] = x.x; qv[c][4 * j + 1] = x.y; qv[c][4 * j + 2] = x.z; qv[c][4 * j + 3] = x.w;
                }
                tc::fence_proxy_async_smem();  // these reads before the next copy into the box
                __syncwarp();
            }
            return true;
        };
        auto epilogue = [&](const MlaItem &it, int k) -> bool {
            if (!wait(LREADY(k), (k >> 1) & 1) || !wait(ODONE, k & 1)) return false;
            tc::fence_after_sync();
            const float2 ml = l_buf[(k & 1) * kRows + r];
            const float inv = 1.f / ml.y;
            const bool whole = it.num_splits == 1;
            // (a key split: O / l over its keys and m + log2 l, the partial of
            // Eq. 1, merged by the split-merge kernel)
            const int64_t prow = static_cast<int64_t>(it.part_base + it.split) * kRows + r;
            float4 *po = reinterpret_cast<float4 *>(p.part_o + prow * kDv + kDvHalf * it.hb);
#pragma unroll 1
            for (int c = 0; c < kDvHalf / 64; ++c) {
                uint32_t o[64];
                tc::tmem_ld32(lane_addr + kColO + 64 * c, *reinterpret_cast<uint32_t(*)[32]>(&o[0]));
                tc::tmem_ld32(lane_addr + kColO + 64 * c + 32, *reinterpret_cast<uint32_t(*)[32]>(&o[32]));
                tc::tmem_wait_ld();
                if (c == kDvHalf / 64 - 1) {  // O is in registers: the next item may write it
                    tc::fence_before_sync();
                    __syncwarp();
                    tc::mbar_arrive_warp(OFREE);
                }
                if (whole) {
                    if (c > 0) {  // the store before has read the box
                        if (lane == 0) tc::bulk_wait_group_read0();
                        __syncwarp();
                    }
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        uint4 v;
                        v.x = pack_bf16x2(__uint_as_float(o[8 * j]) * inv, __uint_as_float(o[8 * j + 1]) * inv);
                        v.y = pack_bf16x2(__uint_as_float(o[8 * j + 2]) * inv, __uint_as_float(o[8 * j + 3]) * inv);
                        v.z = pack_bf16x2(__uint_as_float(o[8 * j + 4]) * inv, __uint_as_float(o[8 * j + 5]) * inv);
                        v.w = pack_bf16x2(__uint_as_float(o[8 * j + 6]) * inv, __uint_as_float(o[8 * j + 7]) * inv);
                        *reinterpret_cast<uint4 *>(box + lane * 128 + ((j ^ (lane & 7)) << 4)) = v;
                    }
                    tc::fence_proxy_async_smem();  // these writes before the TMA store reads them
                    __syncwarp();
                    if (lane == 0) {
                        tc::tma_store_3d(&maps.out32, box_addr, kDvHalf * it.hb + 64 * c, 32 * quarter, it.token);
                        tc::bulk_commit_group();
                    }
                } else {
#pragma unroll
                    for (int x = 0; x < 16; ++x)
                        po[c * 16 + x] = make_float4(__uint_as_float(o[4 * x]) * inv, __uint_as_float(o[4 * x + 1]) * inv,
                                                     __uint_as_float(o[4 * x + 2]) * inv, __uint_as_float(o[4 * x + 3]) * inv);
                }
            }
            if (whole && lane == 0) tc::bulk_wait_group_read0();
            if (it.hb == 0) {
                const float lse2 = ml.x + log2f(ml.y);
                if (whole) p.lse[static_cast<int64_t>(it.token) * kRows + r] = lse2 * kLn2;
                else p.part_lse[prow] = lse2;
            }
            __syncwarp();
            tc::mbar_arrive_warp(ITEMEMPTY(k % kItemSlots));
            return true;
        };
        int idx;
        if (next_item(0, idx) && idx >= 0) {
            MlaItem it = p.mitems[idx], prev = it;
            bool ok = load_q(it);
            for (int k = 0; ok; ++k) {
                // Q of item k, once the last S of the item before is done
                if (k >= 1 && !wait(QFREE, (k - 1) & 1)) break;
                tc::fence_after_sync();
#pragma unroll
                for (int c = 0; c < kQtChunks; ++c) tc::tmem_st32(lane_addr + kColQ + 32 * c, qv[c]);
                tc::tmem_wait_st();
                tc::fence_before_sync();
                __syncwarp();
                tc::mbar_arrive_warp(QREADY);
                if (k >= 1 && !epilogue(prev, k - 1)) break;
                prev = it;
                if (!next_item(k + 1, idx)) break;
                if (idx < 0) {
                    epilogue(prev, k);
                    break;
                }
                it = p.mitems[idx];
                ok = load_q(it);
            }
        }
    }

    tc::fence_before_sync();
    __syncthreads();
    if (*abort_flag && warp == 4) {
        tc::drain_copies(NFULL(0), kStages);
        tc::drain_copies(VFULL(0), kStages);
        tc::drain_copies(QFULL, 1);
        tc::drain_copies(STAGE(0), 4);
    }
    if (warp == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, kTmemCols);
    }
    if (tid == 0) {  // the last CTA out resets the work queue for the next run
        __threadfence();
        if (atomicAdd(p.sched + 1, 1) == static_cast<int>(gridDim.x) - 1) {
            p.sched[0] = 0;
            p.sched[1] = 0;
            __threadfence();
        }
    }
}

// 3-D map over rows of `cols` values (a multiple of 64), `rows` of them per
// outer index: the latent cache [blocks, bs, 576], Q [T, 128, 576] or the
// output [T, 128, 512]. Boxes of 64 columns x `box_rows` rows, 128-byte swizzle.
bool encode_rows_map(CUtensorMap *m, const void *base, int cols, int64_t row_stride_elems, int rows, int64_t outer,
                     int box_rows) {
    EncodeTiledFn enc = tensor_map_encoder();
    if (!enc) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(outer)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(row_stride_elems) * 2,
                             static_cast<cuuint64_t>(row_stride_elems) * 2 * rows};
    cuuint32_t box[3] = {64, static_cast<cuuint32_t>(box_rows), 1};
    cuuint32_t es[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool mla_tc_supported(int d_qk, int d_v, int hq, int hkv, int block_size) {
    return d_qk == kDq && d_v == kDv && hkv == 1 && hq == kRows &&
           (block_size == 16 || block_size == 32 || block_size == 64);
}

int mla_tc_keys_per_tile() { return kKeysT; }

int launch_mla_tc(const AttnParams &p, void *stream, int max_ctas) {
    if (p.num_mitems == 0) return FNPU_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (p.k_slot_stride % 8 != 0) return FNPU_EUNSUPPORTED;  // TMA strides are multiples of 16 bytes
    MlaMaps maps;
    if (!encode_rows_map(&maps.kv, p.k_cache, kDq, p.k_slot_stride, p.block_size, p.num_blocks, p.block_size) ||
        !encode_rows_map(&maps.q, p.q, kDq, kDq, kRows, p.num_tokens, kRows) ||
        !encode_rows_map(&maps.q32, p.q, kDq, kDq, kRows, p.num_tokens, 32) ||
        !encode_rows_map(&maps.out32, p.out, kDv, kDv, kRows, p.num_tokens, 32))
        return cuda_fail(cudaErrorInvalidValue, "cuTensorMapEncodeTiled (latent)");
    FNPU_CUDA_TRY(cudaFuncSetAttribute(mla_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
    FNPU_CUDA_TRY(launch_ex(mla_tc_kernel, p.num_mitems < max_ctas ? p.num_mitems : max_ctas, kThreads, kSmemBytes, st,
                            true, nullptr, p, maps));
    return launch_split_merge(p, stream);
}

}  // namespace fnpu
