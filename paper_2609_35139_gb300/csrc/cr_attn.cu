// Chunk-block-causal attention of the Repair Blocks (Sec. 4.1):
//   o_i = sum_{j : c(j) <= c(i)} softmax_j(q_i . k_j / sqrt(d)) v_j
// inside each request.  Chunk ids are non-decreasing along a request, so the
// keys visible to query i are exactly j < chunk_end[i]: a prefix.  The
// attention-topology ablations of App. F keep that shape: with A1 (token-
// causal) the keys are j <= i, with A2 (bidirectional) the whole request, with
// A3 (block-diagonal) j in [chunk_start[i], chunk_end[i]).  In every mode the
// visible keys of row i are one interval [lo(i), hi(i)) whose ends never
// decrease with i, so a query tile needs key tiles
// floor(lo(first row) / 128) .. ceil(hi(last row) / 128) - 1 and nothing
// else; other tiles are never loaded or multiplied.  Rows whose interval ends
// inside a key tile mask the rest of it; fully visible tiles do no masking
// work at all.
//
// A work item is a (request, head, pair of consecutive 128-query tiles w = 0, 1).  A
// CTA runs one item after another: its own block's, then items of blocks that have not
// started, which it takes over by cluster launch control as soon as an item's loads are
// out, so that the next item's Q, K and V arrive under this one's last tiles.  The item
// scheduler hands those on through two slots of shared memory; the own one is located
// before the wait for the kernel before, and nothing waits for the scheduler there.  Three
// warpgroups, the first of which gives registers to the other two:
//   warp 0      TMA: both Q tiles of an item (two buffers), then K_j and V_j per key
//               tile into a 4-deep ring shared by the two query tiles
//   warp 1 + w  MMA issue for query tile w (warp 1 also owns TMEM): per key
//               tile j, S_w,j+1 = Q_w K_j+1^T (M=128, N=128, K=d) as soon as
//               softmax w has read S_w,j into registers, and O_w += P_w,j V_j
//               (M=128, N=d, K=128, P read from TMEM, V MN-major from smem)
//               in halves of 64 keys, each once it is written.  Issue runs in a
//               converged warp with one elected lane, and each query tile has
//               its own issuer: the small MMAs of a d <= 64 head are cheap
//               enough that issue and barrier latency, not the tensor core, set
//               the pace.
//   warp 3      the item scheduler
//   warps 4..7  softmax group 0 (query tile 0), one row per thread
//   warps 8..11 softmax group 1 (query tile 1)
// Per key tile a softmax thread loads its whole S row (128 fp32) from TMEM in one
// round trip, masks it where the tile is partly visible, and writes
// P = 2^(s*scale*log2e - m) as bf16 pairs into its group's TMEM columns, from where
// the PV MMA reads it as the A operand (TMEM holds S_0, S_1, O_0, O_1, P_0, P_1: 512
// columns).  The two groups overlap each other's exponentials with their MMAs.
//
// The reference m of a row is its running maximum, moved lazily: only where a tile outgrows
// it by more than 2^8 in some row of the warp does the warp wait for the last product and
// rescale its O rows in TMEM and its row sums.  Any m gives the same softmax (it cancels in
// O / l), but not the same rounding of P to bf16: a row's largest P is 1 and exact, which
// is what counts where one key takes most of the weight.  With the maximum of the first
// visible key tile as a fixed reference the kernel was 9 % faster and up to 35 % less exact
// there (scores of 12 times unit variance, relative error 1.7e-3 -> 2.2e-3).
//
// What bounds it: with d = 64, a pair of 128 x 128 tiles costs the tensor core 1024
// clocks and each SM sub-partition's special-function unit 1024 (two tiles'
// exponentials at 8 a clock; 1126 measured with the packing and the sums), but only
// two softmax warps share a sub-partition and each is one serial chain, so the time
// follows the number of instructions in it (about 5.7 clocks each) and how well its
// registers hold a whole row.  Hence the mask built from one word per 32 keys, the unvoted
// waits, no wait for the last product before the exponentials unless O is rescaled, item
// fields re-read from shared memory instead of kept, and the rescale as a loop (unrolled, its
// code cost the short calls 0.1 us in instruction fetches).  One block per item cost 8700
// clocks around its tiles (block start, TMEM, barriers, first loads, last products).
// Measured, us: 5120 tokens of 10 chunks, 16 heads of 64 | 4102 tokens bidirectional |
// 5120 tokens block-diagonal | 16 ragged requests of 95617 tokens, 8 heads:
//   a block per item, groups in turns   64.2 | 81.8 | 25.3 | 836
//   as built                            56.9 | 73.3 | 21.5 | 669
// Tried and slower: four softmax warpgroups of half rows (76 us on the second shape:
// more barrier work and MIO queueing), the next tile's chunks loaded under the last
// exponentials (89 us), one hand-over of P instead of two halves (+4 %), spinning waits.
// O_w is read back and divided by l after the last tile.
#include <cuda_bf16.h>

#include "cr_internal.h"
#include "cr_ptx.cuh"

namespace cr {
namespace {

template <int D>
struct AttnCfg {
    static constexpr uint32_t kRowBytes = D * 2;            // one K/V/Q row
    static constexpr uint32_t kAtomBytes = 8 * kRowBytes;    // swizzle atom (8 rows)
    static constexpr uint32_t kTileBytes = 128 * kRowBytes;
    static constexpr uint32_t kSwz = (D == 64) ? SWZ_128B : SWZ_64B;
    static constexpr int kStages = 4;
    static constexpr uint32_t kQOff = 0;                                  // Q0, Q1 of two items
    static constexpr uint32_t kKVOff = 4 * kTileBytes;                    // K, V per stage
    static constexpr uint32_t kBarOff = kKVOff + kStages * 2 * kTileBytes;
    static constexpr uint32_t kSmemBytes = 1024 + kBarOff + 512;
    static constexpr uint32_t kTmemS = 0;      // S_w at w * 128 (fp32)
    static constexpr uint32_t kTmemO = 256;    // O_w at 256 + w * D (fp32)
    static constexpr uint32_t kTmemP = 384;    // P_w at 384 + w * 64 (bf16 pairs)
};

// Three warpgroups: control (TMA, two MMA issuers, the item scheduler) and two
// softmax groups.
// At launch each thread gets 65536 / 384 = 168 registers (the host checks
// this); the control warpgroup gives up most of its share so that the softmax
// threads can hold a whole S row: 48 * 128 + 2 * 224 * 128 <= 168 * 384 (the
// control warps keep only descriptors, counters and phases).
constexpr int kThreads = 384;
constexpr uint32_t kRegsLaunch = 168;
constexpr uint32_t kRegsCtl = 48;
constexpr uint32_t kRegsSoftmax = 224;
static_assert(kRegsCtl * 128 + 2 * kRegsSoftmax * 128 <= kRegsLaunch * kThreads,
              "register split exceeds the launch allocation");
constexpr float kRescaleLog2 = 8.0f;   // how far a row may outgrow its reference (log2 units)

// Scores 32 c .. 32 c + 31 of a row whose visible keys, relative to the tile, are
// [lo, hi): the others become -inf (a fully visible chunk is left alone).
template <int C>
__device__ __forceinline__ void mask_chunk(float (&s)[128], int lo, int hi, float neg_inf) {
    lo -= 32 * C;
    hi -= 32 * C;
    if (hi < 32 || lo > 0) {
        const uint32_t below = hi >= 32 ? ~0u : (hi <= 0 ? 0u : (1u << hi) - 1u);
        const uint32_t vis = lo <= 0 ? below : (lo >= 32 ? 0u : below & (~0u << lo));
#pragma unroll
        for (int i = 0; i < 32; ++i) s[32 * C + i] = (vis & (1u << i)) ? s[32 * C + i] : neg_inf;
    }
}
// 2^(s sc - m) of scores 32 c .. 32 c + 31 as bf16 pairs, added to the tile's row sums.
// A tile has eight of them, of 16 terms each, which tile_sum adds up: one sum that runs
// over the keys of a long row loses its small terms (262144 keys of weight 2^-24.3 under
// one of 1: half their part of the row sum).
template <int C>
__device__ __forceinline__ void exp_chunk(const float (&s)[128], float sc, float m, uint32_t* pk,
                                          float (&rs)[8]) {
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
        float t0, t1;
        ffma2(t0, t1, s[32 * C + i], s[32 * C + i + 1], sc, sc, -m, -m);
        const float e0 = ex2(t0);
        const float e1 = ex2(t1);
        const int q = (i >> 1) & 3;
        if (C == 0 && i < 8) {
            rs[2 * q] = e0;
            rs[2 * q + 1] = e1;
        } else {
            fadd2(rs[2 * q], rs[2 * q + 1], rs[2 * q], rs[2 * q + 1], e0, e1);
        }
        pk[i >> 1] = pack_bf16x2(e0, e1);
    }
}
__device__ __forceinline__ float tile_sum(const float (&rs)[8]) {
    return ((rs[0] + rs[1]) + (rs[2] + rs[3])) + ((rs[4] + rs[5]) + (rs[6] + rs[7]));
}
__device__ __forceinline__ float row_max(const float (&s)[128]) {
    float mx[8];   // independent chains
#pragma unroll
    for (int q = 0; q < 8; ++q) mx[q] = fmaxf(s[2 * q], s[2 * q + 1]);
#pragma unroll
    for (int i = 16; i < 128; i += 2) mx[(i >> 1) & 7] = fmax3(mx[(i >> 1) & 7], s[i], s[i + 1]);
    return fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])),
                 fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
}

// Exclusive end and start of the visible keys of request-local row i.
__device__ __forceinline__ int key_hi(const AttnParams& p, int rs, int len, int i) {
    if (p.mask_mode == CR_MASK_TOKEN_CAUSAL) return i + 1;
    if (p.mask_mode == CR_MASK_BIDIRECTIONAL) return len;
    return __ldg(p.chunk_end + rs + i);
}
__device__ __forceinline__ int key_lo(const AttnParams& p, int rs, int i) {
    return p.mask_mode == CR_MASK_BLOCK_DIAGONAL ? __ldg(p.chunk_start + rs + i) : 0;
}

// Byte offsets of a query tile's barriers from s_full[w].
constexpr int kOffS = 0, kOffFree = 16, kOffP0 = 32, kOffP1 = 48, kOffPV = 64, kOffO = 80;
template <int N>
struct At { static constexpr int value = N; };

// One work item: a (request, pair of query tiles, head), by its block index.
struct Item {
    int bid;     // < 0: no more items
    int head, q0, rs, len, kbase, n0, n1;
};
constexpr int kDesc = 8;
static_assert(sizeof(Item) == kDesc * 4, "descriptor size");

// Heaviest pairs of each request first.
__device__ __forceinline__ void locate_item(const AttnParams& p, int bid, Item& d) {
    const int order = bid / p.n_heads, pair = p.n_items - 1 - order;
    int a = 0, b = p.n_req - 1;   // the request with tile_prefix[r] <= pair
    while (a < b) {
        const int mid = (a + b + 1) >> 1;
        if (p.tile_prefix[mid] <= pair) a = mid;
        else b = mid - 1;
    }
    d.bid = bid;
    d.head = bid - order * p.n_heads;
    d.q0 = (pair - p.tile_prefix[a]) * 256;
    d.rs = p.req_start[a];
    d.len = p.req_start[a + 1] - d.rs;
}
// Both query tiles start at the key tile of the pair's first visible key,
// kbase = 128 * floor(lo(q0) / 128), so that every role takes the ring's tiles in order.
// (Under the block-diagonal mask the second tile's rows may start later; their leading key
// tiles are fully masked and contribute exact zeros.)  Tile j of an item is key tile
// kbase / 128 + j; query tile w needs j in [0, n_w), an empty second tile (past the
// request's end) none.  n_w is never negative: every role counts its ring slots by
// max(n0, n1), also where the chunk map, which is device memory that no host check sees,
// ends a tile's keys before the pair's first key tile.
__device__ __forceinline__ void count_tiles(const AttnParams& p, Item& d) {
    d.kbase = key_lo(p, d.rs, d.q0) & ~127;
    d.n0 = max(0, (key_hi(p, d.rs, d.len, min(d.q0 + 127, d.len - 1)) - d.kbase + 127) / 128);
    d.n1 = d.q0 + 128 < d.len
               ? max(0, (key_hi(p, d.rs, d.len, min(d.q0 + 255, d.len - 1)) - d.kbase + 127) / 128)
               : 0;
}

// kLse: also write each row's log-sum-exp (for the training step's backward); the
// inference forward's instantiation has none of that code.
template <int D, bool kLse>
__global__ void __launch_bounds__(kThreads, 1)
    attn_kernel(const __grid_constant__ CUtensorMap tmQKV, const __grid_constant__ AttnParams p) {
    using Cfg = AttnCfg<D>;
    constexpr int NS = Cfg::kStages;
    constexpr uint32_t IDESC_S = idesc_bf16(128, 128, false, false);
    constexpr uint32_t IDESC_PV = idesc_bf16(128, D, false, true);
    const float NEG_INF = -__int_as_float(0x7f800000);

    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Cfg::kBarOff);
    uint64_t* q_full = bars;              // [2] Q tiles of an item in buffer it & 1
    uint64_t* q_empty = bars + 2;         // [2] both issuers are done with them
    uint64_t* kv_full = bars + 4;
    uint64_t* kv_empty = kv_full + NS;
    // (the softmax groups address these five at fixed offsets, kOffS ..)
    uint64_t* s_full = kv_empty + NS;     // [2] S_w,j in TMEM
    uint64_t* s_free = s_full + 2;        // [2] S_w,j read into registers
    uint64_t* p_full = s_free + 2;        // [h][w] half h of P_w,j (64 keys) in TMEM
    uint64_t* pv_done = p_full + 4;       // [2] O_w += P_w,j V_j complete
    uint64_t* o_free = pv_done + 2;       // [2] O_w of an item read into registers
    uint64_t* drain = o_free + 2;         // [2]
    uint64_t* item_full = drain + 2;      // [2] the descriptor of item it in slot it & 1
    uint64_t* item_empty = item_full + 2; // [2] producer and issuers have read it, and the 8
                                          //     softmax warps are done with the item
    uint64_t* loads_out = item_empty + 2; // the loads of an item have all been issued
    uint64_t* clc_full = loads_out + 1;   // the answer to a request for another item
    // (32 barriers: 256 bytes)
    uint4* clc_answer = reinterpret_cast<uint4*>(smem + Cfg::kBarOff + 320);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + Cfg::kBarOff + 336);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
    volatile int* desc = abort_flag + 3;  // [2][kDesc]

    const uint32_t warp = warp_id(), lane = lane_id();
    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(&kv_full[s], 1);
            mbar_init(&kv_empty[s], 2);   // both issuers release each stage
        }
        for (int w = 0; w < 2; ++w) {
            mbar_init(&q_full[w], 1);
            mbar_init(&q_empty[w], 2);
            mbar_init(&s_full[w], 1);
            mbar_init(&s_free[w], 4);
            mbar_init(&p_full[2 * w], 4);
            mbar_init(&p_full[2 * w + 1], 4);
            mbar_init(&pv_done[w], 1);
            mbar_init(&o_free[w], 4);
            mbar_init(&drain[w], 1);
            mbar_init(&item_full[w], 1);
            mbar_init(&item_empty[w], 11);
        }
        mbar_init(loads_out, 1);
        mbar_init(clc_full, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    // The CTA's own block, as far as it does not depend on an earlier kernel, before the wait
    // for that; each role then counts its key tiles by itself.  With item 0 handed from the
    // scheduler through its slot, after the wait, a call of one round of short items was
    // slower (us: 60 tokens 5.0 instead of 4.3, 1024 tokens block-diagonal 7.4 instead of
    // 6.5).  The softmax warps read it from the slot: kept in registers it cost them 1 to 6 %.
    Item own{};
    locate_item(p, static_cast<int>(blockIdx.x), own);
    if (threadIdx.x == 96) {
        const int* v = reinterpret_cast<const int*>(&own);
#pragma unroll
        for (int k = 0; k < kDesc; ++k) desc[k] = v[k];
    }
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();   // qkv and the chunk map come from earlier kernels
    const uint32_t tmem_base = *tmem_slot;
    const WaitCtx wc{abort_flag, p.status};

    // The descriptor of the CTA's it-th item, for the producer and issuer warps; false at
    // the end (or when a role has given up).
    auto next_item = [&](uint32_t it, Item* d) -> bool {
        if (it == 0) {
            *d = own;
            count_tiles(p, *d);
        } else {
            if (!mbar_wait_warp(&item_full[it & 1u], (it >> 1) & 1u, wc, 131)) return false;
            int* v = reinterpret_cast<int*>(d);
#pragma unroll
            for (int k = 0; k < kDesc; ++k) v[k] = desc[(it & 1u) * kDesc + k];
            __syncwarp();
        }
        if (lane == 0) mbar_arrive(&item_empty[it & 1u]);
        return d->bid >= 0;
    };

    if (warp < 4) {
        setmaxnreg_dec<kRegsCtl>();
        if (warp == 0) {
            // ---------------------------------------------------- TMA producer
            // (the whole warp runs the loop; one elected lane issues)
            if (elect_one()) tma_prefetch(&tmQKV);
            __syncwarp();
            bool ok = true;
            int st = 0;
            uint32_t ph = 0;
            uint32_t it = 0;   // items
            // An issuer whose wait gave up releases buffers whose fill it has not seen land:
            // once any role has given up (its flag is set before such a release, and read
            // after the release was seen), nothing is filled again.
            auto may_fill = [&](uint64_t* empty, uint32_t parity, unsigned site) -> bool {
                const uint32_t a = smem_u32(empty);
                const bool ready = mbar_test_wait(a, parity);
                int gone = *wc.abort;
                if (!ready) gone = mbar_wait_slow(a, parity, wc, site) ? *wc.abort : 1;
                return __all_sync(0xffffffffu, gone == 0);
            };
            for (Item d; ok && next_item(it, &d); ++it) {
                const int head = d.head, n_max = max(d.n0, d.n1);
                uint64_t* qf = &q_full[it & 1u];
                uint8_t* qt = smem + Cfg::kQOff + (it & 1u) * 2 * Cfg::kTileBytes;
                if (!(ok = may_fill(&q_empty[it & 1u], ((it >> 1) & 1u) ^ 1u, 122))) break;
                if (elect_one()) {
                    mbar_expect_tx(qf, 2 * Cfg::kTileBytes);
                    tma_load_2d(qt, &tmQKV, qf, head * D, d.rs + d.q0);
                    tma_load_2d(qt + Cfg::kTileBytes, &tmQKV, qf, head * D, d.rs + d.q0 + 128);
                }
                __syncwarp();
                for (int j = 0; j < n_max; ++j) {
                    if (!(ok = may_fill(&kv_empty[st], ph ^ 1u, 121))) break;
                    uint8_t* kt = smem + Cfg::kKVOff + st * 2 * Cfg::kTileBytes;
                    if (elect_one()) {
                        mbar_expect_tx(&kv_full[st], 2 * Cfg::kTileBytes);
                        tma_load_2d(kt, &tmQKV, &kv_full[st], p.d_b + head * D, d.rs + d.kbase + j * 128);
                        tma_load_2d(kt + Cfg::kTileBytes, &tmQKV, &kv_full[st], 2 * p.d_b + head * D,
                                    d.rs + d.kbase + j * 128);
                    }
                    __syncwarp();
                    if (++st == NS) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
                if (ok && elect_one()) mbar_arrive(loads_out);
                __syncwarp();
            }
            __syncthreads();   // all roles meet: none gives up after this
            if (__any_sync(0xffffffffu, *wc.abort != 0)) {
                // copies may be under way whose reader has given up: the last fill of each
                // ring slot (those from st on a lap earlier) and of each Q buffer; a wait for
                // the phase before the first passes
                for (int s = 0; s < NS; ++s) mbar_wait_landed(&kv_full[s], s < st ? ph : ph ^ 1u);
                for (uint32_t b = 0; b < 2; ++b) mbar_wait_landed(&q_full[b], (((it + 1u - b) >> 1) - 1u) & 1u);
            }
        } else if (warp == 1 || warp == 2) {
            // ---------------------------------------------------- MMA issuers
            // Warp 1 + w issues for query tile w: per key tile j, S_w,j+1 as
            // soon as softmax w has read S_w,j out of TMEM, then O_w += P_w,j V_j
            // once P_w,j is written.  The whole warp runs the loop and computes
            // the descriptors; one elected lane issues the MMAs and commits.
            const int w = static_cast<int>(warp) - 1;
            // Descriptors are built once; a K=16 step adds 32 bytes (2 units of
            // 16 B) to the start address, a stage adds 2 tiles, a V step 16 rows.
            constexpr uint64_t kStageStep = (2 * Cfg::kTileBytes) >> 4;
            const uint64_t dq0 = smem_desc(smem_u32(smem + Cfg::kQOff + w * Cfg::kTileBytes), 16,
                                           Cfg::kAtomBytes, Cfg::kSwz);
            const uint64_t dk0 = smem_desc(smem_u32(smem + Cfg::kKVOff), 16, Cfg::kAtomBytes, Cfg::kSwz);
            const uint64_t dv0 = smem_desc(smem_u32(smem + Cfg::kKVOff + Cfg::kTileBytes),
                                           Cfg::kTileBytes, Cfg::kAtomBytes, Cfg::kSwz);
            const uint32_t ds = tmem_base + Cfg::kTmemS + w * 128;
            const uint32_t dout = tmem_base + Cfg::kTmemO + w * D;
            const uint32_t pa = tmem_base + Cfg::kTmemP + w * 64;
            // A wait that gives up leaves stale operands behind, which only this CTA's own
            // accumulators would show; the later waits give up at once.
            const uint32_t bar = smem_u32(&s_full[w]);
            const bool leader = elect_one();
            auto settle = [&](bool ready, uint32_t a, uint32_t parity, unsigned site) {
                if (!ready) mbar_wait_slow(a, parity, wc, site);
                __syncwarp();
                tc_fence_after();
            };
            auto wait = [&](uint64_t* b, uint32_t parity, unsigned site) {
                const uint32_t a = smem_u32(b);
                settle(mbar_test_wait(a, parity), a, parity, site);
            };
            int sl = 0;           // ring slot of the tile in hand, its phase: every role walks
            uint32_t sp = 0;      // all n_max slots of an item
            uint32_t ns = 0, np = 0, no = 0;   // S tiles read, P tiles multiplied, O tiles started
            int n, n_max;
            uint32_t it = 0;   // items
            for (;; ++it) {
                {
                    Item d;
                    if (!next_item(it, &d)) break;
                    n = w == 0 ? d.n0 : d.n1;
                    n_max = max(d.n0, d.n1);
                }
                const uint64_t dq = dq0 + (it & 1u) * ((2 * Cfg::kTileBytes) >> 4);
                auto issue_s = [&](int slot) {
                    const uint64_t dk = dk0 + static_cast<uint64_t>(slot) * kStageStep;
                    if (leader) {
#pragma unroll
                        for (int k = 0; k < D / 16; ++k)
                            mma_bf16_ss(ds, dq + 2 * k, dk + 2 * k, IDESC_S, k != 0 ? 1u : 0u);
                        mma_commit(&s_full[w]);
                    }
                    __syncwarp();
                };
                wait(&q_full[it & 1u], (it >> 1) & 1u, 221);
                if (n > 0) {
                    wait(&kv_full[sl], sp, 222);
                    issue_s(sl);
                }
                for (int j = 0; j < n; ++j) {
                    const int s1 = sl + 1 == NS ? 0 : sl + 1;
                    const uint32_t p1 = s1 == 0 ? sp ^ 1u : sp;
                    // the next tile's operands first, so that S_w,j+1 goes out as soon as
                    // S_w,j has been read (as it has to be before the next item's first)
                    if (j + 1 < n) wait(&kv_full[s1], p1, 222);
                    settle(mbar_test_wait_at<kOffFree>(bar, ns & 1u), bar + kOffFree, ns & 1u, 223);
                    ++ns;
                    if (j + 1 < n) {
                        issue_s(s1);
                    } else {
                        if (leader) mma_commit(&q_empty[it & 1u]);
                        __syncwarp();
                    }
                    // the item before has had its O_w read
                    if (j == 0 && no++ > 0) wait(&o_free[w], (no - 2u) & 1u, 225);
                    // PV in two halves of 64 keys, each issued as soon as softmax w has
                    // written it (its V tile arrived with the K tile of S_w,j)
                    const uint64_t dv = dv0 + static_cast<uint64_t>(sl) * kStageStep;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const bool ready = h == 0 ? mbar_test_wait_at<kOffP0>(bar, np & 1u)
                                                  : mbar_test_wait_at<kOffP1>(bar, np & 1u);
                        settle(ready, bar + (h == 0 ? kOffP0 : kOffP1), np & 1u, 224);
                        if (leader) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                // P from TMEM (16 keys = 8 columns); V: rows = keys (the K
                                // dimension), d contiguous (MN-major); 16 keys = two 8-row atoms.
                                const int kk = 4 * h + q;
                                mma_bf16_ts(dout, pa + kk * 8, dv + kk * ((16 * Cfg::kRowBytes) >> 4),
                                            IDESC_PV, (j > 0 || kk != 0) ? 1u : 0u);
                            }
                            if (h == 1) {
                                mma_commit(&pv_done[w]);
                                mma_commit(&kv_empty[sl]);
                            }
                        }
                        __syncwarp();
                    }
                    ++np;
                    sl = s1;
                    sp = p1;
                }
                // the other query tile's key tiles past this one's: released in order,
                // so that no wait of this warp is ever two fills of a slot ahead
                if (n == 0 && leader) mbar_arrive(&q_empty[it & 1u]);
                __syncwarp();
                for (int j = n; j < n_max; ++j) {
                    wait(&kv_full[sl], sp, 226);
                    if (leader) mbar_arrive(&kv_empty[sl]);
                    __syncwarp();
                    if (++sl == NS) {
                        sl = 0;
                        sp ^= 1u;
                    }
                }
            }
            if (elect_one()) mma_commit(&drain[w]);
            __syncwarp();
            // (an early exit must not leave an MMA that still writes TMEM)
            if (!mbar_wait_warp(&drain[w], 0, wc, 227)) mbar_wait_landed(&drain[w], 0);
            __syncthreads();
        } else {
            // ---------------------------------------------------- item scheduler
            // The CTA's first item is its own block; once an item's loads are out, the
            // next one is taken over from a block that has not started yet (cluster
            // launch control), so that its first tiles load under this item's last ones.
            // (one item_empty barrier per slot: a softmax group without a tile runs ahead
            // by one item, never by two)
            uint32_t asked = 0;   // requests made
            auto publish = [&](uint32_t it, int bid) -> bool {
                Item d{};
                d.bid = bid;
                if (bid >= 0) {
                    locate_item(p, bid, d);
                    count_tiles(p, d);
                }
                if (!mbar_wait_warp(&item_empty[it & 1u], ((it >> 1) & 1u) ^ 1u, wc, 132)) return false;
                const int* v = reinterpret_cast<const int*>(&d);
                if (lane == 0) {
#pragma unroll
                    for (int k = 0; k < kDesc; ++k) desc[(it & 1u) * kDesc + k] = v[k];
                    mbar_arrive(&item_full[it & 1u]);
                }
                __syncwarp();
                return true;
            };
            int bid = -1;
            uint32_t it = 0;
            bool ok = true;
            if (lane == 0) mbar_arrive(&item_full[0]);   // item 0 stands there already
            do {
                if (!(ok = mbar_wait_warp(loads_out, it & 1u, wc, 134))) break;
                ++it;
                if (elect_one()) {
                    mbar_expect_tx(clc_full, 16);
                    clc_try_cancel(clc_answer, clc_full);
                }
                __syncwarp();
                if (!(ok = mbar_wait_warp(clc_full, asked & 1u, wc, 135))) {
                    mbar_wait_landed(clc_full, asked & 1u);   // the answer is a copy, too
                    break;
                }
                ++asked;
                bid = clc_cancelled_block(clc_answer);
                fence_async_smem();   // read before the next answer overwrites it
                __syncwarp();
            } while (bid >= 0 && (ok = publish(it, bid)));
            if (ok) publish(it, -1);
            __syncthreads();
        }
    } else {
        setmaxnreg_inc<kRegsSoftmax>();
        // ---------------------------------------------------- softmax groups
        const int w = (warp >= 8) ? 1 : 0;
        const uint32_t quad = warp & 3u;
        const uint32_t lane_off = (quad * 32u) << 16;
        const uint32_t ts = tmem_base + lane_off + Cfg::kTmemS + w * 128;
        const uint32_t to = tmem_base + lane_off + Cfg::kTmemO + w * D;
        const uint32_t tp = tmem_base + lane_off + Cfg::kTmemP + w * 64;
        const float sc = p.scale_log2;
        float m = NEG_INF, l = 0.0f;
        uint32_t ns = 0, np = 0;         // S tiles read, P tiles written
        int n = 0, cend = 0, cbeg = 0;   // the item's key tiles, the row's visible keys
        const uint32_t bar = smem_u32(&s_full[w]);
        // A wait that gives up (the status word then says so) leaves stale scores
        // behind, which only this CTA's own rows would show: the loop goes on, its
        // later waits give up at once, and every role still reaches the end.
        auto settle = [&](bool ready, uint32_t off, uint32_t parity, unsigned site) {
            if (!ready) mbar_wait_slow(bar + off, parity, wc, site);
            __syncwarp();
            tc_fence_after();
        };
        auto hand_over = [&](auto off) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_at<decltype(off)::value>(bar);
        };
        // the whole S row of the next tile in registers: one TMEM round trip, after
        // which the tensor core may overwrite S
        auto take_s = [&](float (&s)[128]) {
            settle(mbar_test_wait_at<kOffS>(bar, ns & 1u), kOffS, ns & 1u, 321);
            ++ns;
            tmem_ld64(ts, s);
            tmem_ld64(ts + 64, s + 64);
            tmem_wait_ld();
        };
        auto mask_s = [&](float (&s)[128], int j) {
            const int lo = cbeg - j * 128, hi = cend - j * 128;
            if (__any_sync(0xffffffffu, hi < 128 || lo > 0)) {
                mask_chunk<0>(s, lo, hi, NEG_INF);
                mask_chunk<1>(s, lo, hi, NEG_INF);
                mask_chunk<2>(s, lo, hi, NEG_INF);
                mask_chunk<3>(s, lo, hi, NEG_INF);
            }
        };
        // P of one tile (2^(s*sc - m_ref) as bf16 pairs) in two halves of 64 keys, each
        // handed over once its store has landed.  P_w is free once PV_w of the tile
        // before has completed: the probe's answer comes in under the second chunk's
        // exponentials.
        auto put_p = [&](const float (&s)[128], float m_ref) {
            uint32_t pk[32];
            float rs[8];
            exp_chunk<0>(s, sc, m_ref, pk, rs);
            const bool pv = mbar_test_wait_at<kOffPV>(bar, (np & 1u) ^ 1u);
            exp_chunk<1>(s, sc, m_ref, pk + 16, rs);
            settle(pv, kOffPV, (np & 1u) ^ 1u, 322);
            ++np;
            tmem_st32u(tp, pk);
            tmem_wait_st();
            hand_over(At<kOffP0>{});
            exp_chunk<2>(s, sc, m_ref, pk, rs);
            exp_chunk<3>(s, sc, m_ref, pk + 16, rs);
            tmem_st32u(tp + 32, pk);
            l += tile_sum(rs);
            tmem_wait_st();
            hand_over(At<kOffP1>{});
        };
        // the last PV product of an item
        auto wait_last = [&]() {
            settle(mbar_test_wait_at<kOffPV>(bar, (np & 1u) ^ 1u), kOffPV, (np & 1u) ^ 1u, 324);
        };
        // m, P and l of every key tile
        auto sweep = [&]() {
            m = NEG_INF;
            l = 0.0f;
            for (int j = 0; j < n; ++j) {
                float s[128];
                take_s(s);
                mask_s(s, j);
                hand_over(At<kOffFree>{});
                const float mx = row_max(s) * sc;
                if (j == 0) {
                    m = mx;
                } else if (__any_sync(0xffffffffu, mx > m + kRescaleLog2)) {
                    const float m_new = fmaxf(m, mx);
                    const float alpha = (m == m_new) ? 1.0f : ex2(m - m_new);
                    wait_last();   // O_w is free
#pragma unroll 1
                    for (int c = 0; c < D; c += 16) {
                        float o[16];
                        tmem_ld16(to + c, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] *= alpha;
                        tmem_st16(to + c, o);
                    }
                    l *= alpha;
                    m = m_new;
                }
                // (a row whose keys start in a later tile has m = -inf: its P is 0)
                put_p(s, (m == NEG_INF) ? 0.0f : m);
            }
        };
        // (few values live across the key tiles: the softmax threads' registers are full,
        // and the item's descriptor stays in its slot until all of them are done with it)
        uint32_t it = 0;
        for (bool more = true; more; ++it) {
            const volatile Item* d = reinterpret_cast<const volatile Item*>(desc + (it & 1u) * kDesc);
            more = it == 0 || (mbar_wait_warp(&item_full[it & 1u], (it >> 1) & 1u, wc, 131) && d->bid >= 0);
            n = 0;
            if (more) {
                // visible keys of this row, relative to the first key tile (a row past
                // the request's end is never stored, but shares its warp's votes: one key)
                Item o;
                o.q0 = d->q0;
                o.rs = d->rs;
                o.len = d->len;
                const int qrow = o.q0 + 128 * w + static_cast<int>(quad * 32 + lane);
                const bool in = qrow < o.len;
                cend = in ? key_hi(p, o.rs, o.len, qrow) : 1;
                cbeg = in ? key_lo(p, o.rs, qrow) : 0;
                if (it == 0) {
                    count_tiles(p, o);
                    n = w == 0 ? o.n0 : o.n1;
                } else {
                    o.kbase = d->kbase;
                    n = w == 0 ? d->n0 : d->n1;
                }
                cend -= o.kbase;
                cbeg -= o.kbase;
            }
            if (n > 0) {
                sweep();
                // (what does not need O before the wait for it)
                const int qrow = d->q0 + 128 * w + static_cast<int>(quad * 32 + lane);
                const bool valid = qrow < d->len;
                const int head = d->head;
                const int64_t row = d->rs + qrow;
                uint4* d4 = reinterpret_cast<uint4*>(p.out + row * p.d_b + head * D);
                const float inv = 1.0f / l;
                // the row's log-sum-exp for a backward pass: P = 2^(s sc - (m + log2 l))
                if (kLse && valid)
                    p.lse[static_cast<int64_t>(head) * p.req_start[p.n_req] + row] = m + log2f(l);
                wait_last();
                // O_w into registers, so that the next item may overwrite it
                float o[D];
                if constexpr (D == 64) {
                    tmem_ld64(to, o);
                } else {
                    tmem_ld32(to, o);
                }
                tmem_wait_ld();
                hand_over(At<kOffO>{});
                if (valid) {
#pragma unroll
                    for (int c = 0; c < D; c += 8)
                        d4[c / 8] = make_uint4(pack_bf16x2(o[c] * inv, o[c + 1] * inv),
                                               pack_bf16x2(o[c + 2] * inv, o[c + 3] * inv),
                                               pack_bf16x2(o[c + 4] * inv, o[c + 5] * inv),
                                               pack_bf16x2(o[c + 6] * inv, o[c + 7] * inv));
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&item_empty[it & 1u]);
        }
        tc_fence_before();
        __syncthreads();
    }
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

template <int D, bool kLse>
cr_status launch_d(const CUtensorMap& tm, const AttnParams& p, cudaStream_t st) {
    using Cfg = AttnCfg<D>;
    auto kern = attn_kernel<D, kLse>;
    static unsigned long long attr_done = 0;   // one per template instantiation
    const cr_status sa = ensure_smem_attr(kern, static_cast<int>(Cfg::kSmemBytes), &attr_done);
    if (sa != CR_OK) return sa;
    // The softmax warpgroups raise their register budget inside the kernel;
    // that only completes if the launch reserved the 168 registers per thread
    // the split assumes.  Refuse to launch a build that reserves fewer.
    static int regs_ok = -1;   // per template instantiation; same answer on every device
    int ok = __atomic_load_n(&regs_ok, __ATOMIC_ACQUIRE);
    if (ok < 0) {
        cudaFuncAttributes fa;
        const cr_status sf = cuda_check(cudaFuncGetAttributes(&fa, kern));
        if (sf != CR_OK) return sf;
        ok = (fa.numRegs >= static_cast<int>(kRegsLaunch) && fa.maxThreadsPerBlock >= kThreads) ? 1 : 0;
        __atomic_store_n(&regs_ok, ok, __ATOMIC_RELEASE);
    }
    if (!ok) return CR_ERR_UNSUPPORTED;
    const int grid = p.n_items * p.n_heads;
    return launch_pdl(kern, dim3(grid), dim3(kThreads), Cfg::kSmemBytes, st, tm, p);
}

// chunk_start[t] = the request-local index of the first token of t's chunk:
// the smallest u with chunk_end[u] > i, i = t's request-local index (tokens of
// earlier chunks have chunk_end <= their chunk's end <= i, tokens of i's chunk
// have chunk_end > i).  One thread per token, binary searches over the
// request starts and over the request's non-decreasing chunk_end; the result
// lies in [0, i] whatever the map holds.
__global__ void __launch_bounds__(256)
    chunk_start_kernel(const int32_t* __restrict__ chunk_end, int32_t* __restrict__ chunk_start,
                       const __grid_constant__ AttnParams p, int n_tokens) {
    pdl_launch_dependents();
    pdl_wait();   // the chunk map comes from an earlier kernel
    const int t = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
    if (t >= n_tokens) return;
    int r0 = 0, r1 = p.n_req - 1;       // the request r with req_start[r] <= t
    while (r0 < r1) {
        const int mid = (r0 + r1 + 1) >> 1;
        if (p.req_start[mid] <= t) r0 = mid;
        else r1 = mid - 1;
    }
    const int rs = p.req_start[r0];
    const int i = t - rs;
    int a = 0, b = i;
    while (a < b) {
        const int mid = (a + b) >> 1;
        if (__ldg(chunk_end + rs + mid) > i) b = mid;
        else a = mid + 1;
    }
    chunk_start[t] = a;
}

}  // namespace

cr_status launch_chunk_starts(const int32_t* chunk_end, const AttnParams& p, int64_t n_tokens,
                              int32_t* chunk_start, cudaStream_t st) {
    if (n_tokens < 1) return CR_OK;
    const int grid = static_cast<int>((n_tokens + 255) / 256);
    return launch_pdl(chunk_start_kernel, dim3(grid), dim3(256), 0, st, chunk_end, chunk_start, p,
                      static_cast<int>(n_tokens));
}

cr_status launch_attention(const uint16_t* qkv, int64_t n_tokens, int head_dim,
                           const AttnParams& p, cudaStream_t st) {
    if (head_dim != 32 && head_dim != 64) return CR_ERR_UNSUPPORTED;
    if (p.n_items <= 0) return CR_OK;
    CUtensorMap tm;
    if (!make_tmap_2d(&tm, qkv, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3ull * p.d_b, n_tokens,
                      3ull * p.d_b * 2, head_dim, 128,
                      head_dim == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B))
        return CR_ERR_INVALID_ARG;
    if (p.lse) return head_dim == 64 ? launch_d<64, true>(tm, p, st) : launch_d<32, true>(tm, p, st);
    return head_dim == 64 ? launch_d<64, false>(tm, p, st) : launch_d<32, false>(tm, p, st);
}

}  // namespace cr
