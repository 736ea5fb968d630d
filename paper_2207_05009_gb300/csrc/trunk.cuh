// Layer-fused forward of the network's trunk (Sec. 4.2: eight fully
// connected layers of 256 with ReLU) and of the linear head on sm_103a: a
// tile's activations stay in shared memory from the encoded input to the
// head's output; only that and what the backward pass needs leaves the SM (each
// layer's bf16 output, stored by TMA straight from the shared-memory tile, and
// its ReLU bits).
//
// A pair of CTAs (a cluster of 2, tcgen05 cta_group::2) works on a tile of 256
// rows, 128 in each, against the layer's 256 x K weights, half of whose rows
// each CTA holds.  Per CTA (persistent, one per SM) two tiles are in flight,
// in slots 0 and 1, each with its own 64 KB activation buffer and 256 TMEM
// columns; the jobs (slot, layer) run in the order A0 B0 A1 B1 ... A7 B7, so
// the epilogue of one slot overlaps the MMAs of the other.  The weights
// stream from L2 through a ring of five 16 KB stages (one K-block of 64 inputs
// of a half matrix each); both slots' jobs of a layer use a K-block before its
// stage is refilled.  So a CTA takes 64 KB of weights for two jobs (256 KB
// through three stages when each CTA worked alone), which leaves room for
// the biases and the ReLU bits: those used to be 4-byte accesses to global
// memory in every epilogue.
//
// Measured on 524,288 rows (ncu): the forward 645 us with one CTA per tile and
// the head 45 us as a GEMM that read its input back; the trunk alone now takes
// 515 us with ReLU bits and all layers stored, with the head as a ninth job 556
// us.  Seven data-gradient layers 495 us, now eight in 445 us.  The stores of 2.15
// GB alone take 345 us at the rate the memory takes them, the MMAs alone 246
// us (everything but them taken out), everything but the stores 400 us.  So
// it is bound by its epilogue, whose warps serve the two slots in turn, and by
// what the stores take from it.
//
// Warp roles: 0 weight loads; 1 TMEM, MMA issue (lane 0 of the even CTA; the
// odd one's passes "this K-block has landed here" on to the even CTA); 2 lane
// 0 TMA stores of the finished activation tiles; 3 lane 0 input tiles; 4..19
// the epilogue (warp w reads TMEM lanes 32 (w % 4) .. +31 and a quarter of the
// 32-column chunks).
//
// The odd CTA's arrivals on the even one's barriers have the default scope,
// .cta.  What each announces is complete, in the memory that the tensor core
// reads, before it is made: kready, the K-block, waited for on wfull and passed
// through fence.proxy.async; px, the input tile, whose TMA load has been waited
// for on xfull; aready, the tile's bf16 values, written before
// fence.proxy.async, and the accumulator, read before tcgen05.wait::ld and
// tcgen05.fence::before_thread_sync.  No generic read of the other CTA's memory
// follows.  Release and acquire at cluster scope cost (forward of 200,001
// points / training step of 4096 x 128 / distillation at depth 7, us): none 230
// / 1760 / 6773, px alone 231.5 / 1775 / 6940; releases on all 230 -> 244 /
// 1760 -> 1880 / 7867 -> 8913.
//
// The epilogue writes its bf16 results into
// the activation buffer in the layout a 128-byte-swizzled TMA load would
// produce (row r's 16-byte chunk c at r * 128 + ((c ^ (r & 7)) * 16) of
// its 64-column block), so the next layer's MMA and the TMA store read it
// as they read TMA-loaded tiles.  Every mbarrier wait is bounded, as in
// k_gemm: a wait that gives up raises the abort flag and bit 1 of the error
// word, every role drains what it has in flight, and the CTAs of a pair meet
// before either exits.
#pragma once

#include "gemm.cuh"

namespace plo {
namespace gemm {

constexpr int TR_LAYERS = 8;
constexpr int TR_N = 256;
constexpr int TR_HEAD = 64;  // outputs of the linear head (padded)
constexpr int TR_WSTAGES = 5;
constexpr int TR_WROWS = TR_N / 2;             // weight rows in each CTA of the pair
constexpr int TR_WBYTES = TR_WROWS * 128;      // one K-block of half a weight matrix: 128 rows x 128 B
constexpr int TR_KBYTES = BM * 128;            // one K-block of an activation tile: 128 rows x 128 B
constexpr int TR_ABYTES = 4 * TR_KBYTES;       // a 128 x 256 bf16 activation tile
constexpr int TR_BIAS_BYTES = (TR_LAYERS * TR_N + TR_HEAD) * 4;
constexpr int TR_BITS_BYTES = BM * TR_N / 8;   // ReLU bits of an activation tile: 128 rows x 32 B
constexpr int TR_EPI_WARP0 = 4;
constexpr int TR_EPI_GROUPS = 4;                      // epilogue warps per TMEM lane quadrant
constexpr int TR_CHUNKS = TR_N / 32 / TR_EPI_GROUPS;  // 32-column chunks per epilogue warp
constexpr int TR_EPI_WARPS = 4 * TR_EPI_GROUPS;
constexpr int TR_THREADS = 32 * (TR_EPI_WARP0 + TR_EPI_WARPS);
static_assert(TR_CHUNKS == 2, "an epilogue warp's two chunks share one 8-byte word of ReLU bits");
__host__ __device__ constexpr size_t trunk_smem_bytes() {
    return 1024 + 2 * (size_t)TR_ABYTES + (size_t)TR_WSTAGES * TR_WBYTES + TR_BIAS_BYTES + 2 * TR_BITS_BYTES + 512;
}

// Indexed by job j of a tile: the forward's layer j, or in the backward chain
// the data gradient through layer 8 - j.
struct TrunkMaps {
    CUtensorMap x;                 // input tile, boxes 64 x 128, 128-byte swizzle: the encoded samples [M][64]
                                   // (forward), the gradient after the trunk [M][64 XKB] (backward)
    CUtensorMap h[TR_LAYERS];      // job j's output [M][256], boxes 64 x 128 (TMA stores)
    CUtensorMap raw;               // HEAD: the head's FP32 output [M][64], boxes 32 x 128, 128-byte swizzle
};

struct TrunkArgs {
    const __nv_bfloat16* w[TR_LAYERS + 1];  // B operand [256][K]: W_j (forward; the head's last, [64][256]), W_l^T
                                            // (backward); K = 64 XKB for j = 0
    const float* bias[TR_LAYERS + 1];  // forward: layer j's bias
    float* out;                    // HEAD without BITS: if not NULL the head's output goes here, [M][n_out], 16-byte aligned,
    int n_out;                     // instead of through `raw`
    uint32_t* bits[TR_LAYERS];     // [M][8] words: forward, layer j's ReLU bits (written if BITS);
                                   // backward, the ReLU bits of H_l (read: the mask of the gradient)
    uint32_t store;                // bit j: store job j's output through h[j]
    unsigned int* err;          // bit 1: a pipeline wait gave up
    uint32_t wait_limit;        // polls per wait (0: sm100::WAIT_LIMIT)
    int M;
};

struct TrCtl {
    uint64_t wfull[TR_WSTAGES], wempty[TR_WSTAGES];
    uint64_t xfull[2], xfree[2], tfull[2], adone[2], sdone[2];  // xfree: the slot's last store has read its tile
    uint64_t kready[TR_WSTAGES], px[2], aready[2];  // even CTA: both halves of a K-block / the odd CTA's input
                                                    // tile have landed; both CTAs have written the slot's tile
                                                    // (wfull: the odd CTA's own half)
    uint64_t mfull[2];                               // backward: the slot's mask bits have landed
    uint64_t drain;
    uint32_t tmem;
    int abort;
};

// A wait of at most `limit` polls.
__device__ __forceinline__ bool tr_wait(uint64_t* bar, uint32_t ph, uint32_t limit, TrCtl* ctl, unsigned int* err) {
    const uint32_t a = sm100::smem_addr(bar);
    for (uint32_t it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(ph)
            : "memory");
        if (done) return true;
        if ((it & 1023u) == 1023u && *(volatile int*)&ctl->abort) return false;
    }
    *(volatile int*)&ctl->abort = 1;
    atomicOr(err, 2u);
    return false;
}

// The pair's tiles are P + k n_pairs (P: index of the CTA pair); tiles 2j and
// 2j + 1 of that list form round j (slots 0 and 1).  Every role walks the
// same job list.
__device__ __forceinline__ int tr_tile(int round, int slot, int n_tiles) {
    const int t = (int)(blockIdx.x >> 1) + (2 * round + slot) * (int)(gridDim.x >> 1);
    return t < n_tiles ? t : -1;
}

// A stage of the weight ring and the parity of its current use.
struct TrStage {
    int s = 0;
    uint32_t ph = 0;
    __device__ __forceinline__ void next() {
        if (++s == TR_WSTAGES) {
            s = 0;
            ph ^= 1u;
        }
    }
};

// Two FP32 values rounded to bf16, the first in the low half.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}
// x += b for two neighbouring accumulators, one instruction
__device__ __forceinline__ void add2(float& x0, float& x1, float b0, float b1) {
    asm("{\n\t.reg .b64 x, b;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\tadd.rn.f32x2 x, x, b;\n\t"
        "mov.b64 {%0, %1}, x;\n\t}"
        : "+f"(x0), "+f"(x1)
        : "f"(b0), "f"(b1));
}
// max(0, .) of both halves (NaN becomes 0, as fmaxf does)
__device__ __forceinline__ uint32_t relu2(uint32_t w) {
    const __nv_bfloat162 h = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&w), __nv_bfloat162{});
    return *reinterpret_cast<const uint32_t*>(&h);
}
// Bits 15 and 31 of the result: the halves of a non-negative pair that are
// not zero (no carry leaves a half: finite values and infinity are <= 0x7F80).
__device__ __forceinline__ uint32_t nonzero2(uint32_t w) { return (w + 0x7FFF7FFFu) & 0x80008000u; }
// ReLU bits of 32 columns within the trunk: bit j for column 2j, bit 16 + j
// for column 2j + 1, as the shifts above leave them and half_mask takes them:
// of w with the pair's bits at 15 and 31, all ones in the halves that are kept.
__device__ __forceinline__ uint32_t half_mask(uint32_t w) {
    uint32_t m;
    asm("prmt.b32 %0, %1, 0, 0xBB99;" : "=r"(m) : "r"(w));
    return m;
}
// BWD: the data-gradient chain instead of the forward, with no bias: job 0
// from the gradient of the layer after the trunk, then per job dZ_{l-1} =
// (dZ_l W_l) masked by the ReLU bits of H_l.  (A GEMM of its own for job 0
// took 90 us per 524,288 rows, and the chain read its 268 MB back.)  BITS
// (forward): write the layers' ReLU bits, which only a training step needs.
// XKB: K-blocks of the input tile.  HEAD (forward): the linear head (64
// outputs, FP32, no ReLU) as a ninth job.
template <bool BWD, bool BITS, int XKB, bool HEAD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TR_THREADS, 1)
    k_trunk(const __grid_constant__ TrunkMaps maps, TrunkArgs a) {
    constexpr uint32_t IDESC = sm100::idesc_bf16(2 * BM, TR_N, 0, 0);
    constexpr uint32_t IDESC_HEAD = sm100::idesc_bf16(2 * BM, TR_HEAD, 0, 0);
    constexpr int NJ = TR_LAYERS + (HEAD ? 1 : 0);  // jobs per tile
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* act[2] = {smem, smem + TR_ABYTES};
    uint8_t* wbuf = smem + 2 * TR_ABYTES;
    float* s_bias = reinterpret_cast<float*>(wbuf + TR_WSTAGES * TR_WBYTES);
    uint8_t* s_bits = wbuf + TR_WSTAGES * TR_WBYTES + TR_BIAS_BYTES;
    TrCtl* ctl = reinterpret_cast<TrCtl*>(s_bits + 2 * TR_BITS_BYTES);
    static_assert(sizeof(TrCtl) <= 512, "barriers");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = sm100::cluster_rank();
    const uint32_t limit = a.wait_limit ? a.wait_limit : sm100::WAIT_LIMIT;

    if (threadIdx.x == 0) {
        for (int s = 0; s < TR_WSTAGES; ++s) {
            sm100::mbar_init(&ctl->wfull[s], 32);
            sm100::mbar_init(&ctl->wempty[s], 1);
            sm100::mbar_init(&ctl->kready[s], 33);
        }
        for (int p = 0; p < 2; ++p) {
            sm100::mbar_init(&ctl->xfull[p], 1);
            sm100::mbar_init(&ctl->px[p], 1);
            sm100::mbar_init(&ctl->xfree[p], 1);
            sm100::mbar_init(&ctl->mfull[p], 1);
            sm100::mbar_init(&ctl->tfull[p], 1);
            sm100::mbar_init(&ctl->adone[p], TR_EPI_WARPS);
            sm100::mbar_init(&ctl->aready[p], 2 * TR_EPI_WARPS);
            sm100::mbar_init(&ctl->sdone[p], 1);
        }
        sm100::mbar_init(&ctl->drain, 1);
        ctl->abort = 0;
        sm100::fence_mbar_init();
    }
    if (!BWD)
        for (int j = threadIdx.x; j < TR_LAYERS * TR_N + (HEAD ? TR_HEAD : 0); j += TR_THREADS)
            s_bias[j] = __ldg(a.bias[j / TR_N] + j % TR_N);
    if (warp == 1) sm100::tmem_alloc_pair(&ctl->tmem, 2 * TR_N);
    sm100::tc_fence_before();
    __syncthreads();
    sm100::cluster_sync();  // the barriers of both CTAs are set up
    sm100::tc_fence_after();
    const uint32_t tmem = ctl->tmem;
    const int n_tiles = (a.M + 2 * BM - 1) / (2 * BM);
    const int pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
    const int mine = pair < n_tiles ? (n_tiles - 1 - pair) / n_pairs + 1 : 0;
    const int rounds = (mine + 1) / 2;

    if (warp == 0) {
        // ---------------- weight K-blocks, in job order: once per layer and
        // round.  Asynchronous copies by the warp's lanes: the TMA unit is
        // left to the output stores.
        TrStage w;
        bool ok = true;
        const int c = lane & 7, r0 = lane >> 3;  // 16-byte chunk; rows r0, r0 + 4, ...
        for (int r = 0; ok && r < rounds; ++r)
            for (int l = 0; ok && l < NJ; ++l) {
                const int nkb = l == 0 ? XKB : 4;
                const int rows = HEAD && l == TR_LAYERS ? TR_HEAD / 2 : TR_WROWS;
                const uint8_t* src = reinterpret_cast<const uint8_t*>(a.w[l]) +
                                     ((size_t)((int)rank * rows + r0)) * (nkb * 128) + c * 16;
                for (int kb = 0; kb < nkb; ++kb, w.next()) {
                    ok = __all_sync(0xffffffffu, tr_wait(&ctl->wempty[w.s], w.ph ^ 1u, limit, ctl, a.err));
                    if (!ok) break;
                    const uint32_t dst = sm100::smem_addr(wbuf + (size_t)w.s * TR_WBYTES) + r0 * 128;
#pragma unroll 8
                    for (int i = 0; i < rows / 4; ++i)  // row r0 + 4 i
                        sm100::copy_async_16(dst + i * 512 + ((c ^ ((r0 + 4 * i) & 7)) << 4),
                                             src + (size_t)(4 * i) * (nkb * 128) + kb * 128);
                    sm100::copy_async_arrive(rank == 0 ? &ctl->kready[w.s] : &ctl->wfull[w.s]);
                }
            }
        sm100::copy_async_wait_all();  // nothing is in flight when the CTA exits,
#pragma unroll 1
        for (int i = 0; ok && lane == 0 && i < TR_WSTAGES; ++i, w.next())  // nor the last MMAs' arrivals here
            ok = tr_wait(&ctl->wempty[w.s], w.ph ^ 1u, limit, ctl, a.err);
    } else if (warp == 3 && lane == 0) {
        // ---------------- input tiles
        sm100::prefetch_tmap(&maps.x);
        const uint32_t px[2] = {sm100::cluster_addr(&ctl->px[0], 0), sm100::cluster_addr(&ctl->px[1], 0)};
        int xs[2] = {0, 0};
        bool ok = true;
        for (int r = 0; ok && r < rounds; ++r)
            for (int p = 0; ok && p < 2; ++p) {
                const int tile = tr_tile(r, p, n_tiles);
                if (tile < 0) continue;
                // the slot's buffer is free once the last store of its previous tile has read it
                if (xs[p] > 0 && !tr_wait(&ctl->xfree[p], (uint32_t)(xs[p] - 1) & 1u, limit, ctl, a.err)) {
                    ok = false;
                    break;
                }
                sm100::mbar_arrive_expect_tx(&ctl->xfull[p], (uint32_t)(XKB * TR_KBYTES));
                for (int kb = 0; kb < XKB; ++kb)
                    sm100::tma_load_2d(act[p] + (size_t)kb * TR_KBYTES, &maps.x, kb * 64, (2 * tile + (int)rank) * BM,
                                       &ctl->xfull[p]);
                ++xs[p];
                if (rank == 1) {  // tell the CTA that issues the MMAs
                    if (!tr_wait(&ctl->xfull[p], (uint32_t)(xs[p] - 1) & 1u, limit, ctl, a.err)) {
                        ok = false;
                        break;
                    }
                    sm100::mbar_arrive_cluster(px[p]);
                }
            }
        if (!ok)
            for (int p = 0; p < 2; ++p)
                if (xs[p] > 0) sm100::mbar_wait(&ctl->xfull[p], (uint32_t)(xs[p] - 1) & 1u);
    } else if (warp == 1 && lane == 0 && rank == 1) {
        // ---------------- odd CTA: its half of a K-block has landed
        TrStage w;
        bool ok = true;
        for (int r = 0; ok && r < rounds; ++r)
            for (int l = 0; ok && l < NJ; ++l) {
                const int nkb = l == 0 ? XKB : 4;
                for (int kb = 0; kb < nkb; ++kb, w.next()) {
                    if (!tr_wait(&ctl->wfull[w.s], w.ph, limit, ctl, a.err)) {
                        ok = false;
                        break;
                    }
                    sm100::fence_proxy_async();  // the copies, before the tensor core reads them
                    sm100::mbar_arrive_cluster(sm100::cluster_addr(&ctl->kready[w.s], 0));
                }
            }
    } else if (warp == 1 && lane == 0 && rank == 0) {
        // ---------------- even CTA: MMA issuer
        TrStage w;
        int jobs[2] = {0, 0}, xs[2] = {0, 0};
        bool ok = true, issued = false;
        for (int r = 0; ok && r < rounds; ++r) {
            const int slots = tr_tile(r, 1, n_tiles) >= 0 ? 2 : 1;
            for (int l = 0; ok && l < NJ; ++l) {
                const int nkb = l == 0 ? XKB : 4;
                TrStage v = w;
                for (int p = 0; ok && p < slots; ++p) {
                    // the slot's previous job: its output is the input, or (l == 0) the epilogues are done
                    // with its accumulator.  Every phase of aready is waited for, also that of a tile's last
                    // job: a parity wait that skips one returns at once while the skipped one is incomplete.
                    bool in = jobs[p] == 0 ||
                              tr_wait(&ctl->aready[p], (uint32_t)(jobs[p] - 1) & 1u, limit, ctl, a.err);
                    if (in && l == 0) {  // the loaded tile
                        in = tr_wait(&ctl->xfull[p], (uint32_t)xs[p] & 1u, limit, ctl, a.err) &&
                             tr_wait(&ctl->px[p], (uint32_t)xs[p] & 1u, limit, ctl, a.err);
                        ++xs[p];
                    }
                    if (!in) {
                        ok = false;
                        break;
                    }
                    sm100::tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(p * TR_N);
                    v = w;
                    for (int kb = 0; kb < nkb; ++kb, v.next()) {
                        if (p == 0) {
                            if (!tr_wait(&ctl->kready[v.s], v.ph, limit, ctl, a.err)) {
                                ok = false;
                                break;
                            }
                            sm100::fence_proxy_async();
                        }
                        sm100::tc_fence_after();
                        const uint32_t a0 = sm100::smem_addr(act[p] + (size_t)kb * TR_KBYTES);
                        const uint32_t b0 = sm100::smem_addr(wbuf + (size_t)v.s * TR_WBYTES);
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) {
                            const uint64_t adesc = sm100::smem_desc_sw128(a0 + 32 * k, 16, 1024);
                            const uint64_t bdesc = sm100::smem_desc_sw128(b0 + 32 * k, 16, 1024);
                            sm100::mma_bf16_pair(d, adesc, bdesc, HEAD && l == TR_LAYERS ? IDESC_HEAD : IDESC,
                                                 (kb | k) != 0);
                        }
                        issued = true;
                        if (p == slots - 1) sm100::mma_commit_pair(&ctl->wempty[v.s]);
                    }
                    if (!ok) break;
                    sm100::mma_commit_pair(&ctl->tfull[p]);
                    ++jobs[p];
                }
                w = v;
            }
        }
        if (!ok && issued) {  // let issued MMAs finish before TMEM is freed
            sm100::mma_commit_pair(&ctl->drain);
            sm100::mbar_wait(&ctl->drain, 0);
        }
    } else if (warp == 2 && lane == 0) {
        // ---------------- TMA stores of finished activation tiles and their
        // ReLU bits (forward); loads of the mask bits of the slot's next job
        // (backward)
        int jobs[2] = {0, 0}, masks[2] = {0, 0};
        bool ok = true;
        auto load_mask = [&](int r, int l, int p) {
            const int tile = r < rounds ? tr_tile(r, p, n_tiles) : -1;
            if (!BWD || tile < 0) return;
            const int row0 = (2 * tile + (int)rank) * BM;
            ++masks[p];
            if (row0 >= a.M) {
                sm100::mbar_arrive(&ctl->mfull[p]);
                return;
            }
            const uint32_t bytes = (uint32_t)min(BM, a.M - row0) * (TR_N / 8);
            sm100::mbar_arrive_expect_tx(&ctl->mfull[p], bytes);
            sm100::bulk_load(s_bits + p * TR_BITS_BYTES, a.bits[l] + (size_t)row0 * (TR_N / 32), bytes, &ctl->mfull[p]);
        };
        // the head's output: two boxes of the padded rows, or the packed
        // rows as one copy (16 bytes at a time: of a last tile whose rows are
        // not a multiple of four, the last 1 to 3 rows one value at a time)
        auto store_head = [&](int p, int row0) {
            if (BITS || !a.out) {
                for (int c = 0; c < 2; ++c)
                    sm100::tma_store_2d(&maps.raw, c * 32, row0, act[p] + (size_t)c * TR_KBYTES);
            } else {
                const int rows = min(BM, a.M - row0), whole = rows & ~3;
                float* dst = a.out + (size_t)row0 * a.n_out;
                const float* src = reinterpret_cast<const float*>(act[p]);
                if (whole > 0) sm100::bulk_store(dst, src, (uint32_t)(whole * a.n_out * 4));
                for (int i = whole * a.n_out; i < rows * a.n_out; ++i) dst[i] = src[i];
            }
            sm100::bulk_commit();
            sm100::bulk_wait_read_0();
        };
        load_mask(0, 0, 0);
        load_mask(0, 0, 1);
        for (int r = 0; ok && r < rounds; ++r)
            for (int l = 0; ok && l < NJ; ++l)
                for (int p = 0; ok && p < 2; ++p) {
                    const int tile = tr_tile(r, p, n_tiles);
                    if (tile < 0) continue;
                    if (!tr_wait(&ctl->adone[p], (uint32_t)jobs[p] & 1u, limit, ctl, a.err)) {
                        ok = false;
                        break;
                    }
                    load_mask(l + 1 < NJ ? r : r + 1, l + 1 < NJ ? l + 1 : 0, p);
                    const int row0 = (2 * tile + (int)rank) * BM;
                    if (HEAD && l == TR_LAYERS) {
                        if (row0 < a.M) store_head(p, row0);
                        sm100::mbar_arrive(&ctl->sdone[p]);
                        sm100::mbar_arrive(&ctl->xfree[p]);
                        ++jobs[p];
                        continue;
                    }
                    constexpr bool bits = !BWD && BITS;
                    if ((((a.store >> l) & 1u) || bits) && row0 < a.M) {
                        if ((a.store >> l) & 1u)
                            for (int kb = 0; kb < 4; ++kb)
                                sm100::tma_store_2d(&maps.h[l], kb * 64, row0, act[p] + (size_t)kb * TR_KBYTES);
                        if (bits)
                            sm100::bulk_store(a.bits[l] + (size_t)row0 * (TR_N / 32), s_bits + p * TR_BITS_BYTES,
                                              (uint32_t)min(BM, a.M - row0) * (TR_N / 8));
                        sm100::bulk_commit();
                        sm100::bulk_wait_read_0();
                    }
                    sm100::mbar_arrive(&ctl->sdone[p]);
                    if (l == NJ - 1) sm100::mbar_arrive(&ctl->xfree[p]);
                    ++jobs[p];
                }
        if (!ok)  // drain the mask loads still in flight
            for (int p = 0; p < 2; ++p)
                if (masks[p] > 0) sm100::mbar_wait(&ctl->mfull[p], (uint32_t)(masks[p] - 1) & 1u);
        sm100::bulk_wait_all();  // the stores are complete before the CTA exits
    } else if (warp >= TR_EPI_WARP0) {
        // ---------------- epilogue: bias + ReLU -> bf16 into the slot's buffer, ReLU bits
        const int q = warp & 3;
        const int grp = (warp - TR_EPI_WARP0) >> 2;
        const int rl = q * 32 + lane;  // row within the CTA's half of the tile
        const uint32_t ready[2] = {sm100::cluster_addr(&ctl->aready[0], 0), sm100::cluster_addr(&ctl->aready[1], 0)};
        int jobs[2] = {0, 0};
        bool ok = true;
        for (int r = 0; ok && r < rounds; ++r)
            for (int l = 0; ok && l < NJ; ++l)
                for (int p = 0; ok && p < 2; ++p) {
                    const int tile = tr_tile(r, p, n_tiles);
                    if (tile < 0) continue;
                    if (!tr_wait(&ctl->tfull[p], (uint32_t)jobs[p] & 1u, limit, ctl, a.err) ||
                        (BWD && !tr_wait(&ctl->mfull[p], (uint32_t)jobs[p] & 1u, limit, ctl, a.err)) ||
                        (l > 0 && !tr_wait(&ctl->sdone[p], (uint32_t)(jobs[p] - 1) & 1u, limit, ctl, a.err))) {
                        ok = false;
                        break;
                    }
                    if (HEAD && l == TR_LAYERS) {
                        sm100::tc_fence_after();
                        constexpr int HC = TR_HEAD / TR_EPI_GROUPS;  // columns per epilogue warp
                        static_assert(HC == 16, "tmem_ld16");
                        float v[HC];
                        sm100::tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(p * TR_N + grp * HC), v);
                        const float4* b4 = reinterpret_cast<const float4*>(s_bias + TR_LAYERS * TR_N + grp * HC);
#pragma unroll
                        for (int j = 0; j < HC / 4; ++j) {
                            const float4 b = b4[j];
                            v[4 * j] += b.x;
                            v[4 * j + 1] += b.y;
                            v[4 * j + 2] += b.z;
                            v[4 * j + 3] += b.w;
                        }
                        if (!BITS && a.out) {
                            float* row = reinterpret_cast<float*>(act[p]) + rl * a.n_out + grp * HC;
#pragma unroll
                            for (int j = 0; j < HC; ++j)
                                if (grp * HC + j < a.n_out) row[j] = v[j];
                        } else {
                            uint8_t* row = act[p] + (size_t)(grp >> 1) * TR_KBYTES + (size_t)rl * 128;
#pragma unroll
                            for (int u = 0; u < HC / 4; ++u)
                                *reinterpret_cast<float4*>(row + ((((grp & 1) * 4 + u) ^ (rl & 7)) << 4)) =
                                    make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
                        }
                        sm100::fence_proxy_async();
                        sm100::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) {
                            sm100::mbar_arrive(&ctl->adone[p]);
                            sm100::mbar_arrive_cluster(ready[p]);
                        }
                        ++jobs[p];
                        continue;
                    }
                    uint2* bits = reinterpret_cast<uint2*>(s_bits + p * TR_BITS_BYTES + rl * (TR_N / 8)) + grp;
                    const uint2 mask = BWD ? *bits : make_uint2(0u, 0u);
                    sm100::tc_fence_after();
                    uint8_t* A = act[p];
                    uint32_t pos0 = 0u;
#pragma unroll 1
                    for (int h = 0; h < TR_CHUNKS; ++h) {
                        const int c = grp * TR_CHUNKS + h;
                        float v[32];
                        sm100::tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(p * TR_N + c * 32), v);
                        uint32_t packed[16];
                        if (BWD) {  // keep the gradient where the forward pre-activation was > 0
                            const uint32_t mw = h == 0 ? mask.x : mask.y;
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                packed[j] = pack_bf16(v[2 * j], v[2 * j + 1]) & half_mask(mw << (15 - j));
                        } else {
                            const float4* b4 = reinterpret_cast<const float4*>(s_bias + l * TR_N + c * 32);
                            uint32_t pos = 0u;
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const float4 b = b4[j];
                                float x0 = v[4 * j], x1 = v[4 * j + 1], x2 = v[4 * j + 2], x3 = v[4 * j + 3];
                                add2(x0, x1, b.x, b.y);
                                add2(x2, x3, b.z, b.w);
                                packed[2 * j] = relu2(pack_bf16(x0, x1));
                                packed[2 * j + 1] = relu2(pack_bf16(x2, x3));
                                if (BITS) {
                                    pos = (pos >> 1) | nonzero2(packed[2 * j]);
                                    pos = (pos >> 1) | nonzero2(packed[2 * j + 1]);
                                }
                            }
                            if (BITS) {
                                if (h == 0) pos0 = pos;
                                else *bits = make_uint2(pos0, pos);
                            }
                        }
                        uint8_t* blk = A + (size_t)(c >> 1) * TR_KBYTES + (size_t)rl * 128;
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int ch = (c & 1) * 4 + u;
                            *reinterpret_cast<uint4*>(blk + ((ch ^ (rl & 7)) << 4)) =
                                make_uint4(packed[4 * u], packed[4 * u + 1], packed[4 * u + 2], packed[4 * u + 3]);
                        }
                    }
                    sm100::fence_proxy_async();
                    sm100::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        sm100::mbar_arrive(&ctl->adone[p]);
                        sm100::mbar_arrive_cluster(ready[p]);
                    }
                    ++jobs[p];
                }
    }
    sm100::tc_fence_before();
    __syncthreads();
    sm100::cluster_sync();  // neither CTA's memory is read or signalled any more
    if (warp == 1) {
        sm100::tc_fence_after();
        sm100::tmem_dealloc_pair(tmem, 2 * TR_N);
    }
}

}  // namespace gemm
}  // namespace plo
