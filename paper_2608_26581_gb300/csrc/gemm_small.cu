// gemm_small.cu -- RFQ GEMM for few rows of X, or few output columns (Algorithm 1,
// Eq. rfq):
//   Y = X~ W~ + phi X^ W~
// with the operands swapped and the reduction split over a cluster: a CTA's
// MMA takes 128 W~ rows (output columns) as its M side and a tile of T rows
// of X (a multiple of 16, at most 128) as its N side, so few rows of X cost
// few MMA cycles and few loads instead of a padded 128-row tile; and the CTAs
// of a cluster of CS share one output tile, each multiplying its share of the
// k-stages, so that a layer with few output tiles still reads W~ with the
// whole chip.  The partial accumulators meet in shared memory: every CTA
// writes its own, and after a cluster barrier each CTA sums its share of the
// tile over the cluster's CTAs in rank order (distributed shared memory) and
// stores it.  No workspace, and the same Y on every run.
//
// Operands (template F4): MXFP4 codes with MMA-layout scales (kind::mxf4, a
// k-stage is 256 elements), or exact bf16 expansions (HiF4, kind::f16, 64
// elements); 128-byte rows either way.  FUSED: X is bf16 and converter warps
// quantize the tile's rows (main and residual, as the activation quantizer)
// straight into the swizzled operand tiles and the scale atoms.
//
// Per CTA (352 threads, 608 with FUSED):
//   warp 0      TMA producer: WT boxes of 128 W~ rows, the T-row boxes of X~
//               and X^, and the scale atoms (bulk copies)
//   warp 1      MMA issuer: per K step and 128-row W~ block the main and the
//               residual MMA into one accumulator of T columns
//   warps 2-9   scale writers (shared memory -> TMEM, one warp per lane
//               quarter, two sets taking the stages in turn), then the
//               epilogue of their lane quarter
//   warp 10     scale-atom producer
//   warps 11-18 (FUSED) converters
// A stage's scale slot in TMEM has the stage's index in the ring: the slot is
// rewritten only after the stage's copies, which were issued once the MMAs
// that read the slot had completed.
//
// Selective phi is not looked at here: the stored residual of a phi = 0 tile
// is zero, so including it adds exact zeros.  The choice of the kernel counts
// with a tiled kernel that skips it (choose()).
//
// Shared memory is requested in proportion to the TMEM columns (a CTA with
// all 512 columns takes a whole SM's shared memory, 256 columns half of it),
// so CTAs that fit on an SM together never wait for each other's TMEM.
//
// Every mbarrier wait is bounded (kWaitLimitNs, or the limit in the caller's
// workspace) and also gives up as soon as any CTA has recorded a timeout in
// the caller's status word.  A CTA that gave up waits (bounded) for its copies
// and MMAs in flight, whichever of its roles gave up and when, still meets its
// cluster at both barriers, and no CTA of its cluster stores anything.
#include <cuda_bf16.h>
#include <cmath>
#include <cstdint>

#include "internal.h"
#include "mxfp4_math.cuh"
#include "ptx.cuh"

namespace rfq {
namespace {
RFQ_DEBUG_WORD_DECL

constexpr int WROWS = 128;               // W~ rows per MMA
constexpr int ROW = 128;                 // operand bytes per row per stage
constexpr int W_BYTES = WROWS * ROW;
constexpr int ATOM = 512;                // scale bytes of 128 rows x one 128-element chunk
constexpr int MAX_STAGES = 8;
constexpr int SLOT_COLS = 32;            // W~ block w, chunk c at 8w + 4c; then X~ at 4c, then X^
                                         // (SWAP: X~ at 4c, X^ at 8 + 4c, W~ at 16 + 8c)
constexpr int SF_WARPS = 4;              // one per TMEM lane quarter
constexpr int SF_SETS = 2;               // sets of them, taking the ring's slots in turn
constexpr int SFP_WARP = 2 + SF_SETS * SF_WARPS;  // scale-atom producer
constexpr int CONV_WARP0 = SFP_WARP + 1;
constexpr int CONV_WARPS = 8;
constexpr int MAX_CLUSTER = 8;           // (the portable limit)

template <int V>
struct Int {
    static constexpr int value = V;
};

__device__ __forceinline__ bool wait_for(uint64_t *bar, uint32_t parity, uint64_t limit_ns,
                                         const volatile int32_t *abort_word = nullptr)
{
    return mbar_wait<false, true>(bar, parity, limit_ns, abort_word);
}

struct Ctl {
    uint64_t full[MAX_STAGES];           // the stage's operand tiles landed
    uint64_t sf_full[MAX_STAGES];        // its scale atoms landed
    uint64_t empty[MAX_STAGES];          // its MMAs completed
    uint64_t sf_ready[MAX_STAGES];       // its scale words are in TMEM
    uint64_t conv[MAX_STAGES];           // FUSED: its rows of X are quantized
    uint64_t acc_full;
    uint64_t drain;
    uint64_t wait_ns;
    uint32_t tmem_base;
    int32_t abort_flag;
    int32_t hold;                        // the workspace asks for a held start
    int32_t issued, sf_issued;           // stages whose copies each producer issued (valid once its role ends)
};
constexpr size_t kCtlBytes = (sizeof(Ctl) + 1023) / 1024 * 1024;

// Position in the ring of stages and the parity of its current round.
struct Ring {
    int slot = 0, stages;
    uint32_t phase = 0;
    __device__ explicit Ring(int n) : stages(n) {}
    __device__ void next()
    {
        if (++slot == stages) {
            slot = 0;
            phase ^= 1;
        }
    }
};

// Launch shape, computed on the host.
struct Shape {
    int M, N, K;
    int T;              // rows of X per tile (multiple of 16)
    int NT;             // output columns (W~ rows) per tile: 128 WT, or with SWAP a multiple of 16
    int w_atoms;        // 128-row scale atoms a tile's W~ rows can span
    int stages;         // ring depth
    int stage_bytes;
    int x_off, r_off, sf_off;   // byte offsets of X~, X^ and the scale atoms in a stage
    int x_atoms;        // 128-row scale atoms a tile's rows of X can span (1 or 2)
    int tmem_cols, acc_cols;    // allocated columns; columns between the accumulators of two W~ blocks
    int sf_col0;                // first scale slot's column
    int prefetch;               // k-stages of W~ prefetched into L2 at the start
    int res, cat, out_bf16;
};

__device__ __forceinline__ void flag_timeout(Ctl &S, int32_t *status)
{
    S.abort_flag = 1;
    atomicExch(status, kDevTimeout);
}

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t caddr)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(caddr)
                 : "memory");
    return v;
}

template <bool F4, bool FUSED, int WT, bool SWAP>
__global__ void __launch_bounds__(FUSED ? 32 * (CONV_WARP0 + CONV_WARPS) : 32 * CONV_WARP0, FUSED ? 1 : 2)
    gemm_small_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                      const __grid_constant__ CUtensorMap tmR, const uint8_t *__restrict__ sfw,
                      const uint8_t *__restrict__ sfx, const uint8_t *__restrict__ sfr,
                      const uint4 *__restrict__ xbf, void *__restrict__ y, int32_t *status,
                      const __grid_constant__ Shape sh)
{
    static_assert(!FUSED || F4, "the fused quantizer writes MXFP4 operands");
    static_assert(!SWAP || (WT == 2 && !FUSED), "X on the M side: 128 rows of X by 256 W~ rows");
    constexpr int PS = SWAP ? WT * WROWS + 4 : WT * WROWS;   // floats per row of the partial tile
    constexpr int KS = F4 ? 256 : 64;    // elements per stage
    constexpr int W_COLS = SWAP ? 16 : 8 * WT;   // scale columns before X~'s (SWAP: before W~'s)
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Ctl &S = *reinterpret_cast<Ctl *>(base);
    uint8_t *ring = base + kCtlBytes;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const volatile int32_t *gstat = status;
    const int T = sh.T, ST = sh.stages;
    const bool res = sh.res != 0;
    // cat (up to 64 rows of X): X~ and X^, side by side in the stage, are the
    // N side of one MMA, their products in separate columns until the epilogue
    // adds them; otherwise two MMAs add into the same columns
    const bool cat = sh.cat != 0, sep = res && !cat;
    const int NB = cat ? 2 * T : T;

    uint32_t rank, CS;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(CS));
    const int tile = blockIdx.x / CS;
    const int n0 = tile * sh.NT;                 // first output column (W~ row)
    const int t0 = blockIdx.y * T;                      // first row of X
    const int nw = WT > 1 && n0 + WROWS < sh.N ? WT : 1;
    const int kc = sh.K >> 7;                           // 128-element chunks (F4: scale atoms along K)
    const int nks = (sh.K + KS - 1) / KS;
    const int k_lo = (int)((int64_t)nks * rank / CS);   // this CTA's k-stages
    const int n_st = (int)((int64_t)nks * (rank + 1) / CS) - k_lo;

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&S.full[s], 1);
            mbar_init(&S.sf_full[s], 1);
            mbar_init(&S.empty[s], 1);
            mbar_init(&S.sf_ready[s], SF_WARPS);
            mbar_init(&S.conv[s], FUSED ? T / 4 : 1);
        }
        mbar_init(&S.acc_full, 1);
        mbar_init(&S.drain, 1);
        S.issued = S.sf_issued = 0;
        fence_mbar_init();
    }
    if (threadIdx.x == 32 * SFP_WARP) {
        // the workspace's words in one load (they are read before anything is
        // copied: one trip to L2 instead of three)
        grid_dependency_wait();
        const int4 w = __ldcv(reinterpret_cast<const int4 *>(status));
        S.abort_flag = w.x;              // a bounded wait of an earlier CTA or call gave up: compute nothing
        S.wait_ns = w.y > 0 ? (uint64_t)w.y * 1000ull : kWaitLimitNs;
        S.hold = w.z;
    }
    if (warp == 0) {
        // Before the kernel ahead of this one has ended (see the launch), W~
        // starts on its way from HBM to L2: the first PREFETCH stages' tiles, a
        // hint that is right whatever that kernel writes.
        if (elect_one())
            for (int p = 0; p < min(n_st, sh.prefetch); ++p) {
                tma_prefetch_2d(&tmW, (k_lo + p) * ROW, n0);
                if (!SWAP && WT > 1 && nw > 1)
                    tma_prefetch_2d(&tmW, (k_lo + p) * ROW, n0 + WROWS);
            }
    }
    if (warp == 2 && lane == 0) {
        prefetch_tmap(&tmW);
        if (!FUSED) {
            prefetch_tmap(&tmX);
            if (res)
                prefetch_tmap(&tmR);
        }
    }
    if (warp == 1) {
        tmem_alloc(&S.tmem_base, (uint32_t)sh.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    const uint64_t wl = S.wait_ns;
    const bool skip = S.abort_flag != 0;
    const int sf0 = sh.sf_col0;
    __syncthreads();                                    // (abort_flag is read above before any role sets it)

    auto chunks_of = [&](int ks) { return F4 ? min(2, kc - 2 * ks) : 1; };

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (!skip) {
            // (the whole warp follows the loop and one elected lane issues: see elect_one)
            bool stop = false;
            int p = 0;
            if (S.hold != 0 && !__all_sync(0xffffffffu, held_start_wait(status, wl))) { // never opened
                if (lane == 0)
                    flag_timeout(S, status);
                stop = true;
            }
            const uint32_t op_bytes = (uint32_t)((SWAP ? sh.NT * ROW : nw * W_BYTES) + (FUSED ? 0 : (res ? 2 : 1) * T * ROW));
            Ring at(ST);
            for (; p < n_st && !stop; ++p, at.next()) {
                const int slot = at.slot;
                if (!__all_sync(0xffffffffu, wait_for(&S.empty[slot], at.phase ^ 1, wl, gstat))) {
                    if (lane == 0)
                        flag_timeout(S, status);
                    stop = true;
                    break;
                }
                if (elect_one()) {
                    uint8_t *st = ring + slot * sh.stage_bytes;
                    uint64_t *bar = &S.full[slot];
                    const int kx = (k_lo + p) * ROW;
                    mbar_arrive_expect_tx(bar, op_bytes);
                    tma_load_2d(st, &tmW, bar, kx, n0);
                    if (!SWAP && WT > 1 && nw > 1)
                        tma_load_2d(st + W_BYTES, &tmW, bar, kx, n0 + WROWS);
                    if (!FUSED) {
                        tma_load_2d(st + sh.x_off, &tmX, bar, kx, t0);
                        if (res)
                            tma_load_2d(st + sh.r_off, &tmR, bar, kx, t0);
                    }
                }
            }
            if (lane == 0)
                S.issued = p;
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (!skip) {
            bool stop = false;
            const int nb = SWAP ? sh.NT : NB;      // N side of the MMAs
            const uint32_t idn = F4 ? idesc_mxf4(WROWS, nb, 0, 0) : idesc_bf16(WROWS, nb);
            const uint32_t ring0 = smem_u32(ring), stage16 = (uint32_t)sh.stage_bytes >> 4;
            const uint64_t wd0 = sdesc_k_sw128(ring0), xd0 = sdesc_k_sw128(ring0 + sh.x_off),
                           rd0 = sdesc_k_sw128(ring0 + sh.r_off);
            Ring at(ST);
            for (int p = 0; p < n_st; ++p, at.next()) {
                const int slot = at.slot;
                const uint32_t par = at.phase;
                // F4: sf_ready stands for the operands too (and FUSED: the converted
                // rows), except with SWAP (see the scale writers)
                if (!__all_sync(0xffffffffu, (!(F4 && SWAP) || wait_for(&S.full[slot], par, wl, gstat)) &&
                                                 wait_for(F4 ? &S.sf_ready[slot] : &S.full[slot], par, wl, gstat))) {
                    if (lane == 0)
                        flag_timeout(S, status);
                    stop = true;
                    break;
                }
                tc_fence_after();
                if (elect_one()) {
                    // descriptors of the stage: slot 0's plus its offset in 16-byte units
                    const uint32_t so = (uint32_t)slot * stage16;
                    const uint64_t wd = wd0 + so, xd = xd0 + so, rd = rd0 + so;
                    const uint32_t sf = tmem + sf0 + SLOT_COLS * slot;
                    const uint32_t first = p == 0 ? 0u : 1u;
                    auto step = [&](int j) {
                        const int c = j >> 1;
                        const uint32_t id = F4 ? idn + ((uint32_t)(2 * (j & 1)) << 4) + ((uint32_t)(2 * (j & 1)) << 29)
                                               : idn;
                        const uint32_t acc_in = j == 0 ? first : 1u;
                        if constexpr (SWAP) {
                            if (F4) {
                                tc_mma_mxf4(tmem, xd + 2 * j, wd + 2 * j, id, sf + 4 * c, sf + 16 + 8 * c, acc_in);
                                if (res)
                                    tc_mma_mxf4(tmem, rd + 2 * j, wd + 2 * j, id, sf + 8 + 4 * c, sf + 16 + 8 * c, 1);
                            } else {
                                tc_mma_f16(tmem, xd + 2 * j, wd + 2 * j, id, acc_in);
                                if (res)
                                    tc_mma_f16(tmem, rd + 2 * j, wd + 2 * j, id, 1);
                            }
                        } else {
#pragma unroll
                            for (int w = 0; w < WT; ++w) {
                                if (w >= nw)
                                    break;
                                const uint64_t wj = wd + (W_BYTES >> 4) * w + 2 * j;
                                const uint32_t acc = tmem + w * sh.acc_cols;
                                if (F4) {
                                    tc_mma_mxf4(acc, wj, xd + 2 * j, id, sf + 8 * w + 4 * c, sf + W_COLS + 4 * c,
                                                acc_in);
                                    if (sep)
                                        tc_mma_mxf4(acc, wj, rd + 2 * j, id, sf + 8 * w + 4 * c,
                                                    sf + W_COLS + 8 + 4 * c, 1);
                                } else {
                                    tc_mma_f16(acc, wj, xd + 2 * j, id, acc_in);
                                    if (sep)
                                        tc_mma_f16(acc, wj, rd + 2 * j, id, 1);
                                }
                            }
                        }
                    };
                    step(0);
                    step(1);
                    if (!F4 || 2 * (k_lo + p) + 1 < kc) {   // (the odd last chunk has two steps)
                        step(2);
                        step(3);
                    }
                    tc_commit(&S.empty[slot]);
                }
            }
            if (!stop && elect_one())
                tc_commit(&S.acc_full);
        }
    } else if (warp < SFP_WARP) {
        // ------------------------------------------------ scale writers, then the epilogue
        const int q = warp & 3;          // TMEM lane quarter this warp may access
        const int set = (warp - 2) >> 2;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
        bool stop = skip;
        if (F4) {
            const int rbase = t0 & 127;  // the tile's first row inside its scale atom
            Ring at(ST);
            for (int p = 0; p < n_st && !stop; ++p, at.next()) {
                // a set owns its slots: waiting for every phase of a barrier, it
                // cannot take an older phase of the same parity for the awaited one
                if ((at.slot & 1) != set)
                    continue;
                const int slot = at.slot;
                const uint32_t par = at.phase;
                // warp-uniform outcome: the tcgen05 stores below need the whole warp
                if (!__all_sync(0xffffffffu, wait_for(&S.sf_full[slot], par, wl, gstat) &&
                                                 (!FUSED || wait_for(&S.conv[slot], par, wl, gstat)))) {
                    if (lane == 0)
                        flag_timeout(S, status);
                    stop = true;
                    break;
                }
                tc_fence_after();
                const uint8_t *sw = ring + slot * sh.stage_bytes + sh.sf_off;
                const uint8_t *sx = sw + sh.w_atoms * 2 * ATOM, *sr = sx + sh.x_atoms * 2 * ATOM;
                const uint32_t tb = tq + sf0 + SLOT_COLS * slot;
                // word of 128-row scale atoms from p0: chunk c's four scales of row `row`
                // past their start (both chunks of the stage are moved, also
                // where the last stage holds one: the other's words are unused)
                auto word = [&](const uint8_t *p0, int c, int row) {
                    return *reinterpret_cast<const uint32_t *>(p0 + (row >> 7) * 2 * ATOM + c * ATOM + (row & 31) * 16 +
                                                               ((row >> 5) & 3) * 4);
                };
                auto row4 = [&](uint32_t *v, const uint8_t *p0) {   // rows 32 j + lane, j = 0..3, of one atom
                    const uint4 t = *reinterpret_cast<const uint4 *>(p0 + lane * 16);
                    v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
                };
                const int x_last = sh.x_atoms * 128 - 1;
                uint32_t v[32];
                if constexpr (SWAP) {
                    const int wbase = (n0 & 127) + lane, w_last = sh.w_atoms * 128 - 1;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        if (rbase == 0) {
                            row4(v + 4 * c, sx + c * ATOM);
                            if (res)
                                row4(v + 8 + 4 * c, sr + c * ATOM);
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int r = min(rbase + lane + 32 * j, x_last);
                                v[4 * c + j] = word(sx, c, r);
                                v[8 + 4 * c + j] = res ? word(sr, c, r) : 0u;
                            }
                        }
                        if ((sh.NT & 127) == 0) {
                            row4(v + 16 + 8 * c, sw + c * ATOM);
                            if (sh.w_atoms > 1)
                                row4(v + 20 + 8 * c, sw + (2 + c) * ATOM);
                        } else {
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                v[16 + 8 * c + j] = 32 * j < sh.NT ? word(sw, c, min(wbase + 32 * j, w_last)) : 0u;
                        }
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
#pragma unroll
                        for (int w = 0; w < WT; ++w)
                            row4(v + 8 * w + 4 * c, sw + (2 * w + c) * ATOM);   // (past N: unused)
                        uint32_t *vx = v + W_COLS + 4 * c, *vr = v + W_COLS + 8 + 4 * c;
                        if (cat) {
                            // the N side's rows: the tile's rows of X~, then of X^
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int r = 32 * j + lane;
                                vx[j] = 32 * j < NB ? word(r < T ? sx : sr, c, r < T ? r : min(r - T, T - 1)) : 0u;
                            }
                        } else if (rbase == 0) {
                            row4(vx, sx + c * ATOM);
                            if (sep)
                                row4(vr, sr + c * ATOM);
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int r = min(rbase + lane + 32 * j, x_last);
                                vx[j] = word(sx, c, r);
                                if (sep)
                                    vr[j] = word(sr, c, r);
                            }
                        }
                    }
                }
                if (WT == 1 && !sep)
                    tmem_st_32x32b_x16(tb, v);
                else
                    tmem_st_32x32b_x32(tb, v);
                // narrow tiles: the MMA thread's own work per stage is the bottleneck, so
                // the operand tiles' barrier is waited for here; wide ones (SWAP, three
                // stages in flight) wait for the two in parallel
                const bool landed = SWAP || __all_sync(0xffffffffu, wait_for(&S.full[slot], par, wl, gstat));
                tmem_st_wait();
                if (!landed) {
                    if (lane == 0)
                        flag_timeout(S, status);
                    stop = true;
                    break;
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(&S.sf_ready[slot]);
            }
        }
        if (!stop && !__all_sync(0xffffffffu, wait_for(&S.acc_full, 0, wl, gstat))) {
            if (lane == 0)
                flag_timeout(S, status);
            stop = true;
        }
        if (!stop) {
            // the partial tile as [row of X][output column] fp32 over the ring
            // (every copy has landed and every MMA has completed)
            tc_fence_after();
            float *part = reinterpret_cast<float *>(ring);
            if constexpr (SWAP) {
                // lane = row of X: four output columns per store, rows 16
                // bytes apart in the banks (stride PS)
                float *row = part + (q * 32 + lane) * PS;
                for (int c = 32 * set; c < sh.NT; c += 32 * SF_SETS) {   // (past NT: unused columns of the row)
                    uint32_t v[32];
                    tmem_ld_32x32b_x32(tq + c, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; i += 4)
                        *reinterpret_cast<uint4 *>(row + c + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                }
            } else
#pragma unroll
            for (int w = 0; w < WT; ++w) {
                if (w >= nw)
                    break;
                for (int c = 32 * set; c < T; c += 32 * SF_SETS) {
                    uint32_t v[32], r[32];
                    tmem_ld_32x32b_x32(tq + w * sh.acc_cols + c, v);
                    if (cat)
                        tmem_ld_32x32b_x32(tq + w * sh.acc_cols + T + c, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (i < 16 || c + 16 < T)
                            part[(c + i) * PS + w * WROWS + q * 32 + lane] =
                                cat ? __uint_as_float(v[i]) + __uint_as_float(r[i]) : __uint_as_float(v[i]);
                }
            }
        }
    } else if (F4 && warp == SFP_WARP) {
        // ------------------------------------------------ scale producer
        // (a warp of its own: one bulk copy takes its issuing lane about a
        // hundred cycles, and the operand copies of the next stage would wait)
        if (!skip) {
            bool stop = S.hold != 0 && !__all_sync(0xffffffffu, held_start_wait(status, wl));
            int p = 0;
            const int m_atom = t0 >> 7;
            const int xa = FUSED ? 0 : min(sh.x_atoms, ((sh.M + 127) >> 7) - m_atom);
            const int wa = min(sh.w_atoms, ((sh.N + 127) >> 7) - (n0 >> 7));
            const uint32_t n_at = (uint32_t)(wa + xa * (res ? 2 : 1));
            // the first stage's atoms; a stage's two atoms of a row band are contiguous
            const int64_t band = (int64_t)kc * ATOM;
            const uint8_t *gw = sfw + (n0 >> 7) * band + (int64_t)k_lo * 2 * ATOM;
            const uint8_t *gx = FUSED ? nullptr : sfx + m_atom * band + (int64_t)k_lo * 2 * ATOM;
            const uint8_t *gr = FUSED || !res ? nullptr : sfr + m_atom * band + (int64_t)k_lo * 2 * ATOM;
            Ring at(ST);
            for (; p < n_st && !stop; ++p, at.next()) {
                const int slot = at.slot;
                if (!__all_sync(0xffffffffu, wait_for(&S.empty[slot], at.phase ^ 1, wl, gstat))) {
                    stop = true;
                    break;
                }
                if (elect_one()) {
                    const uint32_t bytes = (uint32_t)chunks_of(k_lo + p) * ATOM;
                    uint64_t *bar = &S.sf_full[slot];
                    uint8_t *sw = ring + slot * sh.stage_bytes + sh.sf_off;
                    uint8_t *sx = sw + sh.w_atoms * 2 * ATOM, *sr = sx + sh.x_atoms * 2 * ATOM;
                    mbar_arrive_expect_tx(bar, n_at * bytes);
                    bulk_load(sw, gw, bytes, bar);
                    if (WT > 1 && wa > 1)
                        bulk_load(sw + 2 * ATOM, gw + band, bytes, bar);
                    if (SWAP && wa > 2)
                        bulk_load(sw + 4 * ATOM, gw + 2 * band, bytes, bar);
                    if (!FUSED) {
                        bulk_load(sx, gx, bytes, bar);
                        if (res)
                            bulk_load(sr, gr, bytes, bar);
                        if (xa > 1) {
                            bulk_load(sx + 2 * ATOM, gx + band, bytes, bar);
                            if (res)
                                bulk_load(sr + 2 * ATOM, gr + band, bytes, bar);
                        }
                    }
                }
                gw += 2 * ATOM;
                gx += 2 * ATOM;
                gr += 2 * ATOM;
            }
            if (stop && lane == 0)
                flag_timeout(S, status);
            if (lane == 0)
                S.sf_issued = p;
        }
    } else if constexpr (FUSED) {
        // ------------------------------------------------ converters
        // A step quantizes 4 rows x one k-stage, one 32-element block per lane
        // (row lane / 8 of the step, block lane % 8); a stage has T / 4 steps,
        // dealt to the warps in order over all stages.  The next step's loads
        // are issued before this one waits for its stage's buffers.
        // A warp's place, stage and step in it, is counted on (128 x 4096 x 24576
        // without a residual: 56.0 us; dividing by steps and the ring's length 59.8).
        const int steps = T / 4;
        const int kb = sh.K >> 5;
        struct Place {
            int p, i;                    // k-stage, step
        };
        auto forth = [&](Place &at) {
            for (at.i += CONV_WARPS; at.i >= steps; at.i -= steps)
                ++at.p;
        };
        auto load = [&](const Place &at, uint32_t (&w)[16]) {
            const int m = at.i * 4 + (lane >> 3), b = (k_lo + at.p) * 8 + (lane & 7);
            if (at.p < n_st && m < sh.M && b < kb) {
                const uint4 *px = xbf + (int64_t)m * (sh.K >> 3) + (int64_t)b * 4;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 t = __ldg(px + i);
                    w[4 * i] = t.x;
                    w[4 * i + 1] = t.y;
                    w[4 * i + 2] = t.z;
                    w[4 * i + 3] = t.w;
                }
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    w[i] = 0;
            }
        };
        uint32_t cur[16], nxt[16];
        Place now = {0, warp - CONV_WARP0 - CONV_WARPS}, ahead;
        forth(now);
        load(now, cur);
        int slot = 0, slot_p = 0;        // ring slot of stage slot_p, and its phase
        uint32_t phase = 0;
        for (; now.p < n_st && !skip; now = ahead) {
            ahead = now;
            forth(ahead);
            load(ahead, nxt);
            for (; slot_p < now.p; ++slot_p)
                if (++slot == ST) {
                    slot = 0;
                    phase ^= 1;
                }
            if (!__all_sync(0xffffffffu, wait_for(&S.empty[slot], phase ^ 1, wl, gstat))) {
                if (lane == 0)
                    flag_timeout(S, status);
                break;
            }
            float xf[32];
            bf16x32_to_f32(cur, xf);
            const int r = now.i * 4 + (lane >> 3), b = lane & 7;
            uint8_t *st = ring + slot * sh.stage_bytes;
            uint8_t *sx = st + sh.sf_off + sh.w_atoms * 2 * ATOM, *sr = sx + 2 * ATOM;
            const int co = r * ROW + ((b ^ (r & 7)) << 4);   // 128-byte swizzle
            const int so = (b >> 2) * ATOM + (r & 31) * 16 + ((r >> 5) & 3) * 4 + (b & 3);
            if (res) {
                const Mx32 qz = mxfp4_quant32<true>(xf);
                *reinterpret_cast<uint4 *>(st + sh.x_off + co) = qz.code;
                *reinterpret_cast<uint4 *>(st + sh.r_off + co) = qz.rcode;
                sx[so] = (uint8_t)qz.sb;
                sr[so] = (uint8_t)qz.rb;
            } else {
                const Mx32 qz = mxfp4_quant32<false>(xf);
                *reinterpret_cast<uint4 *>(st + sh.x_off + co) = qz.code;
                sx[so] = (uint8_t)qz.sb;
            }
            // codes are read by the tensor core (async proxy), scales by the writers
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&S.conv[slot]);
#pragma unroll
            for (int i = 0; i < 16; ++i)
                cur[i] = nxt[i];
        }
    }

    // ---------------------------------------------------- cluster reduction
    tc_fence_before();
    __syncthreads();
    if (S.abort_flag != 0 && !skip) {
        // A role gave up, perhaps after the producers or the MMA issuer had
        // ended theirs: what they have in flight still writes this CTA's shared
        // and tensor memory, which its next owner gets when the CTA ends.
        if (warp == 0 && lane == 0)
            for (int q = max(0, S.issued - ST); q < S.issued; ++q)
                (void)wait_for(&S.full[q % ST], (q / ST) & 1, wl);
        if (warp == SFP_WARP && lane == 0)
            for (int q = max(0, S.sf_issued - ST); q < S.sf_issued; ++q)
                (void)wait_for(&S.sf_full[q % ST], (q / ST) & 1, wl);
        if (warp == 1 && elect_one()) {  // (the lane that issued the MMAs: the election is the same each time)
            tc_commit(&S.drain);
            (void)wait_for(&S.drain, 0, wl);
        }
        __syncthreads();
    }
    if (CS > 1)
        cluster_sync();                  // every CTA's partial tile is in its shared memory
    bool ok = true;
    for (uint32_t j = 0; j < CS; ++j)
        ok = ok && ld_cluster_s32(mapa_shared(smem_u32(&S.abort_flag), j)) == 0;
    if (ok) {
        // groups of 4 output columns; a thread has the loads of PEERS x U
        // groups in flight, and sums in rank order
        const int groups = sh.NT / 4;                    // per row of X
        const int total = min(T, sh.M - t0) * groups;
        const int lo = (int)((int64_t)total * rank / CS), hi = (int)((int64_t)total * (rank + 1) / CS);
        const uint32_t part_at = smem_u32(ring);
        const int step = (int)blockDim.x;
        auto reduce = [&](auto peers_t, auto u_t) {
            constexpr int PEERS = decltype(peers_t)::value, U = decltype(u_t)::value;
            uint32_t base_at[PEERS];
#pragma unroll
            for (int j = 0; j < PEERS; ++j)
                base_at[j] = j < (int)CS ? mapa_shared(part_at, j) : 0;
            for (int i0 = lo + (int)threadIdx.x; i0 < hi; i0 += U * step) {
                float4 v[PEERS][U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = i0 + u * step, t = i / groups;
                    const uint32_t off = 4 * (t * PS + 4 * (i - t * groups));
#pragma unroll
                    for (int j = 0; j < PEERS; ++j)
                        if (i < hi && j < (int)CS)
                            v[j][u] = PEERS == 1 ? *reinterpret_cast<const float4 *>(ring + off)
                                                 : ld_cluster_f4(base_at[j] + off);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = i0 + u * step, t = i / groups, n = n0 + 4 * (i - t * groups);
                    if (i >= hi || n >= sh.N)            // (N % 16 == 0: a group of 4 is in or out)
                        continue;
                    float4 a = v[0][u];
#pragma unroll
                    for (int j = 1; j < PEERS; ++j)
                        if (j < (int)CS) {
                            a.x += v[j][u].x;
                            a.y += v[j][u].y;
                            a.z += v[j][u].z;
                            a.w += v[j][u].w;
                        }
                    const int64_t at = (int64_t)(t0 + t) * sh.N + n;
                    if (!RFQ_IN_BOUNDS(at + 3, (int64_t)sh.M * sh.N))
                        continue;
                    if (sh.out_bf16) {
                        const __nv_bfloat162 b0 = __floats2bfloat162_rn(a.x, a.y), b1 = __floats2bfloat162_rn(a.z, a.w);
                        *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(y) + at) = make_uint2(
                            *reinterpret_cast<const uint32_t *>(&b0), *reinterpret_cast<const uint32_t *>(&b1));
                    } else {
                        *reinterpret_cast<float4 *>(static_cast<float *>(y) + at) = a;
                    }
                }
            }
        };
        if (CS == 1)
            reduce(Int<1>{}, Int<8>{});
        else if (CS == 2)
            reduce(Int<2>{}, Int<4>{});
        else if (CS <= 4)
            reduce(Int<4>{}, Int<2>{});
        else
            reduce(Int<8>{}, Int<1>{});
    }
    __syncwarp();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, (uint32_t)sh.tmem_cols);
    }
    if (CS > 1)
        cluster_sync();                  // no CTA leaves while a peer still reads its partial tile
}

// Shared memory of a CTA that allocates `cols` TMEM columns (see above).
constexpr size_t smem_for(int cols) { return (size_t)cols * 456 - 1024; }
static_assert(smem_for(512) == 227 * 1024 && smem_for(256) == 113 * 1024, "shared memory budget");

// wt: 128-row W~ blocks per tile; cs: cluster size; cols: TMEM columns (256:
// two CTAs per SM); nt > 0: X on the M side, nt output columns per tile
struct Plan {
    int wt, cs, cols, nt;
};

// Fills the launch shape of a plan; false when the plan does not fit.
bool make_shape(const GemmSmallArgs &a, int64_t plan_rows, const Plan &p, Shape &s)
{
    const bool f4 = !a.bf16, swap = p.nt > 0;
    const int tiles_t = (int)((a.M + 127) / 128);
    s.M = (int)a.M;
    s.N = (int)a.N;
    s.K = (int)a.K;
    s.T = (int)(((a.M + tiles_t - 1) / tiles_t + 15) / 16 * 16);
    s.NT = swap ? p.nt : p.wt * WROWS;
    s.res = a.residual;
    s.cat = s.res && plan_rows <= 64 && !swap;   // (a chunk of a taller matrix sums as the whole does)
    s.out_bf16 = a.out_bf16;
    s.x_atoms = s.T % 128 == 0 || tiles_t == 1 ? 1 : 2;
    s.w_atoms = s.NT % 128 == 0 ? s.NT / 128 : (s.NT + 112 + 127) / 128;   // (starts are multiples of 16)
    s.x_off = s.NT * ROW;
    s.r_off = s.x_off + s.T * ROW;
    s.sf_off = s.r_off + (s.res ? s.T * ROW : 0);
    s.stage_bytes = s.sf_off + (f4 ? (s.w_atoms + s.x_atoms * (s.res ? 2 : 1)) * 2 * ATOM : 0);
    if (swap) {   // the MMA reads 128 rows of X from the tile's first, whatever follows its T
        const int end = (s.res ? s.r_off : s.x_off) + WROWS * ROW;
        s.stage_bytes = s.stage_bytes > end ? s.stage_bytes : end;
    }
    s.acc_cols = swap ? 0 : (s.T * (s.cat ? 2 : 1) + 31) / 32 * 32;
    s.sf_col0 = swap ? (s.NT + 31) / 32 * 32 : p.wt * s.acc_cols;
    s.tmem_cols = p.cols;
    const int64_t ring = (int64_t)smem_for(p.cols) - 1024 - (int64_t)kCtlBytes;
    int st = (int)(ring / s.stage_bytes);
    st = st < MAX_STAGES ? st : MAX_STAGES;
    if (f4) {
        const int slots = (p.cols - s.sf_col0) / SLOT_COLS;
        st = st < slots ? st : slots;
    }
    s.stages = st;
    // (of 0, 4, 16 and 64 stages in a layer call: 1 x 4096 x 24576 15.5 / 15.0 /
    // 15.9 / 15.9 us, HiF4 32 x 12288 x 4096 27.0 / 26.4 / 25.6 / 28.5, 333 rows best
    // with none; the fused form has no quantizer ahead of it)
    s.prefetch = plan_rows > 128 || a.fused ? 0 : f4 ? 4 : 16;
    const int ps = swap ? 2 * WROWS + 4 : s.NT;
    if (a.fused && (swap || a.M > 128))
        return false;
    return st >= 2 && s.sf_col0 <= p.cols && (int64_t)(swap ? WROWS : s.T) * ps * 4 <= ring;
}

template <bool F4, bool FUSED, int WT, bool SWAP = false>
cudaError_t launch_variant(const GemmSmallArgs &a, const Plan &p, const Shape &s, cudaStream_t st)
{
    auto kern = gemm_small_kernel<F4, FUSED, WT, SWAP>;
    const size_t smem = smem_for(p.cols);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_for(512));
    if (e != cudaSuccess)
        return e;
    CUtensorMap tw, tx, tr;
    const uint64_t rb = F4 ? (uint64_t)a.K / 2 : (uint64_t)a.K * 2;   // bytes per operand row
    if (!encode_tmap_2d_u8(&tw, a.w, rb, (uint64_t)a.N, rb, ROW, (uint32_t)(SWAP ? s.NT : WROWS), 128))
        return cudaErrorInvalidValue;
    if (FUSED)
        tx = tw;   // (unused: the converters read X)
    else if (!encode_tmap_2d_u8(&tx, a.x, rb, (uint64_t)a.M, rb, ROW, (uint32_t)s.T, 128))
        return cudaErrorInvalidValue;
    if (FUSED || !a.residual)
        tr = tx;
    else if (!encode_tmap_2d_u8(&tr, a.r, rb, (uint64_t)a.M, rb, ROW, (uint32_t)s.T, 128))
        return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((a.N + s.NT - 1) / s.NT * p.cs), (unsigned)((a.M + s.T - 1) / s.T));
    cfg.blockDim = dim3(FUSED ? 32 * (CONV_WARP0 + CONV_WARPS) : 32 * CONV_WARP0);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)p.cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    // The kernel ahead in the stream is usually the activation quantizer (2-4 us
    // for few rows): this one's set-up and its first look at W~ overlap it.
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = a.plain ? 1 : 2;
    return cudaLaunchKernelEx(&cfg, kern, tw, tx, tr, (const uint8_t *)a.w_sf, (const uint8_t *)a.x_sf,
                              (const uint8_t *)a.r_sf, FUSED ? (const uint4 *)a.x : nullptr, a.y, a.status, s);
}

// Clusters of cs CTAs that the GPU holds at once, one CTA per SM (all 512 TMEM
// columns) and two (256): cudaOccupancyMaxActiveClusters on a GB300.
constexpr int kClusters[2][MAX_CLUSTER] = {{152, 76, 46, 36, 28, 23, 15, 15}, {304, 152, 97, 74, 58, 46, 38, 36}};

// How a plan's tiles run: clusters in turn on the SMs, `share` CTAs of an SM at
// once, n k-stages per CTA.
struct Walk {
    int tiles, waves, share, nks, n;
};

Walk walk_of(const GemmSmallArgs &a, const Plan &p, const Shape &s)
{
    Walk w;
    w.tiles = (int)((a.N + s.NT - 1) / s.NT * ((a.M + s.T - 1) / s.T));
    const bool two = p.cols == 256 && !a.fused;        // (the fused form's threads fill an SM)
    const int cap = kClusters[two][p.cs - 1];
    w.waves = (w.tiles + cap - 1) / cap;
    w.share = two && w.tiles * p.cs > kClusters[0][0] ? 2 : 1;
    w.nks = (int)((a.K + (a.bf16 ? 63 : 255)) / (a.bf16 ? 64 : 256));
    w.n = (w.nks + p.cs - 1) / p.cs;
    return w;
}

// Estimated microseconds of a plan.  The constants are a fit to the times of
// 3,900 (shape, plan) pairs, M 8-900, K 1024-12288, N 1536-24576, both operand
// kinds; choosing by it costs 2% on average against the best plan measured.
//   a stage takes what its bytes need at 118 KB/us per SM (92 with three stages
//   in flight, 85 with two), or its MMAs;
//   5.4 us are launch, set-up and the first stage's latency, 4.8 of them again
//   for each further wave, 0.4 per CTA of a cluster its barriers and reads;
//   0.73 us per 10,000 outputs the epilogue;
//   W~ from HBM at 5.1 TB/s is the least.
float plan_us(const GemmSmallArgs &a, const Plan &p, const Shape &s)
{
    const bool f4 = !a.bf16, swap = p.nt > 0;
    const Walk w = walk_of(a, p, s);
    const int waves = w.waves, share = w.share, n = w.n;
    const float xrows = a.fused ? 0.f : (float)(s.T * (s.res ? 2 : 1));
    const float kb = ((float)s.NT + xrows) / 8.f + (f4 ? (float)(s.w_atoms + (a.fused ? 0 : s.x_atoms * (s.res ? 2 : 1))) : 0.f);
    const int depth = s.stages * share;
    float per = kb * share / (depth >= 4 ? 118.f : depth == 3 ? 92.f : 85.f);
    auto mma = [](float cols) { return cols > 128.f ? cols / 2 : 32.f + cols / 4; };   // cycles of 128 x cols
    const float c = swap     ? 4.f * (s.res ? 2 : 1) * mma((float)s.NT)
                    : s.cat  ? 4.f * p.wt * mma(2.f * s.T)
                             : 4.f * (s.res ? 2 : 1) * p.wt * mma((float)s.T);
    per = fmaxf(per, c * share / 1900.f);
    if (a.fused)
        // a converter warp's step (four rows): 0.93 us while its stage's other waits show,
        // beyond 64 rows, where its steps follow one another, 0.78, without a residual 0.57
        per = fmaxf(per, (s.T <= 64 ? 0.93f : s.res ? 0.78f : 0.57f) * s.T / (4.f * CONV_WARPS));
    const float t = 0.6f + (p.cs > 1 ? 0.4f * p.cs : 0.f) +
                    waves * (4.8f + n * per + 0.73e-4f * s.T * s.NT / p.cs);
    const float hbm = (float)a.N * a.K * (f4 ? 0.53125f : 2.f) / 5.1e6f;
    return fmaxf(t, 5.4f + hbm) + 0.02f * n * per;      // (the shorter plan among those that HBM bounds)
}

// The same for the kernels this one competes with: 256 x 256 tiles on CTA
// pairs (MXFP4, M > 128), or 128 x 256 tiles on single CTAs.
float tiled_us(const GemmSmallArgs &a, int64_t rows)
{
    const int nt = (int)((a.N + 255) / 256);
    if (!a.bf16 && rows > 128) {
        const int waves = (int)(((rows + 255) / 256 * nt + 75) / 76);
        return 5.f + waves * (0.56f * ((a.K + 255) / 256) + 1.6f);
    }
    const int tiles = (int)((rows + 127) / 128 * nt), waves = (tiles + 151) / 152;
    if (a.bf16)
        return 4.4f + waves * 0.58f * (a.K / 64);
    return 4.2f + waves * (0.63f + 0.35f * tiles / 152.f) * ((a.K + 255) / 256);
}

// The estimates above are for layers whose residual is multiplied in full; the
// tiled kernels skip what is not there, and need a quarter less.  A layer
// without a residual, or with phi (of which nothing is known here, so with no
// tile kept, the tiled kernels' best), therefore has to pass a second
// comparison, of estimates fitted to 2,144 layers that were timed on both
// kernels, M 1-4096, K 512-13824, N 512-24576 (relative error 5%; bf16 7%):
//   here   one + cluster cs + wave waves + kb (100 KB copied per SM, in turn) +
//          hbm (MB of W~) + epi (10,000 outputs of a CTA, in turn) + moved (MB
//          copied by all) + wide (stages of 256 W~ rows on the M side by 128
//          rows of X, in turn)
//   tiled  one + wave waves + k_wave (k-stages, in turn) + k_tile (k-stages
//          times tiles per CTA or pair) + hbm
// The margins are those with the fewest layers slower than on the other kernel.
struct LightFit {
    float one, cluster, wave, kb, hbm, epi, moved, wide;
    struct Tiled {
        float one, wave, k_wave, k_tile, hbm;
    } pair, single;
    float margin, slack;
};
constexpr LightFit kNoResidual[2] = {
    {1.095f, 0.678f, 3.953f, 0.451f, 0.069f, 0.794f, 0.036f, 0.066f,
     {5.215f, 1.042f, 0.276f, 0.054f, 0.086f}, {0.f, 4.151f, 0.391f, 0.f, 0.099f}, 0.97f, 0.3f},
    {0.f, 0.468f, 5.747f, 0.396f, 0.087f, 0.469f, 0.027f, 0.121f,
     {}, {4.657f, 0.078f, 0.346f, 0.065f, 0.066f}, 1.04f, 1.5f}};
constexpr LightFit kPhi[2] = {
    {1.283f, 0.63f, 3.62f, 0.321f, 0.081f, 0.954f, 0.042f, 0.043f,
     {6.315f, 1.022f, 0.275f, 0.06f, 0.086f}, {0.f, 5.198f, 0.399f, 0.f, 0.096f}, 0.97f, 0.3f},
    {0.f, 0.353f, 6.028f, 0.236f, 0.092f, 0.323f, 0.033f, 0.142f,
     {}, {5.522f, 0.093f, 0.353f, 0.064f, 0.066f}, 1.02f, 1.f}};
// bf16 operands with the whole residual, up to 128 rows: the first comparison
// underrates what a split reduction costs where W~ (2 bytes an element) comes
// from HBM.  32 x 3584 x 18944: 48.5 us here against 43.5.
constexpr LightFit kBf16Decode = {0.f, 0.353f, 6.028f, 0.236f, 0.092f, 0.323f, 0.033f, 0.142f,
                                  {}, {5.39f, 0.244f, 0.513f, 0.067f, 0.037f}, 1.02f, 0.f};

float light_plan_us(const GemmSmallArgs &a, const LightFit &f, const Plan &p, const Shape &s)
{
    const Walk w = walk_of(a, p, s);
    const float kb = (float)(s.NT + s.T * (s.res ? 2 : 1)) / 8.f + (a.bf16 ? 0.f : 2.f);
    const float in_turn = (float)(w.waves * w.n * w.share);
    const bool wide = p.nt == 0 && s.NT == 2 * WROWS && !s.cat;
    return f.one + (p.cs > 1 ? f.cluster * p.cs : 0.f) + f.wave * w.waves + f.kb * in_turn * kb / 100.f +
           f.hbm * ((float)a.N * a.K * (a.bf16 ? 2.f : 0.53125f) / 1e6f) + f.epi * w.waves * s.T * s.NT / p.cs / 1e4f +
           f.moved * ((float)w.tiles * w.nks * kb / 1e3f) + (wide ? f.wide * in_turn * s.T / 128.f : 0.f);
}

float light_tiled_us(const GemmSmallArgs &a, const LightFit &f, int64_t rows)
{
    const int64_t nt = (a.N + 255) / 256;
    const bool pair = !a.bf16 && rows > 128;
    const LightFit::Tiled &t = pair ? f.pair : f.single;
    const int64_t tiles = pair ? (rows + 255) / 256 * nt : (rows + 127) / 128 * nt, at_once = pair ? 76 : 152;
    const float waves = (float)((tiles + at_once - 1) / at_once), n = (float)((a.K + (a.bf16 ? 63 : 255)) / (a.bf16 ? 64 : 256));
    return t.one + t.wave * waves + t.k_wave * waves * n + t.k_tile * n * tiles / at_once +
           t.hbm * ((float)a.N * a.K * (a.bf16 ? 2.f : 0.53125f) / 1e6f);
}

// The second comparison, of a plan that the first one took.
bool still_faster(const GemmSmallArgs &a0, int64_t rows, const Plan &p)
{
    const bool full = a0.residual && !a0.phi;
    if (full && (!a0.bf16 || rows > 128))
        return true;
    GemmSmallArgs a = a0;
    a.M = rows;
    Shape s;
    if (!make_shape(a, rows, p, s))
        return false;
    const LightFit &f = full ? kBf16Decode : (a.phi ? kPhi : kNoResidual)[a.bf16 != 0];
    return light_plan_us(a, f, p, s) * f.margin < light_tiled_us(a, f, rows) + f.slack;
}

// The fastest plan for a layer of `rows` rows; its estimate, or a huge number.
float best_plan(const GemmSmallArgs &a0, int64_t rows, Plan &best)
{
    GemmSmallArgs a = a0;
    a.M = rows;
    const int nks = (int)((a.K + (a.bf16 ? 63 : 255)) / (a.bf16 ? 64 : 256));
    float t = 1e30f;
    auto offer = [&](const Plan &p) {
        Shape s;
        if (!make_shape(a, rows, p, s))
            return;
        const float e = plan_us(a, p, s);
        if (e < t) {
            t = e;
            best = p;
        }
    };
    constexpr int kCs[6] = {1, 2, 3, 4, 6, 8};
    constexpr int kNt[10] = {96, 112, 128, 144, 160, 176, 192, 208, 224, 256};
    for (int cs : kCs) {
        if (cs > nks)
            break;
        offer({1, cs, 512, 0});
        offer({1, cs, 256, 0});
        offer({2, cs, 512, 0});
        if (rows > 64 && !a.fused)                     // (fewer rows: X on the N side is the narrower tile)
            for (int nt : kNt)
                offer({2, cs, 512, nt});
    }
    return t;
}

// Whether this kernel may take a layer of more than 1024 rows: where the tiled
// kernels' tiles (256 x 256 on 76 CTA pairs, bf16 128 x 256 on 152 CTAs) make at
// most three waves, so that a first or last wave that is nearly empty weighs.
// GEMM times, tiled -> here, us: MXFP4 1800 x 12288 x 512 32.1 -> 19.5, 1300 x
// 4096 x 1024 14.8 -> 14.2, 1025 x 4096 x 4096 24.4 -> 18.6, 1025 x 12288 x 4096
// 58.4 -> 38.7; HiF4 1025 x 12288 x 800 113 -> 33, 1800 x 4096 x 1024 42.4 -> 25.1,
// 1300 x 12288 x 4096 223 -> 157.  Of 276 such shapes (700 to 8190 rows, 512 to 7168
// columns) the estimates gave this kernel none that the tiled one does faster,
// and beyond two waves hardly any MXFP4 shape; with more waves the tiled kernels'
// larger tiles are the faster ones.  With phi the tiled kernels may skip up to
// the whole residual, so half their time has to be beaten.
bool few_waves(const GemmSmallArgs &a, int64_t rows)
{
    const int64_t nt = (a.N + 255) / 256;
    return a.bf16 ? (rows + 127) / 128 * nt <= 3 * 152 : (rows + 255) / 256 * nt <= 3 * 76;
}

// A layer's choice: its plan (cs = 0: none fits) and whether this kernel is the
// faster one.  The search costs a few microseconds of host time, so each host
// thread keeps the choices of its last shapes (a direct-mapped table).
struct Choice {
    int64_t rows = -1, N = 0, K = 0;
    int flags = 0;
    Plan plan = {};
    bool take = false;
};

const Choice &choose(const GemmSmallArgs &a, int64_t rows)
{
    constexpr int kEntries = 64;
    static thread_local Choice table[kEntries];
    const int flags = (a.residual ? 1 : 0) | (a.bf16 ? 2 : 0) | (a.fused ? 4 : 0) | (a.phi ? 8 : 0);
    const uint64_t h = ((uint64_t)rows * 0x9E3779B97F4A7C15ull ^ (uint64_t)a.N * 0xC2B2AE3D27D4EB4Full ^
                        (uint64_t)a.K * 0x165667B19E3779F9ull ^ (uint64_t)flags * 0x27D4EB2F165667C5ull) >> 40;
    Choice &c = table[h % kEntries];
    if (c.rows != rows || c.N != a.N || c.K != a.K || c.flags != flags) {
        c.rows = rows;
        c.N = a.N;
        c.K = a.K;
        c.flags = flags;
        c.plan = {};
        c.take = (rows <= 1024 || few_waves(a, rows)) &&
                 best_plan(a, rows, c.plan) * 1.05f < tiled_us(a, rows) * (rows > 1024 && a.phi ? 0.5f : 1.f) &&
                 still_faster(a, rows, c.plan);
    }
    return c;
}

} // namespace

bool gemm_small_takes(const GemmSmallArgs &a, int64_t plan_rows) { return choose(a, plan_rows).take; }

namespace {
// (a layer that the choice never offers to this kernel has no plan in the table)
Plan plan_of(const GemmSmallArgs &a, int64_t plan_rows)
{
    Plan p = choose(a, plan_rows).plan;
    if (p.cs == 0)
        best_plan(a, plan_rows, p);
    return p;
}
} // namespace

void gemm_small_plan(const GemmSmallArgs &a, int64_t plan_rows, rfq_linear_plan &out)
{
    const Plan p = plan_of(a, plan_rows);
    Shape s;
    out.cluster = 0;
    out.tiled_us = a.fused ? 0.f : tiled_us(a, plan_rows);
    if (p.cs == 0 || !make_shape(a, plan_rows, p, s))
        return;
    out.cluster = p.cs;
    out.rows = s.T;
    out.cols = s.NT;
    out.x_on_m = p.nt > 0;
    out.joint = s.cat;
    out.ctas_per_sm = p.cols == 256 && !a.fused ? 2 : 1;
    out.stages = s.stages;
    out.cluster_us = plan_us(a, p, s);
}

cudaError_t launch_gemm_small(const GemmSmallArgs &a, int64_t plan_rows, cudaStream_t st)
{
    const Plan p = plan_of(a, plan_rows);
    Shape s;
    if (p.cs == 0)
        return cudaErrorInvalidValue;
    if (!make_shape(a, plan_rows, p, s))
        return cudaErrorInvalidValue;
    if (p.nt > 0)
        return a.bf16 ? launch_variant<false, false, 2, true>(a, p, s, st)
                      : launch_variant<true, false, 2, true>(a, p, s, st);
    if (a.bf16)
        return p.wt == 2 ? launch_variant<false, false, 2>(a, p, s, st) : launch_variant<false, false, 1>(a, p, s, st);
    if (a.fused)
        return p.wt == 2 ? launch_variant<true, true, 2>(a, p, s, st) : launch_variant<true, true, 1>(a, p, s, st);
    return p.wt == 2 ? launch_variant<true, false, 2>(a, p, s, st) : launch_variant<true, false, 1>(a, p, s, st);
}

RFQ_DEBUG_WORD_ACCESSOR(debug_word_gemm_small)

} // namespace rfq
