// Grouped GEMM on CTA pairs with dynamic tile scheduling: every product of a
// pass that has no bottleneck between them in one launch, whatever the
// majorness of its operands and the type of its output.
//
// The pair protocol (tc_pair.cuh), per tile of 256 x bn:
//   producer (warp 0 of each CTA) -> MMA issuer (warp 1 of the leader) ->
//   epilogue (warps 2-9 of each CTA).
// Launches of several products add four warps per CTA: a scheduler (warp 10 of
// the leader), the others sum the bottleneck kernel's partials meanwhile.
//
// Tiles: with a counter in memory (published by an earlier kernel of the call),
// each tile goes to the pair that asks first, in order of index: pairs that a
// programmatic launch starts early, on SMs that the previous kernel leaves
// free, take more tiles than late ones, and with the heavy tiles first the
// order is list scheduling, without a schedule computed on the host.  Without
// one, pair c takes tiles c, c + pairs, ...  Where nothing runs beside the launch
// (`together`) all pairs start at once and pair c begins with tile c by itself,
// without the first draw's way through the scheduler (7893 x 3848 -> 256, r = 0:
// 61.1 -> 60.3 us).  The scheduler asks for tile j + 1 when the producer starts to
// load tile j and passes the index on to every warp of both CTAs through shared
// memory; producer and MMA issuer fetch it a few k-blocks before the end of tile j
// and locate it a few k-blocks later, so that neither step alone outlasts what
// the ring holds.  The epilogue warps hand a slot back once the tile's accumulator
// is complete: by then producers and MMA issuer, whose copies and MMAs depend on
// what they read, have read it.  (Arrivals of their own, a release at cluster
// scope per tile, stall the threads that issue copies and MMAs: 16384 x 8192 ->
// 2048, r = 128, 752 us instead of 730, 49731 x 128 -> 656, r = 0, 58.5 instead of 55.4.)
// Cluster launch control in place of the counter answers later than a tile of 17
// k-blocks takes: 66 us against 48 on 8192 x 1024 x 4096, 427 against 297 on 16384 x
// 2048 x 8192.
//
// The counter is one 64-bit word, [tag of the call | next tile], which only
// atomics of device scope touch while the launch runs.  A pair may draw before
// the kernel that publishes the word is known to have run: only
// griddepcontrol.wait orders a dependent grid after its predecessor, and the
// scheduler does not start with one.  So a draw counts only if it returns the
// call's tag; one that does not waits for the predecessor grid and draws again,
// and what it added to the old word is lost when the new one is published.  The
// last draw clears the word: the tag of a captured call, the same on every
// replay, is then never found in what an earlier replay left.  Tag 0: a memset
// cleared the word, complete before this launch or its predecessor began.
#pragma once

#include "sums.cuh"
#include "tc_pair.cuh"

namespace noble {
namespace tc {
namespace group {

constexpr uint32_t kAMn = 1, kBMn = 2;    // operand is MN-major ([K][rows])
constexpr uint32_t kA4 = 4, kB4 = 8;      // ... copied in the 4-D layout (make_map_mn4)
constexpr uint32_t kF32 = 16;             // C is fp32 (else bf16)
constexpr uint32_t kTma = 32;             // C is stored through a TMA map
constexpr uint32_t kCol0 = 64;            // store column 0 only
constexpr uint32_t kTranspose = 128;      // store transposed (fp32)

struct Problem {
    int64_t M, N;
    int kb0, kb1;          // k-blocks of segment 0 / 1
    int bn;                // N tile, 128 or 256
    int tiles_m, tiles_n;  // 128-row tiles, bn-column tiles
    int nsplit, kb_per_split;
    // > 0 (fp32 C without bias): the K range of a tile is accumulated in pieces
    // of so many k-blocks, added up in fp32 in C; the tensor core's accumulation
    // rounds more the longer it runs
    int piece_kb;
    int tile_begin;
    int dep;               // bit s: segment s reads what an earlier kernel of the call wrote
    // k-block of segment 0 whose rows end within an 8-row group of a 4-D
    // operand (K % 8 != 0): copied in boxes of 8 rows; -1: none
    int tail_kb;
    uint32_t flags;
    uint8_t map[7];        // A0, B0, A1, B1, C, tail of A0, tail of B0: indexes into maps
    void *C;
    int64_t ldc, split_stride;
    const float *bias;
};

template <int MAXP>
struct ArgsBase {
    static constexpr int kMaxMaps = MAXP == 1 ? 5 : 30;
    CUtensorMap maps[kMaxMaps];
    Problem p[MAXP];
    int nproblems;
    int total_tiles;
    uint32_t *status;
    unsigned long long *counter;  // [tag | next tile] (NULL: round-robin)
    uint32_t tag;
    int together;
};
template <int MAXP>
struct Args : ArgsBase<MAXP> {
    SplitJobs sums;
};
template <>
struct Args<1> : ArgsBase<1> {
};

constexpr int kSlots = 4;
constexpr int kSumWarps = 7;  // per pair
template <int MAXP>
constexpr int threads() { return pair::kPairThreads + (MAXP > 1 ? 128 : 0); }

template <int STAGES>
struct Smem {
    static constexpr uint32_t kA = kBM * kBK * 2;  // 128 rows of A
    static constexpr uint32_t kB = 128 * kBK * 2;  // up to 128 columns of B
    static constexpr uint32_t kStage = kA + kB;
    static constexpr uint32_t kStgOff = STAGES * kStage;  // epilogue staging, 4 KB per epilogue warp
    static constexpr uint32_t kTileOff = kStgOff + 8 * 4096;  // tile indexes
    static constexpr uint32_t kBarOff = kTileOff + 8 * kSlots;
    // full, empty, tfull[2], tempty[2], mma_done, want, tile_full, tile_empty
    static constexpr uint32_t kNumBars = 2 * STAGES + 6 + 2 * kSlots;
    static constexpr uint32_t kBytes = kBarOff + 8 * kNumBars + 16;
    static constexpr uint32_t kDynamic = kBytes + 1024;
};

template <int MAXP, int STAGES>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(threads<MAXP>(), 1)
gemm_group(const __grid_constant__ Args<MAXP> g)
{
    using S = Smem<STAGES>;
    using pair::PairTile;
    constexpr uint32_t kAccCols = 256;
    constexpr uint32_t kCols = 512;
    // launches of one product: round-robin, whole K ranges
    constexpr bool kDynamic = MAXP > 1;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = ptx::smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (sbase - raw);
    const uint32_t bar0 = sbase + S::kBarOff;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 + b); };
    const uint32_t mma_done = bar0 + 8u * (2 * STAGES + 4);
    const uint32_t want = bar0 + 8u * (2 * STAGES + 5);
    auto tile_full = [&](int s) { return bar0 + 8u * (2 * STAGES + 6 + s); };
    auto tile_empty = [&](int s) { return bar0 + 8u * (2 * STAGES + 6 + kSlots + s); };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + S::kBarOff + 8 * S::kNumBars);

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const uint32_t rank = cluster::ctarank();
    const bool leader = rank == 0;

    if (warp == 0 && lane == 0) {
        ptx::griddep_launch();  // the next kernel of the call may take SMs as this grid frees them
        ptx::tma_prefetch_desc(&g.maps[g.p[0].map[0]]);
        ptx::tma_prefetch_desc(&g.maps[g.p[0].map[1]]);
        for (int s = 0; s < STAGES; ++s) {
            ptx::mbar_init(full_bar(s), 1);
            ptx::mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(tfull_bar(b), 1);
            ptx::mbar_init(tempty_bar(b), 16);  // 8 epilogue warps in each CTA of the pair
        }
        ptx::mbar_init(mma_done, 1);
        ptx::mbar_init(want, 1);
        for (int s = 0; s < kSlots; ++s) {
            ptx::mbar_init(tile_full(s), 1);
            ptx::mbar_init(tile_empty(s), 16);  // eight epilogue warps per CTA
        }
        ptx::fence_barrier_init();
    }
    if (warp == 1) {
        pair::tmem_alloc2(ptx::smem_u32(tmem_slot), kCols);
        pair::tmem_relinquish2();
    }
    ptx::tc_fence_before();
    __syncthreads();
    const int pairs = gridDim.x / 2;
    unsigned long long *const counter = kDynamic ? g.counter : nullptr;
    // tiles that are not drawn
    const int given = kDynamic && g.together ? pairs : 0;
    // the tile that a draw gives; total_tiles or more: none left
    auto drawn_tile = [&](unsigned long long v) -> int {
        if ((uint32_t)(v >> 32) != g.tag) {
            ptx::griddep_wait();
            v = atomicAdd(counter, 1ull);
            if ((uint32_t)(v >> 32) != g.tag) {
                raise_status(g.status, kStatusCounter);
                return g.total_tiles;
            }
        }
        // every pair draws until it gets none: the last of those draws
        if ((uint32_t)v == (uint32_t)(g.total_tiles - given + pairs - 1)) atomicExch(counter, 0ull);
        return given + (int)(uint32_t)v;
    };
    unsigned long long drawn = 0;  // the scheduler's first draw, on its way during the set-up
    if (kDynamic && warp == 10 && lane == 0 && leader && counter) drawn = atomicAdd(counter, 1ull);
    cluster::sync();  // the peer's barriers are initialised before any remote use
    ptx::tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // The j-th tile of this pair (-1: none left; -2: the wait gave up).  One
    // thread of each consumer calls it.
    auto get_tile = [&](int j) -> int {
        if (!counter) {
            const int t = (int)(blockIdx.x / 2) + j * pairs;
            return t < g.total_tiles ? t : -1;
        }
        if (given && j == 0) return (int)(blockIdx.x / 2);  // never more pairs than tiles
        const int q = given ? j - 1 : j;
        const int s = q % kSlots;
        if (!ptx::mbar_wait_cluster(tile_full(s), (uint32_t)(q / kSlots) & 1u, g.status)) return -2;
        return *reinterpret_cast<volatile int *>(smem + S::kTileOff + 8 * s);
    };

    if (warp == 0) {
        if (lane == 0) {
            // ---------------- producer (both CTAs)
            uint32_t it = 0;
            bool ok = true;
            bool waited = false;  // for the predecessor grid (programmatic launch)
            int t = get_tile(0);
            for (int j = 0; ok && t >= 0; ++j) {
                if (leader && counter) ptx::mbar_arrive(want);  // the scheduler asks for the next tile
                const PairTile tr = pair::locate_pair(g, t, (int)rank);
                // everything that the k loop reads of the problem, once per tile:
                // it would be fetched again from the parameters after every copy
                // (reloading it made the loop 1.5 times slower than the MMAs)
                const Problem &P = g.p[tr.prob];
                const uint32_t fl = P.flags;
                const int kb0 = P.kb0, dep = P.dep, tail_kb = P.tail_kb;
                const int bh = P.bn / 2;  // B columns held by this CTA
                const uint32_t cta_bytes = S::kA + (uint32_t)bh * kBK * 2;
                const int m0 = (int)tr.m0, nb = (int)tr.n0 + (int)rank * bh;
                const CUtensorMap *mA = &g.maps[P.map[0]], *mB = &g.maps[P.map[1]];
                const CUtensorMap *mA1 = &g.maps[P.map[2]], *mB1 = &g.maps[P.map[3]];
                const CUtensorMap *tA = &g.maps[P.map[5]], *tB = &g.maps[P.map[6]];
                const int kb_begin = tr.kb_begin, kb_end = tr.kb_end;
                int s = it % STAGES;
                uint32_t ph = (it / STAGES) & 1;
                const int kb_fetch = counter ? max(kb_begin, kb_end - 5) : -1;
                for (int kb = kb_begin; kb < kb_end; ++kb, ++it) {
                    if (kb == kb_fetch) t = get_tile(j + 1);
                    if (!ptx::mbar_wait(empty_bar(s), ph ^ 1, g.status)) {
                        ok = false;
                        break;
                    }
                    const bool seg1 = kb >= kb0;
                    if (!waited && (dep & (seg1 ? 2 : 1))) {
                        ptx::griddep_wait();
                        waited = true;
                    }
                    const uint32_t fb = cluster::map_to_rank(full_bar(s), 0);
                    if (leader) ptx::mbar_arrive_expect_tx(full_bar(s), 2 * cta_bytes);
                    const uint32_t sA = sbase + s * S::kStage, sB = sA + S::kA;
                    if (kb == kb0) mA = mA1, mB = mB1;
                    const int k = (seg1 ? kb - kb0 : kb) * kBK;
                    if (kb == tail_kb) {
                        // the same layout in boxes of 64 columns x 8 rows, zeros past K
                        for (int r8 = 0; r8 < 8; ++r8) {
                            for (int c = 0; c < 2; ++c)
                                pair::tma_load_2d_pair(sA + r8 * 2048 + c * 1024, tA, fb, m0 + 64 * c, k + 8 * r8);
                            for (int c = 0; c < bh / 64; ++c)
                                pair::tma_load_2d_pair(sB + (r8 * (bh / 64) + c) * 1024, tB, fb, nb + 64 * c, k + 8 * r8);
                        }
                    } else {
                        if (fl & kA4) {
                            pair::tma_load_4d_pair(sA, mA, fb, m0 / 64, k / 8);
                        } else if (fl & kAMn) {
                            pair::tma_load_2d_pair(sA, mA, fb, m0, k);
                            pair::tma_load_2d_pair(sA + kChunkBytes, mA, fb, m0 + 64, k);
                        } else {
                            pair::tma_load_2d_pair(sA, mA, fb, k, m0);
                        }
                        if (fl & kB4) {
                            pair::tma_load_4d_pair(sB, mB, fb, nb / 64, k / 8);
                        } else if (fl & kBMn) {
                            for (int c = 0; c < bh / 64; ++c)
                                pair::tma_load_2d_pair(sB + c * kChunkBytes, mB, fb, nb + 64 * c, k);
                        } else {
                            pair::tma_load_2d_pair(sB, mB, fb, k, nb);
                        }
                    }
                    if (++s == STAGES) s = 0, ph ^= 1;
                }
                if (!counter) t = get_tile(j + 1);
            }
            // this grid completes only after its predecessor: what later kernels
            // of the call read through this grid's completion is then complete too
            if (!waited) ptx::griddep_wait();
            // the leader's ring barriers also count the peer's bytes: once they
            // complete, no copy of either CTA is still landing
            if (leader) {
                const uint32_t f = it > (uint32_t)STAGES ? it - STAGES : 0;
                for (uint32_t i = f; i < it; ++i)
                    ptx::mbar_wait(full_bar(i % STAGES), (i / STAGES) & 1, nullptr);
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && leader) {
            // ---------------- MMA issuer (leader CTA only).  The loop keeps the
            // work between consecutive k-blocks small: operand descriptors are
            // a per-tile base plus additive offsets (start addresses are below
            // 256 KB, so the 14-bit address field never carries), and the ring
            // position advances incrementally.
            int s = 0;
            uint32_t ph = 0;
            int acc = 0;  // accumulator uses so far
            bool ok = true;
            uint32_t *const status = g.status;
            constexpr uint32_t kStageUnits = S::kStage / 16;
            int t = get_tile(0);
            for (int j = 0; ok && t >= 0; ++j) {
                const PairTile tr = pair::locate_pair(g, t, 0);
                const Problem &P = g.p[tr.prob];
                const uint32_t fl = P.flags;
                const uint32_t idesc = ptx::idesc_bf16(2 * kBM, P.bn, (fl & kAMn) != 0, (fl & kBMn) != 0);
                const uint32_t nchB = (uint32_t)P.bn / 128;  // 64-wide B chunks held per CTA
                const uint64_t a0 = (fl & kA4)    ? ptx::smem_desc_sw128(sbase, 1024, 2048)
                                    : (fl & kAMn) ? ptx::smem_desc_sw128(sbase, kChunkBytes, 1024)
                                                  : ptx::smem_desc_sw128(sbase, 16, 1024);
                const uint64_t b0 = (fl & kB4)    ? ptx::smem_desc_sw128(sbase + S::kA, 1024, 1024 * nchB)
                                    : (fl & kBMn) ? ptx::smem_desc_sw128(sbase + S::kA, kChunkBytes, 1024)
                                                  : ptx::smem_desc_sw128(sbase + S::kA, 16, 1024);
                // descriptor address-field steps (16-byte units) per K-step of 16
                const uint32_t stepA = (fl & kA4) ? 4096u / 16 : (fl & kAMn) ? 2048u / 16 : 2u;
                const uint32_t stepB = (fl & kB4) ? 128u * nchB : (fl & kBMn) ? 2048u / 16 : 2u;
                const int piece = kDynamic && P.piece_kb ? P.piece_kb : tr.kb_end - tr.kb_begin;
                const int kb_end = tr.kb_end;
                // every piece of the K range in an accumulator of its own
                for (int kb = tr.kb_begin; ok && kb < kb_end; kb += piece, ++acc) {
                    const int b = acc & 1;
                    if (!ptx::mbar_wait(tempty_bar(b), ((uint32_t)(acc >> 1) & 1u) ^ 1u, status)) {
                        ok = false;
                        break;
                    }
                    ptx::tc_fence_after();
                    const uint32_t d_tmem = tmem + b * kAccCols;
                    const int nkb = min(piece, kb_end - kb);
                    // a few k-blocks before the tile's end
                    const int i_fetch = counter && kb + piece >= kb_end ? max(0, ((nkb - 1) & ~1) - 4) : -1;
                    for (int i = 0; i < nkb; i += 2) {
                        if (i == i_fetch) t = get_tile(j + 1);
                        const bool two = i + 1 < nkb;
                        int s2 = s + 1;
                        uint32_t ph2 = ph;
                        if (s2 == STAGES) {
                            s2 = 0;
                            ph2 ^= 1;
                        }
                        if (!ptx::mbar_wait(full_bar(s), ph, status) || (two && !ptx::mbar_wait(full_bar(s2), ph2, status))) {
                            ok = false;
                            break;
                        }
                        // no tcgen05 fence here: the stages were written by TMA (the
                        // async proxy, as the MMA) and completed on the barrier waited for
                        const uint64_t so = (uint64_t)((uint32_t)s * kStageUnits);
                        const uint64_t ad = a0 + so, bd = b0 + so;
                        pair::mma2_bf16(d_tmem, ad, bd, idesc, i > 0 ? 1u : 0u);
#pragma unroll
                        for (int kk = 1; kk < kBK / 16; ++kk)
                            pair::mma2_bf16(d_tmem, ad + kk * stepA, bd + kk * stepB, idesc, 1u);
                        pair::mma2_commit_mc(empty_bar(s), 0x3);
                        if (two) {
                            const uint64_t so2 = (uint64_t)((uint32_t)s2 * kStageUnits);
                            const uint64_t ad2 = a0 + so2, bd2 = b0 + so2;
#pragma unroll
                            for (int kk = 0; kk < kBK / 16; ++kk)
                                pair::mma2_bf16(d_tmem, ad2 + kk * stepA, bd2 + kk * stepB, idesc, 1u);
                            pair::mma2_commit_mc(empty_bar(s2), 0x3);
                            s = s2 + 1;
                            ph = ph2;
                            if (s == STAGES) {
                                s = 0;
                                ph ^= 1;
                            }
                        } else {
                            s = s2;
                            ph = ph2;
                        }
                    }
                    pair::mma2_commit_mc(tfull_bar(b), 0x3);
                }
                if (!counter) t = get_tile(j + 1);
            }
            pair::mma2_commit_mc(mma_done, 0x1);
            ptx::mbar_wait(mma_done, 0, nullptr);
        }
    } else if (kDynamic && warp == 10 && leader) {
        if (lane == 0 && counter) {
            // ---------------- tile scheduler
            int t = drawn_tile(drawn);
            // a pair's tile 0 that is given is not asked for: its `want` first, as the
            // producer may start tile 1 as soon as that is published
            const int first = given ? 1 : 0;
            const bool started = !given || ptx::mbar_wait(want, 0, g.status);
            for (int j = first; started; ++j) {
                const int s = (j - first) % kSlots;
                if (t >= g.total_tiles) t = -1;
                if (!ptx::mbar_wait_cluster(tile_empty(s), ((uint32_t)((j - first) / kSlots) & 1u) ^ 1u, g.status)) break;
                const uint32_t slot = sbase + S::kTileOff + 8u * s;
                for (uint32_t q = 0; q < 2; ++q)
                    cluster::put_word(cluster::map_to_rank(slot, q), t, cluster::map_to_rank(tile_full(s), q));
                if (t < 0) break;
                if (!ptx::mbar_wait(want, (uint32_t)j & 1u, g.status)) break;
                t = drawn_tile(atomicAdd(counter, 1ull));
            }
        }
    } else if (kDynamic && warp >= 10) {
        // ---------------- sums of the preceding kernel's partials, 32 outputs a warp
        if constexpr (kDynamic) {
            const int total = (int)g.sums.begin[g.sums.njobs];
            int block = (int)(blockIdx.x / 2) * kSumWarps + (leader ? warp - 11 : warp - 7);
            if (block * 32 < total) ptx::griddep_wait();
            for (; block * 32 < total; block += pairs * kSumWarps) sum_warp(g.sums, block, lane);
        }
    } else {
        // ---------------- epilogue (both CTAs): own 128 accumulator rows
        const int quarter = warp % 4;
        const int half = (warp - 2) / 4;  // two warps per TMEM lane quarter split the columns
        const uint32_t leader_tempty0 = cluster::map_to_rank(tempty_bar(0), 0);
        const uint32_t leader_tempty1 = cluster::map_to_rank(tempty_bar(1), 0);
        const uint32_t stg = sbase + S::kStgOff + (uint32_t)(warp - 2) * 4096u;
        uint8_t *stg_ptr = smem + S::kStgOff + (warp - 2) * 4096;
        int nacc = 0;  // accumulator uses so far
        bool ok = true;
        for (int j = 0; ok; ++j) {
            int t = 0;
            if (lane == 0) t = get_tile(j);
            t = __shfl_sync(0xffffffffu, t, 0);
            if (t < 0) break;
            const PairTile tr = pair::locate_pair(g, t, (int)rank);
            const Problem &P = g.p[tr.prob];
            const uint32_t fl = P.flags;
            const int piece = kDynamic && P.piece_kb ? P.piece_kb : tr.kb_end - tr.kb_begin;
            for (int kb = tr.kb_begin; kb < tr.kb_end; kb += piece, ++nacc) {
                const int b = nacc & 1;
                ok = ptx::mbar_wait(tfull_bar(b), (uint32_t)(nacc >> 1) & 1u, g.status);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                ptx::tc_fence_after();
                const uint32_t acc = tmem + b * kAccCols;
                // the pieces after the first are added to C by the warp that
                // stored the first one, in order
                const bool add = kDynamic && kb > tr.kb_begin;
                if (add && lane == 0) ptx::bulk_wait_all();
                auto store = [&](auto epi) {
                    using Epi = decltype(epi);
                    typename Epi::Params ep{static_cast<typename Epi::out_type *>(P.C), P.ldc, P.bias, P.split_stride};
                    ep.col0 = (fl & kCol0) ? 1 : 0;
                    ep.transpose = (fl & kTranspose) ? 1 : 0;
                    ep.add = add ? 1 : 0;
                    if (fl & kTma)
                        Epi::run_tma(ep, &g.maps[P.map[4]], stg_ptr, stg, acc, P.bn, quarter, lane, tr.m0, tr.n0, P.N,
                                     tr.z, half);
                    else
                        Epi::run_dyn(ep, acc, P.bn, quarter, lane, tr.m0, tr.n0, P.M, P.N, tr.z, 32 * half, 64);
                };
                if (fl & kF32)
                    store(EpiStore<float>{});
                else
                    store(EpiStore<__nv_bfloat16>{});
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) cluster::mbar_arrive(b ? leader_tempty1 : leader_tempty0);
            }
            const int q = given ? j - 1 : j;
            if (ok && counter && q >= 0 && lane == 0) cluster::mbar_arrive(cluster::map_to_rank(tile_empty(q % kSlots), 0));
        }
        if (lane == 0) ptx::bulk_wait_all();  // stores done before the staging buffer goes away
    }

    ptx::tc_fence_before();
    __syncthreads();
    cluster::sync();  // no CTA leaves while its peer may still touch its memory
    if (warp == 1) {
        ptx::tc_fence_after();
        pair::tmem_dealloc2(tmem, kCols);
    }
}

}  // namespace group
}  // namespace tc
}  // namespace noble
