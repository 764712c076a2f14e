// Phased form of the per-fill processing: count, scan and compaction in one
// cooperative launch, the compaction a few tiles behind the count on the same SM, so
// that it re-reads its tiles from L2 instead of HBM.
//
// What bounds the two-pass form is HBM: it reads the samples twice and writes the
// pool once (6.5 TB/s over both kernels on a full fill).  Here chunk k is one tile for
// each CTA, one CTA per SM, and a tile is compacted while at most kPhaseAhead chunks
// of 152 x 48 KB lie between its two reads.  On 24 x 54 x 560,000 samples HBM reads
// fall from 2.9 to 1.6 GB (the samples are 1.45) and a fill from 657 to 487 us.
//
// Warps of a CTA, handing tiles on through mbarriers:
//   8 sum        crystal sums, threshold bits and block sums of a tile in one of two
//                count slots (sum_step_quarters);
//   2 marks      marks words, aggregate and Q bins, a tile each in turn;
//   1 load       fills the count slots; a tile's load waits until the tile
//                kPhaseAhead before it is compacted, which is what keeps the second
//                read in L2;
//   1 prefix     a tile's place.  The marks warp publishes the tile's aggregate in one
//                32-bit word; this warp reads the words of the whole chunk and
//                combines them after what it has kept of the chunks before.  Every CTA
//                does so for itself: no look-back chain, and the wait for the slowest
//                CTA of a chunk is covered by the tiles in between;
//   7 stage      a tile in one of two row slots, in place: the warps read the whole
//                tile into registers, meet, and write the marked samples' rows over it
//                (four slots fit beside each other because no second row buffer is
//                needed);
//   1 out        bulk-copies the rows, writes the records, refills the row slots.
// The waits on other CTAs end because the launch is cooperative: every CTA runs.  A
// CTA counts tile k once it has compacted tile k - kPhaseAhead, whose place needs
// every CTA's count of that chunk only.
//
// Straight-line code is what the warps' speed hangs on: with one or two warps of a
// part on a scheduler, instruction fetch is exposed.  The staging stores without a
// condition (columns that are not marked write to a spare row) and without a case
// for odd crystal counts took a fill from 652 to 552 us, Q bins in 32-bit arithmetic
// and a kernel for each kind of window (kWin32, kWin96: one form of marks_word each)
// from there to 516, kernels without the code for DAQ_DEBUG_CHECKS and odd decimations
// (kPlain) to 500.  With that, kPhaseAhead 6 instead of 5 takes it to 487 (4: 709, 7: 503;
// little noise 333 against 373, post = 64 504 against 565).  At 552, counting by 4 warps
// took 565.  The two jobs in turn by the same warps, two CTAs per SM: 635 at best.
#pragma once

#include "daq_twopass.cuh"

namespace daq {

constexpr int kPhaseTile = 448;    // samples per tile
constexpr int kPhaseAhead = 6;     // tiles of a CTA between a tile's count and the end of its compaction
constexpr unsigned kPhasePoll = 100;  // ns between reads of a chunk's words
constexpr int kPhaseInfo = kPhaseAhead + 1;     // tile records: one more is decoded ahead
constexpr int kPhaseXtal = 56;             // crystals it takes (a multiple of 4): four slots fit up to here
constexpr int kPhaseSum = 8;               // warps that sum
constexpr int kPhaseStage = 7;             // warps that stage rows
constexpr int kPhaseMarks = 2;             // warps that turn bits into marks, a tile each in turn
constexpr int kPhaseThreads = 32 * (kPhaseSum + kPhaseStage + kPhaseMarks + 3);
constexpr int kPhaseGather = 5;            // words a lane of the prefix warp reads: a chunk has at most 160 tiles

// Shared memory, in order.
template <int TW> struct PhaseSmem {
    size_t slot, slot_b, rows, trash, abyte, blocksum, sarr, recs, words, tinfo, prefix, fts, lens, bars, total;
    __host__ __device__ PhaseSmem(int X, int slot_bytes, int need_sarr)
    {
        auto up = [](size_t v, size_t n) { return (v + n - 1) / n * n; };
        slot = up(slot_bytes, 128);
        const size_t r = (size_t)(((TW * 2 * X + 32) + 15) & ~15);
        // (whole for any X: the staging warps read kPhaseXtal rows of a box)
        const size_t b = 2 * up((size_t)kPhaseXtal * 2 * (TW / 2), 128);
        slot_b = up(b > r ? b : r, 128);
        rows = 2 * slot;
        trash = rows + 2 * slot_b;
        abyte = trash + 128;
        blocksum = abyte + 128 * 2;
        sarr = blocksum + 4 * 2 * (TW / 8);
        recs = up(sarr + (need_sarr ? 4 * 2 * TW : 0), 16);
        words = recs + sizeof(TileRec) * kPhaseAhead;
        tinfo = up(words + kPhaseAhead * 4 * 6 * (TW / 32), 16);
        prefix = up(tinfo + sizeof(TileInfo) * kPhaseInfo, 16);
        fts = up(prefix + sizeof(Agg) * kPhaseAhead, 16);
        lens = fts + 8 * (kPlanSmem + 1);
        bars = up(lens + 4 * kPlanSmem, 16);
        total = up(bars + 8 * (10 + 3 * kPhaseAhead) + 16, 128);
    }
};

// A tile's published aggregate in one word (tiles of at most 511 samples): marked
// samples, island starts, trailing run, whether it continues a run; bit 31: there.
__device__ __forceinline__ uint32_t pack_agg(const Agg &g)
{
    return 0x80000000u | (uint32_t)g.m | ((uint32_t)g.s << 9) | ((uint32_t)g.tr << 18) | ((uint32_t)(g.full != 0) << 27);
}
__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_u32(uint32_t *p, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void sts_word(uint32_t at, uint32_t v)
{
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}

// Barrier of the staging warps that tells each whether any of them failed: a warp
// whose wait ran out still meets the others, and all stop together.
__device__ __forceinline__ bool phase_vote(bool failed)
{
    uint32_t any;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, 2, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(any)
        : "r"((uint32_t)failed), "n"(32 * kPhaseStage)
        : "memory");
    return any != 0;
}

template <int TW, int kWin, bool kPlain>
__global__ void __launch_bounds__(kPhaseThreads, 1) daq_phase_kernel(const __grid_constant__ KArgs a)
{
    constexpr int NWT = TW / 32, NBT = TW / 8, R = kPhaseAhead, RI = kPhaseInfo;
    constexpr int kBoxW = TW / 2;  // a tile is two boxes of this many columns
    static_assert(TW <= 64 * kPhaseStage && R >= 4, "a warp stages 64 columns");
    extern __shared__ __align__(128) unsigned char smem[];
    const PhaseSmem<TW> L(a.n_xtal, a.slot_bytes, a.need_sarr);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int X = a.n_xtal;
    uint8_t *abyte0 = smem + L.abyte;                                     // [2][128]
    int32_t *blocksum0 = reinterpret_cast<int32_t *>(smem + L.blocksum);  // [2][NBT]
    int32_t *sarr0 = reinterpret_cast<int32_t *>(smem + L.sarr);          // [2][TW]
    TileRec *recs0 = reinterpret_cast<TileRec *>(smem + L.recs);          // [R]
    auto words_of = [&](int k) {  // [R] marks, starts, ends and prefix counts of the CTA's tile k
        uint32_t *wm = reinterpret_cast<uint32_t *>(smem + L.words) + (k % R) * 6 * NWT;
        return TileWords{wm, wm + NWT, wm + 2 * NWT, reinterpret_cast<int32_t *>(wm + 3 * NWT),
                         reinterpret_cast<int32_t *>(wm + 4 * NWT), reinterpret_cast<int32_t *>(wm + 5 * NWT)};
    };
    TileInfo *tinfo0 = reinterpret_cast<TileInfo *>(smem + L.tinfo);  // [RI]
    Agg *prefix0 = reinterpret_cast<Agg *>(smem + L.prefix);          // [R]
    long long *fts_s = reinterpret_cast<long long *>(smem + L.fts);
    int32_t *lens_s = reinterpret_cast<int32_t *>(smem + L.lens);
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + L.bars);  // [2]: a tile to count has landed
    uint64_t *sums = full + 2;                                     // [2]: its bits and block sums are there
    uint64_t *mdone = sums + 2;                                    // [2]: they have been read
    uint64_t *fullb = mdone + 2;                                   // [2]: a tile to compact has landed
    uint64_t *staged = fullb + 2;                                  // [2]: its rows are in its place
    uint64_t *marked = staged + 2;                                 // [R]: tile k's marks and record are there
    uint64_t *placed = marked + R;                                 // [R]: its prefix is there
    uint64_t *gone = placed + R;                                   // [R]: its rows and records are written
    int *s_sent = reinterpret_cast<int *>(gone + R);               // [2]: loads issued for counts, for compactions

    for (int i = tid; i < 64; i += kPhaseThreads) reinterpret_cast<uint32_t *>(abyte0)[i] = 0u;
    if (tid == 0) {
        for (int r = 0; r < 2; ++r) {
            mbar_init(full + r, 1);
            mbar_init(sums + r, kPhaseSum);
            mbar_init(mdone + r, 1);
            mbar_init(fullb + r, 1);
            mbar_init(staged + r, kPhaseStage);
        }
        for (int r = 0; r < R; ++r) {
            mbar_init(marked + r, 1);
            mbar_init(placed + r, 1);
            mbar_init(gone + r, 1);
        }
        s_sent[0] = s_sent[1] = 0;
        fence_mbar_init();
    }
    const PlanView plan = cache_plan(a, fts_s, lens_s, tid, kPhaseThreads);
    __syncthreads();
    const long long total = plan.fts[a.n_fills];
    const int G = gridDim.x, cta = blockIdx.x;
    const int n_chunks = (int)((total + G - 1) / G);
    // this CTA's tiles are those of chunks 0 .. mine - 1
    const int mine = cta < total ? (int)((total - cta + G - 1) / G) : 0;
    auto tile_of = [&](int k) { return (long long)k * G + cta; };
    uint32_t *published = reinterpret_cast<uint32_t *>(a.status);  // zeroed by the prepare kernel
    auto par2 = [](int k) { return (uint32_t)(k >> 1) & 1u; };
    auto parR = [](int k) { return (uint32_t)(k / R) & 1u; };

    if (warp < kPhaseSum) {
        // ------------------------------------------------------------ sum
        const int n_steps = (a.ew + 63) / 64;
        bool ok = true;
        for (int k = 0; k < mine; ++k) {
            const int b = k & 1;
            ok = warp_wait_abortable(a, full + b, par2(k));
            if (ok && k >= 2) ok = warp_wait_abortable(a, mdone + b, par2(k - 2));
            if (!ok) break;
            const TileInfo T = tinfo0[k % RI];
            for (int it = warp; it < n_steps; it += kPhaseSum)
                sum_step_quarters<kPlain>(a, T, smem_addr(smem + b * L.slot), it, NBT, abyte0 + 128 * b, blocksum0 + NBT * b,
                                  sarr0 + (a.need_sarr ? TW * b : 0), lane);
            __syncwarp();
            if (lane == 0) mbar_arrive(sums + b);
        }
        if (!ok && lane == 0) set_status_bit(a, DAQ_DEV_TIMEOUT);
    } else if (warp < kPhaseSum + kPhaseStage) {
        // ------------------------------------------------------------ stage
        const int c = 64 * (warp - kPhaseSum) + 2 * lane;
        bool failed = false;
        const uint32_t flip = lane >= 16 ? 2u : 0u;
        for (int k = 0; k < mine; ++k) {
            const int s = k & 1;
            unsigned char *slot = smem + L.rows + s * L.slot_b;
            failed = !warp_wait_abortable(a, fullb + s, par2(k));
            const TileWords W = words_of(k);
            const int nt = failed ? 0 : (int)(tinfo0[k % RI].t_end - tinfo0[k % RI].t0);
            // the tile into registers: this lane's two columns of every crystal (past the
            // last crystal: whatever the slot holds there).  Lanes 16-31 keep every other
            // pair of pairs swapped, so that the rows' words, 54 words apart from lane to
            // lane, go to 32 banks.
            uint32_t w[kPhaseXtal], wl0, wl1;
            // columns without a marked sample are passed over (24 calorimeters of little
            // noise: 444 -> 414 us)
            const bool some = __any_sync(kFull, c < nt && ((W.m[c >> 5] >> (c & 31)) & 3u));
            if (some) {
                const int cc = c < nt ? c : 0;
                const uint32_t at = smem_addr(slot) + (uint32_t)((cc >= kBoxW ? a.box_stride_b : 0) + 2 * (cc >= kBoxW ? cc - kBoxW : cc));
                const uint32_t at0 = at + flip * 2 * kBoxW, at2 = at - flip * 2 * kBoxW;
#pragma unroll
                for (int x = 0; x < kPhaseXtal; ++x)
                    w[x] = lds_u32((x & 2 ? at2 : at0) + (uint32_t)(2 * kBoxW * x));
                wl0 = lds_u32(at + (uint32_t)(2 * kBoxW * (X - 2)));
                wl1 = lds_u32(at + (uint32_t)(2 * kBoxW * (X - 1)));
            }
            failed = failed || !warp_wait_abortable(a, placed + k % R, parR(k));
            const Agg ex = prefix0[k % R];
            if ((failed = phase_vote(failed))) break;  // every warp has read the slot
            const long long rb = 2ll * X;
            const int phase = (int)((ex.m * rb) & 15);
            if (some) {
                // a column that is not marked writes to a row of its own, past the slots: the stores need no condition
                const int wi = c >> 5, bit = c & 31;
                const uint32_t mw = c < nt ? W.m[wi] : 0u;
                const uint32_t m0 = (mw >> bit) & 1u, m1 = c + 1 < nt ? (mw >> (bit + 1)) & 1u : 0u;
                const uint32_t first_row = smem_addr(slot) + phase + (uint32_t)((c < nt ? W.mb[wi] : 0) + __popc(mw & ((1u << bit) - 1u))) * (uint32_t)rb;
                const uint32_t trash = smem_addr(smem + L.trash);
                const uint32_t row0 = m0 ? first_row : trash, row1 = m1 ? first_row + (m0 ? (uint32_t)rb : 0u) : trash;
                auto put = [&](uint32_t d0, uint32_t d1, int x, uint32_t lo, uint32_t hi) {  // crystals x, x + 1
                    sts_word(d0 + 2 * x, __byte_perm(lo, hi, 0x5410));
                    sts_word(d1 + 2 * x, __byte_perm(lo, hi, 0x7632));
                };
                const uint32_t a0 = row0 + 2 * flip, a1 = row1 + 2 * flip, b0 = row0 - 2 * flip, b1 = row1 - 2 * flip;
#pragma unroll
                for (int x = 0; x < kPhaseXtal; x += 4) {
                    if (x + 4 > X) break;
                    put(a0, a1, x, w[x], w[x + 1]);
                    put(b0, b1, x + 2, w[x + 2], w[x + 3]);
                }
                if (X & 2) put(row0, row1, X - 2, wl0, wl1);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(staged + s);
        }
        if (failed && lane == 0) set_status_bit(a, DAQ_DEV_TIMEOUT);
    } else if (warp < kPhaseSum + kPhaseStage + kPhaseMarks) {
        // ------------------------------------------------------------ marks, aggregate, Q bins
        const bool skip_q = (a.flags & DAQ_SKIP_Q) != 0;
        bool ok = true;
        for (int k = warp - kPhaseSum - kPhaseStage; k < mine; k += kPhaseMarks) {
            const int b = k & 1;
            if (!(ok = warp_wait_abortable(a, sums + b, par2(k)))) break;
            const TileInfo T = tinfo0[k % RI];
            unsigned edges;
            const uint32_t Mt = tile_marks<TW, kWin>(a, T, abyte0 + 128 * b, &edges, lane);
            const int nt = (int)(T.t_end - T.t0);
            const Agg agg = words_from_marks<TW>(Mt, edges & 1u, edges >> 1, nt, words_of(k), nullptr, lane);
            const uint32_t steps = marked_steps64<TW>(Mt, lane);
            if (lane == 0) {
                st_relaxed_u32(published + tile_of(k), pack_agg(agg));
                TileRec r;
                r.m = (int32_t)agg.m;
                r.s = (int32_t)agg.s;
                r.tr = (int32_t)agg.tr;
                r.flags = (agg.full ? 1 : 0) | (int)((edges & 1u) << 1) | (int)((edges >> 1) << 2) | (int)(steps << kRecStepShift);
                recs0[k % R] = r;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(marked + k % R);
            if (!skip_q) q_partial<kPlain>(a, T, blocksum0 + NBT * b, sarr0 + (a.need_sarr ? TW * b : 0), lane, 32);
            __syncwarp();
            if (lane == 0) mbar_arrive(mdone + b);
        }
        if (!ok && lane == 0) set_status_bit(a, DAQ_DEV_TIMEOUT);
    } else if (warp == kPhaseSum + kPhaseStage + kPhaseMarks) {
        // ------------------------------------------------------------ load: tiles to count
        bool ok = true;
        if (lane == 0 && mine > 0) decode_tile<TW>(a, tile_of(0), tinfo0[0], plan.fts, plan.lens);
        for (int k = 0; k < mine; ++k) {
            const int b = k & 1;
            if (k >= 2) ok = warp_wait_abortable(a, sums + b, par2(k - 2));
            if (ok && k >= R) ok = warp_wait_abortable(a, gone + k % R, parR(k - R));
            if (!ok) break;
            if (lane == 0) {
                fence_proxy_async_smem();
                mbar_arrive_expect_tx(full + b, tile_load_bytes(a));
                issue_tile_load(a, tinfo0[k % RI], smem + b * L.slot, full + b);
                s_sent[0] = k + 1;
                if (k + 1 < mine) decode_tile<TW>(a, tile_of(k + 1), tinfo0[(k + 1) % RI], plan.fts, plan.lens);
            }
            __syncwarp();
        }
        if (!ok && lane == 0) set_status_bit(a, DAQ_DEV_TIMEOUT);
    } else if (warp == kPhaseSum + kPhaseStage + kPhaseMarks + 1) {
        // ------------------------------------------------------------ out: rows and records; loads of tiles to compact
        bool ok = true;
        auto load = [&](int k) -> bool {  // the whole warp
            if (!warp_wait_abortable(a, marked + k % R, parR(k))) return false;
            if (lane == 0) {
                const int s = k & 1;
                const uint32_t steps = (uint32_t)recs0[k % R].flags >> kRecStepShift;
                uint32_t boxes = 0;
                for (int b = 0; b < a.nbox_b; ++b) {
                    const int s0 = (b * a.boxw_b) >> 6, s1 = ((b + 1) * a.boxw_b - 1) >> 6;
                    if (steps & ((s1 >= 31 ? 0xffffffffu : ((2u << s1) - 1u)) & ~((1u << s0) - 1u))) boxes |= 1u << b;
                }
                fence_proxy_async_smem();
                mbar_arrive_expect_tx(fullb + s, (uint32_t)__popc(boxes) * (uint32_t)X * (uint32_t)a.rs_b);
                issue_tile_load_b(a, tinfo0[k % RI], smem + L.rows + s * L.slot_b, fullb + s, boxes);
                s_sent[1] = k + 1;
            }
            __syncwarp();
            return true;
        };
        for (int k = 0; k < 2 && k < mine && ok; ++k) ok = load(k);
        for (int k = 0; ok && k < mine; ++k) {
            const int s = k & 1;
            if (!(ok = warp_wait_abortable(a, staged + s, par2(k)))) break;
            const Agg ex = prefix0[k % R];
            const TileInfo T = tinfo0[k % RI];
            const TileRec r = recs0[k % R];
            const int nt = (int)(T.t_end - T.t0);
            unsigned char *slot = smem + L.rows + s * L.slot_b;
            const long long rb = 2ll * X;
            const long long gs = ex.m * rb;
            const int phase = (int)(gs & 15);
            long long ge = gs + (long long)r.m * rb;
            if (!kPlain && (a.flags & DAQ_DEBUG_CHECKS) && (ex.m < 0 || r.m < 0 || r.m > nt)) {
                if (lane == 0) set_status_bit(a, DAQ_DEV_BAD_INDEX);
                ge = gs;
            }
            const long long cap_b = a.pool_cap * rb;
            if (ge > cap_b) {
                ge = cap_b;
                if (lane == 0) set_status_bit(a, DAQ_DEV_POOL_OVERFLOW);
            }
            if (ge > gs) {
                unsigned char *g = reinterpret_cast<unsigned char *>(a.pool);
                long long a16 = (gs + 15) & ~15ll, b16 = ge & ~15ll;
                if (a16 > ge) a16 = ge;
                if (b16 < a16) b16 = a16;
                if (lane == 0 && b16 > a16) {
                    fence_proxy_async_smem();
                    bulk_s2g_hint(g + a16, slot + phase + (a16 - gs), (uint32_t)(b16 - a16), l2_policy_evict_first());
                    bulk_commit();
                }
                const int n_head = (int)((a16 - gs) >> 1), n_tail = (int)((ge - b16) >> 1);
                if (lane < n_head)
                    *reinterpret_cast<uint16_t *>(g + gs + 2 * lane) = *reinterpret_cast<const uint16_t *>(slot + phase + 2 * lane);
                else if (lane >= 8 && lane < 8 + n_tail) {
                    const long long o = b16 + 2 * (lane - 8);
                    *reinterpret_cast<uint16_t *>(g + o) = *reinterpret_cast<const uint16_t *>(slot + phase + (o - gs));
                }
            }
            write_headers<TW, kPlain>(a, T, words_of(k), ex, lane);
            __syncwarp();
            if (lane == 0) {
                bulk_wait_read0();
                mbar_arrive(gone + k % R);
            }
            __syncwarp();
            if (k + 2 < mine) ok = load(k + 2);
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        if (!ok && lane == 0) set_status_bit(a, DAQ_DEV_TIMEOUT);
    } else {
        // ------------------------------------------------------------ prefix
        Agg carry = agg_identity();
        uint32_t v[kPhaseGather];  // aggregates of the chunk, tile 32 i + lane
        bool ok = true;
        for (int kp = 0; ok && kp < mine; ++kp) {
            const uint32_t *row = published + (long long)kp * G;
            const int there_are = (int)(total - (long long)kp * G < G ? total - (long long)kp * G : G);
#pragma unroll
            for (int i = 0; i < kPhaseGather; ++i) v[i] = 0u;
            // this CTA's own tile first: an entry of the ring is free by then
            if (!(ok = warp_wait_abortable(a, marked + kp % R, parR(kp)))) break;
            const uint64_t t0 = global_ns();
            for (uint32_t tries = 0;; ++tries) {
                bool missing = false;
#pragma unroll
                for (int i = 0; i < kPhaseGather; ++i) {
                    const int g = 32 * i + lane;
                    if (!v[i]) v[i] = g < there_are ? ld_relaxed_u32(row + g) : 0x88000000u;  // past the last tile: identity
                    missing |= !v[i];
                }
                if (!__any_sync(kFull, missing)) break;
                __nanosleep(kPhasePoll);
                if ((tries & 15u) == 15u) {
                    const bool late = lane == 0 && (global_ns() - t0 > a.wait_ns || aborted(a));
                    if (__any_sync(kFull, late)) {
                        ok = false;
                        break;
                    }
                }
            }
            if (!ok) break;
            // marked samples and starts add up; the run entering tile g is the trailing runs of the tiles
            // before it, back to the last that does not continue one
            unsigned m = 0, sn = 0, ma = 0, sa = 0, cut = 0, cuta = 0;  // of the tiles before this CTA's; of all
#pragma unroll
            for (int i = 0; i < kPhaseGather; ++i) {
                const int g = 32 * i + lane;
                const unsigned vm = v[i] & 511u, vs = (v[i] >> 9) & 511u;
                ma += vm;
                sa += vs;
                if (!((v[i] >> 27) & 1u)) cuta = g + 1;
                if (g < cta) {
                    m += vm;
                    sn += vs;
                    if (!((v[i] >> 27) & 1u)) cut = g + 1;
                }
            }
            m = __reduce_add_sync(kFull, m);
            sn = __reduce_add_sync(kFull, sn);
            cut = __reduce_max_sync(kFull, cut);
            unsigned tr = 0;
#pragma unroll
            for (int i = 0; i < kPhaseGather; ++i) {
                const unsigned g = 32 * i + lane, vt = (v[i] >> 18) & 511u;
                if (g + 1 >= cut && (int)g < cta) tr += vt;
            }
            tr = __reduce_add_sync(kFull, tr);
            if (lane == 0) {
                Agg place;
                place.m = carry.m + m;
                place.s = carry.s + sn;
                place.tr = tr + (cut ? 0 : carry.tr);
                place.full = 0;
                place.poison = 0;
                prefix0[kp % R] = place;
                mbar_arrive(placed + kp % R);
            }
            ma = __reduce_add_sync(kFull, ma);
            sa = __reduce_add_sync(kFull, sa);
            cuta = __reduce_max_sync(kFull, cuta);
            unsigned tra = 0;
#pragma unroll
            for (int i = 0; i < kPhaseGather; ++i) {
                const unsigned g = 32 * i + lane, vt = (v[i] >> 18) & 511u;
                if (g + 1 >= cuta) tra += vt;
            }
            tra = __reduce_add_sync(kFull, tra);
            carry.m += ma;
            carry.s += sa;
            carry.tr = tra + (cuta ? 0 : carry.tr);
            if (lane == 0 && kp == n_chunks - 1 && cta == 0) write_counts(a, total - 1, carry);  // CTA 0 has a tile of every chunk
            __syncwarp();
        }
        if (!ok && lane == 0) set_status_bit(a, DAQ_DEV_TIMEOUT);
    }
    // copies in flight land before the CTA may exit (a call that gave up)
    __syncthreads();
    if (tid == 0)
        for (int d = 0; d < 2; ++d)  // counts, compactions: the last two loads issued
            for (int k = s_sent[d] - 1; k >= 0 && k >= s_sent[d] - 2; --k)
                mbar_wait_bounded((d ? fullb : full) + (k & 1), par2(k), kWaitLimitNs);
}

}  // namespace daq
