// Lossless packing of pool rows on the GPU (Sec. 3: the frontend compresses
// island data losslessly before event building).  Stream format:
//   header   u32 magic 0x50514144, u32 n_xtal, u64 rows
//   offsets  u64[n_blocks + 1], n_blocks = ceil(rows / 32): byte offset of each
//            block's payload from the payload start (the last = payload size)
//   payload  block b = rows [32b, 32b + 32), the last block padded with copies
//            of the final row; per crystal x, with v_i the sample of row i:
//            z_0 = 0, z_i = zigzag(v_i - v_{i-1}) (2d for d >= 0, -2d - 1 else),
//            w = bit length of max z_i (0..17); words: (uint16)v_0 | w << 16,
//            then w bit planes, bit i of plane k = bit k of z_i.
// Consecutive pool rows are consecutive samples of an island, so the row to
// row differences of a crystal are small (noise, pulse edges) and a block's
// crystal column typically needs a few bits per sample instead of 16.
//
// The encoder is one pass over the pool (pack_kernel), the decoder one over the
// stream (unpack_kernel); in both a lane owns two crystal columns of a block.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "daq.h"
#include "daq_device.cuh"

namespace daq_pack {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxX = 64;
constexpr uint32_t kMagic = 0x50514144u;
constexpr uint64_t kWaitNs = 4000000000ull;  // a block copy not landed, or an earlier chunk not heard of, after this: give up
constexpr uint64_t kStartNs = 60000000000ull;  // no CTA has taken the next chunk after this: give up

// Copy block b's rows (16-byte vectors; the pool and every block start are
// 16-byte aligned) into the warp's shared rows, rows past the pool's end
// repeating its final row.  Returns the number of real rows.
__device__ __forceinline__ int load_block(const int16_t *pool, long long rows, int X, long long b, int16_t *sm,
                                          int lane)
{
    const long long r0 = 32ll * b;
    const int nv = (int)min(32ll, rows - r0);
    const int n = nv * X;  // int16 elements
    const int16_t *src = pool + r0 * X;
    const int nvec = n >> 3;
    for (int k = lane; k < nvec; k += 32) reinterpret_cast<int4 *>(sm)[k] = reinterpret_cast<const int4 *>(src)[k];
    for (int e = (nvec << 3) + lane; e < n; e += 32) sm[e] = src[e];
    __syncwarp();
    for (int e = n + lane; e < 32 * X; e += 32) sm[e] = sm[(nv - 1) * X + (e - n) % X];
    __syncwarp();
    return nv;
}

// ------------------------------------------------------------------ lanes on crystal columns
// Encoder and decoder give a lane two neighbouring crystal columns of a block:
// np = ceil(X / 2) lanes a block, nsub = 32 / np blocks side by side in a warp.
struct Lanes {
    int np, nsub;
    __host__ __device__ explicit Lanes(int X) : np((X + 1) / 2), nsub(32 / np < 16 ? 32 / np : 16) {}
};

// Bit k of byte j of word m -> bit m of byte j of word k (8 x 8 per byte).
__device__ __forceinline__ void swap_bits8(uint32_t (&p)[8])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t a = p[k], b = p[k + 4];
        p[k] = (a & 0x0f0f0f0fu) | ((b << 4) & 0xf0f0f0f0u);
        p[k + 4] = ((a >> 4) & 0x0f0f0f0fu) | (b & 0xf0f0f0f0u);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = (i & 1) + 4 * (i >> 1);
        const uint32_t a = p[k], b = p[k + 2];
        p[k] = (a & 0x33333333u) | ((b << 2) & 0xccccccccu);
        p[k + 2] = ((a >> 2) & 0x33333333u) | (b & 0xccccccccu);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = 2 * i;
        const uint32_t a = p[k], b = p[k + 1];
        p[k] = (a & 0x55555555u) | ((b << 1) & 0xaaaaaaaau);
        p[k + 1] = ((a >> 1) & 0x55555555u) | (b & 0xaaaaaaaau);
    }
}

// ------------------------------------------------------------------ encoder
// One pass over the pool.  A chunk is one round (nsub blocks) for each encoder
// warp of a CTA.  A warp turns its blocks into words staged in shared memory; the
// last warp of the chunk publishes the chunk's size.  One CTA, the first to run,
// reads the published sizes in order, as far as they are there, adds them up and
// writes each chunk's place over its size.  kEncDepth - 1 chunks later the warps
// write the staged words out at their place: the places come in order, so that
// every chunk waits for the slowest one before it, and the depth keeps that wait
// from the encoders.  Chunks go by ticket, so that whatever a chunk waits for is
// running or done.  (Two stages, and a warp that waited for one chunk's place
// before it took the next ticket: 1.33 ms.  Decoupled look-back, every chunk
// reading its predecessors' words: 1.4 ms with 304 chunks in flight, 2.7 with 760.)
// The two passes before (block sizes, then words, each reading the pool, and
// three scan kernels between) took 205 + 543 + 13 us for 12.06 M rows x 54, the
// second bound by issue: a 32 x 32 transpose across the warp for every four
// columns.  One pass takes 484 us; without the wait for places it would take 395,
// bound by issue (ALU pipe 67% busy, 16 warps an SM), and its bytes 276.
//
// A lane walks its two columns down the block's 32 rows, two samples to a word.
// Where a column's samples span at most 127, all its differences fit a byte, and
// the low bytes give them: four rows' bytes to a word, one bytewise subtraction
// a word, and the bit swaps of the decoder give the planes of the differences;
// the sign plane xor the others gives the zigzag planes, whose highest non-zero
// one is the width.  Where a column of the round is wider (pulses: 3% of the
// blocks of a dense fill, most of those early in a fill), all take 16-bit
// differences and the swaps on low and high bytes, with the differences' signs,
// which 16 bits may not hold, as a plane of their own.  (Every chunk waits for the
// slowest before it, so a slow round costs more than its share: with one column at a
// time for all wide ones the pass took 543 us, with every column of such a round
// sample by sample 646.)  The words' places within the block are
// one scan over the lanes.
//
// A round of noise takes some 6 words a column, one of wide columns up to 18.  The
// staged words of a warp are a ring that holds six of the first or two of the last: a
// round begins at the next free unit, and the oldest rounds are written out early where
// there is no piece for what the last round took.  2 M rows x 54, us for noise of
// sigma 3 / 8 / 24 and for full-range samples: 90 / 91 / 152 / 169.  (Six stages of
// seven words a column, rounds that did not fit encoded a second time from rows read
// again, and one column at a time for differences past 16 bits: 90 / 164 / 295 / 1707;
// the three kernels before: 164 / 164 / 217 / 243.  Emptying the ring and changing the
// stages' size: 350 at sigma 7, where every other round needs it.)
constexpr int kEncWarps = 8;
constexpr int kEncThreads = 32 * kEncWarps;
constexpr int kEncDepth = 6;  // rounds of a warp that are encoded or written out
constexpr int kEncWarpBytes = 14336;  // shared memory of a warp with which two CTAs share an SM
constexpr int kEncUnits = 12;  // units of the ring of staged words
constexpr int kEncRing = 16;  // chunks whose tickets and sizes a CTA remembers: at least 2 kEncDepth + 3

// Shared memory of one encoder warp: a ring of encoded words, a round's rows, where in
// the ring the rounds lie, and the rows' barrier.
struct EncPlan : Lanes {
    int unit, inb;  // words of a unit of the ring, bytes of a round's rows
    // Units of four words a column (two hold a column of 7 planes, five any), or of as
    // many from three and a half on as let two CTAs share an SM; where none do, four again.
    __host__ __device__ explicit EncPlan(int X) : Lanes(X)
    {
        const int cols = nsub * X, least = (7 * cols + 1) / 2;
        inb = 64 * cols;
        const int fit = (kEncWarpBytes - inb - 4 * kEncDepth * (1 + nsub) - 48) / (4 * kEncUnits);
        unit = fit < least || fit > 4 * cols ? 4 * cols : fit;
    }
    __host__ __device__ size_t rows_at() const { return (4 * (size_t)kEncUnits * unit + 15) & ~size_t(15); }
    __host__ __device__ size_t meta_at() const { return rows_at() + (size_t)inb; }
    __host__ __device__ size_t bar_at() const { return meta_at() + 4 * (size_t)kEncDepth * (1 + nsub); }
    __host__ __device__ size_t bytes() const { return ((bar_at() + 15) & ~size_t(15)) + 16; }
    __host__ __device__ long long chunk_blocks() const { return (long long)kEncWarps * nsub; }
};

// What the warps of a CTA tell each other.
struct EncShared {
    long long tk[kEncRing];               // chunk of the CTA's i-th turn
    unsigned words[kEncRing][kEncWarps];  // words of each warp's round in it
    unsigned done[kEncRing];              // warps that have encoded it (counted on from turn to turn)
    int posted;                           // the last turn whose ticket is known
    int fail, scans;
};

constexpr unsigned kAgg = 1, kIncl = 2, kGaveUp = 3;

__device__ __forceinline__ unsigned add_acq_rel_cta(unsigned *p, unsigned v)
{
    unsigned old;
    asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(daq::smem_addr(p)), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ int ld_acquire_cta(const int *p)
{
    int v;
    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(daq::smem_addr(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_cta(int *p, int v)
{
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(daq::smem_addr(p)), "r"(v) : "memory");
}

// The scanning CTA: turns the published sizes of chunks 0, 1, ... into places.
// Each round reads the next 2 kEncThreads words and takes those before the first
// that is not there yet.  Returns the payload's words, -1 when it gave up: the
// chunks that had not got a place are then told so.  A chunk that no CTA has taken
// (`tickets`: chunks taken) is not late: other work may hold all SMs but this CTA's.
__device__ long long enc_places(unsigned long long *st, long long n_chunks, const unsigned long long *tickets)
{
    __shared__ unsigned s_sum[kEncWarps], s_miss[kEncWarps];
    __shared__ int s_stop;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    long long done = 0, at = 0;
    uint64_t t0 = daq::global_ns(), t_last = t0;  // of the next chunk's wait, of the last chunk placed
    if (tid == 0) s_stop = 0;
    __syncthreads();
    while (done < n_chunks) {
        unsigned long long v[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const long long c = done + 2 * tid + j;
            v[j] = c < n_chunks ? daq::ld_relaxed_u64(st + c) : 0ull;
        }
        if ((v[0] & 3u) == kGaveUp || (v[1] & 3u) == kGaveUp) s_stop = 1;
        const unsigned a = (v[0] & 3u) ? (unsigned)(v[0] >> 2) : 0u, b = (v[1] & 3u) ? (unsigned)(v[1] >> 2) : 0u;
        const unsigned miss = __reduce_min_sync(kFull, !(v[0] & 3u) ? 2u * tid : !(v[1] & 3u) ? 2u * tid + 1 : 2u * kEncThreads);
        unsigned incl = a + b;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane == 31) s_sum[warp] = incl;
        if (lane == 0) s_miss[warp] = miss;
        __syncthreads();
        unsigned first = 2 * kEncThreads, ahead = 0;
        for (int w = 0; w < kEncWarps; ++w) {
            first = min(first, s_miss[w]);
            if (w < warp) ahead += s_sum[w];
        }
        const uint64_t now = daq::global_ns();
        if (first > 0) t0 = t_last = now;
        if (tid == 0 && now - t0 > kWaitNs / 2) {
            if (daq::ld_relaxed_u64(tickets) <= (unsigned long long)done) t0 = now;
            if (now - t0 > kWaitNs || now - t_last > kStartNs) s_stop = 1;
        }
        // words before this thread's pair; of them only those before `first` count, and every pair before it is whole
        const long long mine = at + ahead + incl - a - b;
        if (2 * tid < (int)first) daq::st_relaxed_u64(st + done + 2 * tid, ((unsigned long long)mine << 2) | kIncl);
        if (2 * tid + 1 < (int)first)
            daq::st_relaxed_u64(st + done + 2 * tid + 1, ((unsigned long long)(mine + a) << 2) | kIncl);
        __shared__ long long s_next;
        if (first > 0 && (unsigned)tid == (first - 1) / 2) s_next = mine + a + ((first & 1) ? 0u : b);
        __syncthreads();
        if (s_stop) {
            for (long long c = done + tid; c < n_chunks; c += kEncThreads) daq::st_relaxed_u64(st + c, kGaveUp);
            return -1;
        }
        if (first > 0) at = s_next;
        done += first;
        __syncthreads();
    }
    return at;
}

// a - b in every byte, modulo 256.
__device__ __forceinline__ uint32_t sub8x4(uint32_t a, uint32_t b)
{
    return ((a | 0x80808080u) - (b & 0x7f7f7f7fu)) ^ ((a ^ ~b) & 0x80808080u);
}

// The zigzag planes of one column from its samples' low bytes (word k, byte j =
// row 8j + k), in place; returns the width.  All differences fit a byte.
__device__ __forceinline__ int byte_planes(uint32_t (&p)[8])
{
    const uint32_t first = __byte_perm(p[7], p[0], 0x2104);  // rows -1 (row 0 itself), 7, 15, 23
#pragma unroll
    for (int k = 7; k > 0; --k) p[k] = sub8x4(p[k], p[k - 1]);
    p[0] = sub8x4(p[0], first);
    swap_bits8(p);
    const uint32_t sign = p[7];
#pragma unroll
    for (int k = 7; k > 0; --k) p[k] = p[k - 1] ^ sign;
    p[0] = sign;
    int w = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) w = p[k] ? k + 1 : w;
    return w;
}

// Per 16-bit half, modulo 2^16: v - p (no borrow crosses the halves).
__device__ __forceinline__ uint32_t sub16x2(uint32_t v, uint32_t p)
{
    return ((v | 0x80008000u) - (p & 0x7fff7fffu)) ^ ((v ^ ~p) & 0x80008000u);
}

// The zigzag planes of one column from the low and high bytes of its differences
// modulo 2^16 and their signs: planes 0..7 in lo, 8..15 in hi, 16 in sign; returns the
// width.
__device__ __forceinline__ int word_planes(uint32_t (&lo)[8], uint32_t (&hi)[8], uint32_t &sign)
{
    swap_bits8(lo);
    swap_bits8(hi);
    const uint32_t s = sign;
    sign ^= hi[7];
#pragma unroll
    for (int k = 7; k > 0; --k) hi[k] = hi[k - 1] ^ s;
    hi[0] = lo[7] ^ s;
#pragma unroll
    for (int k = 7; k > 0; --k) lo[k] = lo[k - 1] ^ s;
    lo[0] = s;
    int w = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) w = lo[k] ? k + 1 : w;
#pragma unroll
    for (int k = 0; k < 8; ++k) w = hi[k] ? k + 9 : w;
    return sign ? 17 : w;
}

// Encode `blocks` <= nsub blocks side by side from the rows at `in` (block pitch
// 32 X): what a lane has of them.
template <bool kEven> struct Round {
    int sub, pr;       // the lane's block and its pair of columns in it
    bool mine, two;    // the lane has columns, has two
    const int16_t *col;
    int X;
    __device__ __forceinline__ Round(const EncPlan &pl, int X_, const int16_t *in, int blocks, int lane)
        : sub(lane / pl.np), pr(lane - sub * pl.np), mine(sub < blocks), two(mine && 2 * pr + 1 < X_),
          col(in + (mine ? sub * 32 * X_ + 2 * pr : 0)), X(X_)
    {
    }
    __device__ __forceinline__ uint32_t row(int r) const  // both samples of row r
    {
        if (kEven) return *reinterpret_cast<const uint32_t *>(col + r * X);
        return (uint32_t)(uint16_t)col[r * X] | (two ? (uint32_t)(uint16_t)col[r * X + 1] << 16 : 0u);
    }
    // the lane's words, their place in the round (returned) and the round's
    // total; `before`: the words ahead of the lane's block
    __device__ __forceinline__ int place(const EncPlan &pl, int w0, int w1, int lane, int &total, int &before) const
    {
        const int words = mine ? 1 + w0 + (two ? 1 + w1 : 0) : 0;
        int incl = words;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, d);
            if (lane >= d) incl += y;
        }
        total = __shfl_sync(kFull, incl, 31);
        before = __shfl_sync(kFull, incl - words, mine ? sub * pl.np : 0);
        return incl - words;
    }
};

// The head word and planes 0 .. 7 of a column.
__device__ __forceinline__ void store_column(uint32_t *dst, uint32_t first, int w, const uint32_t (&p)[8])
{
    dst[0] = first | ((uint32_t)w << 16);
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (k < w) dst[1 + k] = p[k];
}

// A round with a column that is not narrow.  A function of its own: with both
// forms in one body the narrow one ran 2.3x slower.  Returns the words of the
// round, kWideRound if a column has more than 8 planes, and the words ahead of the
// lane's block.
constexpr int kWideRound = 1 << 30;
template <bool kEven>
__device__ __noinline__ int2 encode_wide_round(int X, const int16_t *in, int blocks, uint32_t *dst, int fit)
{
    const int lane = threadIdx.x & 31;
    const EncPlan pl(X);
    const Round<kEven> R(pl, X, in, blocks, lane);
    uint32_t p0[8], p1[8], h0[8], h1[8], s0 = 0, s1 = 0, prev[4];
    const uint32_t v0 = R.row(0);
#pragma unroll
    for (int j = 0; j < 4; ++j) prev[j] = j ? R.row(8 * j - 1) : v0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        uint32_t d[4], sg[4];  // rows k, k + 8, ..., both columns: differences modulo 2^16, their signs (bits 15 and 31)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t v = R.row(8 * j + k);
            d[j] = sub16x2(v, prev[j]);
            sg[j] = d[j] ^ ((v ^ prev[j]) & (v ^ d[j]));
            prev[j] = v;
        }
        const uint32_t t = __byte_perm(d[0], d[1], 0x6240), u = __byte_perm(d[2], d[3], 0x6240);
        const uint32_t th = __byte_perm(d[0], d[1], 0x7351), uh = __byte_perm(d[2], d[3], 0x7351);
        const uint32_t ts = __byte_perm(sg[0], sg[1], 0x7351), us = __byte_perm(sg[2], sg[3], 0x7351);
        p0[k] = __byte_perm(t, u, 0x5410);
        p1[k] = __byte_perm(t, u, 0x7632);
        h0[k] = __byte_perm(th, uh, 0x5410);
        h1[k] = __byte_perm(th, uh, 0x7632);
        s0 |= (__byte_perm(ts, us, 0x5410) >> (7 - k)) & (0x01010101u << k);
        s1 |= (__byte_perm(ts, us, 0x7632) >> (7 - k)) & (0x01010101u << k);
    }
    const int w0 = word_planes(p0, h0, s0), w1 = word_planes(p1, h1, s1);
    int total, before;
    const int o0 = R.place(pl, w0, w1, lane, total, before);
    const int ret = total | (__any_sync(kFull, R.mine && max(w0, w1) > 8) ? kWideRound : 0);
    if (total > fit) return make_int2(ret, before);
    auto store = [&](uint32_t *at, uint32_t first, int w, const uint32_t (&p)[8], const uint32_t (&h)[8], uint32_t top) {
        store_column(at, first, w, p);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (8 + k < w) at[9 + k] = h[k];
        if (w > 16) at[17] = top;
    };
    if (R.mine) store(dst + o0, v0 & 0xffffu, w0, p0, h0, s0);
    if (R.two) store(dst + o0 + 1 + w0, v0 >> 16, w1, p1, h1, s1);
    return make_int2(ret, before);
}

// Encode a round.  The words go to dst when all of them fit `fit` words.  Returns the
// words of the round; `before` gets those ahead of the lane's block.  `wide`: rounds in
// a row with columns of more than 8 planes; after two the narrow form is not tried
// first (3.03 M rows x 33, sigma 60: 238 -> 218 us).
template <bool kEven>
__device__ __forceinline__ int encode_round(const EncPlan &pl, int X, const int16_t *in, int blocks, uint32_t *dst, int fit,
                                            int lane, int &before, int &wide)
{
    if (wide >= 2) {
        const int2 r = encode_wide_round<kEven>(X, in, blocks, dst, fit);
        before = r.y;
        wide = r.x & kWideRound ? 2 : 0;
        return r.x & ~kWideRound;
    }
    const Round<kEven> R(pl, X, in, blocks, lane);
    uint32_t p0[8], p1[8];
    const uint32_t v0 = R.row(0);
    uint32_t mx = v0, mn = v0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t a = R.row(k), b = R.row(k + 8), c = R.row(k + 16), d = R.row(k + 24);
        mx = __vimax3_s16x2(__vimax3_s16x2(mx, a, b), c, d);
        mn = __vimin3_s16x2(__vimin3_s16x2(mn, a, b), c, d);
        const uint32_t t = __byte_perm(a, b, 0x6240), u = __byte_perm(c, d, 0x6240);  // low bytes of both columns
        p0[k] = __byte_perm(t, u, 0x5410);
        p1[k] = __byte_perm(t, u, 0x7632);
    }
    const int span0 = (int)(int16_t)(mx & 0xffffu) - (int)(int16_t)(mn & 0xffffu);
    const int span1 = ((int)mx >> 16) - ((int)mn >> 16);
    if (__any_sync(kFull, R.mine && max(span0, span1) > 127)) {
        const int2 r = encode_wide_round<kEven>(X, in, blocks, dst, fit);
        before = r.y;
        wide = r.x & kWideRound ? wide + 1 : 0;
        return r.x & ~kWideRound;
    }
    wide = 0;
    const int w0 = byte_planes(p0), w1 = byte_planes(p1);
    int total;
    const int o0 = R.place(pl, w0, w1, lane, total, before);
    if (total > fit) return total;
    if (R.mine) store_column(dst + o0, v0 & 0xffffu, w0, p0);
    if (R.two) store_column(dst + o0 + 1 + w0, v0 >> 16, w1, p1);
    return total;
}

// status: one word a chunk, zeroed, then the ticket and the role counter.  A row
// copy that does not land, or a wait that runs out, makes the chunk and every
// later one give up: *out_bytes is -1.
template <bool kEven>
__global__ void __launch_bounds__(kEncThreads, 2) pack_kernel(const int16_t *pool, long long rows, int X, long long nb,
                                                              unsigned long long *status, long long n_chunks,
                                                              unsigned char *out, long long cap, long long *out_bytes)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ EncShared sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const EncPlan pl(X);
    uint32_t *out32 = reinterpret_cast<uint32_t *>(out);
    unsigned long long *table = reinterpret_cast<unsigned long long *>(out + 16);
    const long long head = 16 + 8 * (nb + 1);
    unsigned long long *tickets = status + n_chunks;
    auto entry = [&](long long b, long long words) {  // the offset of block b
        if (16 + 8 * b + 8 <= cap) table[b] = 4ull * (unsigned long long)words;
    };
    if (threadIdx.x == 0) {
        sh.scans = atomicAdd(tickets + 1, 1ull) == 0ull;  // the first CTA to run
        sh.fail = 0;
        sh.posted = 0;
        for (int k = 0; k < kEncRing; ++k) sh.done[k] = 0;
        if (!sh.scans) sh.tk[0] = (long long)atomicAdd(tickets, 1ull);
    }
    __syncthreads();
    if (sh.scans) {
        if (threadIdx.x == 0 && cap >= 16) {
            out32[0] = kMagic;
            out32[1] = (uint32_t)X;
            reinterpret_cast<unsigned long long *>(out)[1] = (unsigned long long)rows;
        }
        const long long words = enc_places(status, n_chunks, tickets);
        if (threadIdx.x == 0) {
            if (words >= 0) entry(nb, words);
            *out_bytes = words >= 0 ? head + 4 * words : -1ll;
        }
        return;
    }

    unsigned char *base = dsm + warp * pl.bytes();
    uint32_t *ring = reinterpret_cast<uint32_t *>(base);
    int16_t *in = reinterpret_cast<int16_t *>(base + pl.rows_at());
    // per round: words, then those ahead of each block
    auto meta = [&](int j) { return reinterpret_cast<int *>(base + pl.meta_at()) + (j % kEncDepth) * (1 + pl.nsub); };
    uint64_t *bar = reinterpret_cast<uint64_t *>(base + pl.bytes() - 16);
    if (lane == 0) {
        daq::mbar_init(bar, 1);
        daq::fence_mbar_init();
    }
    __syncwarp();
    const long long nfull = rows / 32, cb = pl.chunk_blocks();
    const int sub = lane / pl.np;
    auto block_of = [&](long long c) { return c * cb + (long long)warp * pl.nsub; };  // this warp's first block of chunk c
    auto blocks_at = [&](long long b) { return (int)max(0ll, min((long long)pl.nsub, nb - b)); };
    auto gave_up = [&] { *reinterpret_cast<volatile int *>(&sh.fail) = 1; };
    bool copying = false;  // a copy of the next round's rows is in flight
    uint32_t phase = 0;    // that its wait expects
    auto start_rows = [&](long long c) {
        const long long b = block_of(c);
        const int n = blocks_at(b);
        if (c >= n_chunks || n == 0 || b + n > nfull) return;  // the last, shorter block comes in by plain loads
        copying = true;
        if (lane == 0) {
            daq::fence_proxy_async_smem();
            daq::mbar_arrive_expect_tx(bar, (uint32_t)(n * 64 * X));
            daq::bulk_g2s(in, pool + 32 * b * X, (uint32_t)(n * 64 * X), bar);
        }
    };
    // write turn j out, whose words begin at `unit` of the ring; v: what was read of its place (lane 0)
    auto finish = [&](int j, int unit, unsigned long long v) {
        const long long c = sh.tk[j % kEncRing];
        long long at = -1;
        if (lane == 0) {
            const uint64_t t0 = daq::global_ns();
            while ((v & 3u) < kIncl && !*reinterpret_cast<volatile int *>(&sh.fail)) {
                v = daq::ld_relaxed_u64(status + c);
                if (daq::global_ns() - t0 > 2 * kWaitNs) gave_up();
            }
            if ((v & 3u) == kIncl) at = (long long)(v >> 2);
            else gave_up();
            (void)add_acq_rel_cta(&sh.done[j % kEncRing], 0u);  // the warps' words have been seen
        }
        at = __shfl_sync(kFull, at, 0);
        if (at < 0) return;
        for (int w = 0; w < warp; ++w) at += sh.words[j % kEncRing][w];
        const int *m = meta(j);
        const long long b = block_of(c);
        const int n = blocks_at(b);
        if (lane == sub * pl.np && sub < n) entry(b + sub, at + m[1 + sub]);
        const int room = (int)(max(0ll, min(cap - (head + 4 * at), 1ll << 30)) >> 2);
        uint32_t *dst = out32 + (head >> 2) + at;
        const uint32_t *src = ring + unit * pl.unit;
        const int last = min(m[0], room);
#pragma unroll 4
        for (int k = lane; k < last; k += 32) dst[k] = src[k];
        __syncwarp();
    };
    long long c = sh.tk[0];
    start_rows(c);
    int i = 0, done = 0;                 // turns encoded, written out
    int wide = 0;
    int at = 0, units = kEncUnits;       // a free piece of the ring, for turn i
    int end = 0, want = 1;               // unit after the last round's words, units expected of the next round
    unsigned starts = 0;                 // the unit each of the last rounds begins at, four bits a round
    const unsigned unit_mul = ((1u << 20) + pl.unit - 1) / pl.unit;  // words (< 1,500) to units
    auto start_of = [&](int j) { return (int)((starts >> (4 * (i - 1 - j))) & 15u); };
    // The ring holds turns done .. i - 1 in order, each in one piece.  Is there a piece for turn i?
    auto piece = [&]() -> bool {
        at = 0;
        units = kEncUnits;
        if (done == i) return true;
        const int first = start_of(done);
        at = end;
        units = (end > first ? kEncUnits : first) - end;
        if (units < want && end > first) {
            at = 0;
            units = first;
        }
        return units >= want;
    };
    while (c < n_chunks) {
        unsigned long long ticket = 0, place = 0;
        if (threadIdx.x == 0) ticket = atomicAdd(tickets, 1ull);  // of turn i + 1, used once this one is encoded
        if (lane == 0 && i - done == kEncDepth - 1) place = daq::ld_relaxed_u64(status + sh.tk[done % kEncRing]);
        const long long b = block_of(c);
        const int n = blocks_at(b);
        if (copying) {
            const bool ok = daq::mbar_wait_bounded(bar, phase, kWaitNs);
            phase ^= 1u;
            copying = false;
            if (__any_sync(kFull, !ok) && lane == 0) gave_up();
        } else {
            for (int k = 0; k < n; ++k) load_block(pool, rows, X, b + k, in + k * 32 * X, lane);
        }
        while (!piece()) {
            finish(done, start_of(done), 0ull);
            ++done;
        }
        int before;
        const int words = encode_round<kEven>(pl, X, in, n, ring + at * pl.unit, units * pl.unit, lane, before, wide);
        want = (int)(((unsigned)(words + pl.unit - 1) * unit_mul) >> 20);  // of the next round too: mostly as long
        if (want > units) {  // longer than the round before: again, once there is a piece for it
            while (!piece()) {
                finish(done, start_of(done), 0ull);
                ++done;
            }
            before = encode_wide_round<kEven>(X, in, n, ring + at * pl.unit, units * pl.unit).y;
        }
        end = at + want;
        starts = starts << 4 | (unsigned)at;
        int *m = meta(i);
        if (lane == sub * pl.np && sub < pl.nsub) m[1 + sub] = before;
        if (lane == 0) {
            m[0] = words;
            sh.words[i % kEncRing][warp] = (unsigned)words;
            if (warp == 0) {
                sh.tk[(i + 1) % kEncRing] = (long long)ticket;
                st_release_cta(&sh.posted, i + 1);
            }
            const unsigned turn = (unsigned)kEncWarps * (unsigned)(i / kEncRing + 1);
            if (add_acq_rel_cta(&sh.done[i % kEncRing], 1u) + 1u == turn) {  // the chunk's last warp
                unsigned total = 0;
                for (int w = 0; w < kEncWarps; ++w) total += sh.words[i % kEncRing][w];
                const bool bad = *reinterpret_cast<volatile int *>(&sh.fail);
                daq::st_relaxed_u64(status + c, bad ? (unsigned long long)kGaveUp : ((unsigned long long)total << 2) | kAgg);
            }
            const uint64_t t0 = daq::global_ns();
            while (ld_acquire_cta(&sh.posted) < i + 1)  // warp 0 has encoded this turn
                if (daq::global_ns() - t0 > 3 * kWaitNs) {
                    gave_up();
                    break;
                }
        }
        __syncwarp();
        c = sh.tk[++i % kEncRing];
        start_rows(c);
        if (i - done == kEncDepth) {
            finish(done, start_of(done), place);
            ++done;
        }
    }
    while (done < i) {
        finish(done, start_of(done), 0ull);
        ++done;
    }
}

// ------------------------------------------------------------------ decoder
// Bound by instruction issue and, at the end, by HBM (61% of its rate).  Lanes
// own crystal columns, two neighbouring ones each (np = ceil(X / 2) lanes a
// block, nsub = 32 / np blocks side by side), so a column's bit planes become
// samples inside one lane: seven three-input operations undo the zigzag on the
// planes, three stages of bit swaps among eight words (48 operations) turn
// them into 32 signed bytes (word k, byte j = row 8j + k), and one dp4a a row
// takes its byte and adds it to the running sample.  A row is one 32-bit store
// of the lane's two samples; whole blocks leave by bulk copy.  With lanes on
// rows a column took a 32 x 32 transpose and a prefix sum across the warp, 49
// instructions a column and warp against 12 here: 12.06 M rows x 54 decoded in
// 1.19 ms, now 0.34 (the call 1275 -> 383 us).
// Where the columns' words begin is known only by walking their head words, a
// chain of X shared-memory loads, so a warp stages the payload of up to G = 4
// consecutive blocks (16-byte asynchronous copies) and G lanes walk them at
// once; more would cost occupancy (10 KB a warp, 20 warps an SM).  The next
// group's payload is brought into L2 while this one is decoded (390 -> 383
// us).  Undoing the zigzag on bytes after the swaps, copying rows out with
// 16-byte stores and checking every head word in the walk took 502 us.
// Where one of a warp's columns is wider than 8 bits (pulses: 2% of the blocks of a
// dense fill hold some) all take the same way with 16-bit differences, low and high
// bytes: 2 M rows x 54 take 62 us at sigma 3, 86 at 24, 102 at 60, 132 full-range.
// (Such columns done again one at a time by the whole warp, lanes on rows: 62, 80, 585
// and 808; lanes on rows throughout: 206, 500, 510 and 549.  That loop kept for up to
// three columns: 64 at sigma 3, 82 at 24.  The wide form as a function: 63 and 86, and
// 6% more than this for odd crystal counts, whose registers the call spills.)
constexpr int kDecWarps = 4;
constexpr int kDecThreads = 32 * kDecWarps;

// Lanes, blocks and shared memory of one warp, by the crystal count.
struct DecPlan : Lanes {
    int G, cap;  // blocks staged at once, bytes of staged payload
    __host__ __device__ explicit DecPlan(int X) : Lanes(X)
    {
        G = nsub >= 4 ? nsub : nsub == 3 ? 6 : 4;
        // planes of 6.5 bits a column; one block of the widest columns always fits
        const int want = G * X * 30, least = X * 72;
        cap = ((want > least ? want : least) + 15) & ~15;
    }
    __host__ __device__ size_t pos_at() const { return (size_t)cap + 32; }  // staged words begin at any 4-byte phase
    __host__ __device__ size_t out_at(int X) const { return (pos_at() + 2 * (size_t)G * X + 15) & ~size_t(15); }
    __host__ __device__ size_t bytes(int X) const { return out_at(X) + (size_t)nsub * 64 * X; }
};

// The differences of a column of width w <= 8 as signed bytes: its zigzag
// codes' sign plane is plane 0, and bit k of the difference is plane k + 1
// xor the sign, so seven three-input operations on the planes undo the zigzag
// of 32 samples.  Words read past the column's planes are masked away.
__device__ __forceinline__ void column_steps(const uint32_t *h, int w, uint32_t (&p)[8])
{
    const uint32_t sign = h[1] & (uint32_t)(-w >> 31);
#pragma unroll
    for (int k = 0; k < 7; ++k) p[k] = (h[2 + k] & (uint32_t)((k + 1 - w) >> 31)) ^ sign;
    p[7] = sign;
    swap_bits8(p);
}

// The rows of a lane's two columns (head words at words + at0 and + at1, negative: it
// has none) where one of the warp's is wider than 8 bits: the differences modulo 2^16,
// as low and high bytes.  Their planes are planes 1 .. 16 of the codes, each xor the sign; a
// sample is 16 bits too, so that the carry past them is of no account.
template <bool kEven>
__device__ __forceinline__ void decode_wide(const uint32_t *words, int at0, int at1, int16_t *o, int X)
{
    const bool mine = at0 >= 0, two = at1 >= 0;
    const uint32_t *h0 = words + max(at0, 0), *h1 = words + max(at1, 0);
    uint32_t a0 = mine ? h0[0] : 0u, a1 = two ? h1[0] : 0u, b0 = 0, b1 = 0;  // sample = a + 256 b, modulo 2^16
    auto steps = [](const uint32_t *h, int w, uint32_t (&lo)[8], uint32_t (&hi)[8]) {
        const uint32_t sign = h[1] & (uint32_t)(-w >> 31);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            lo[k] = (h[2 + k] & (uint32_t)((k + 1 - w) >> 31)) ^ sign;
            hi[k] = (h[10 + k] & (uint32_t)((k + 9 - w) >> 31)) ^ sign;
        }
        swap_bits8(lo);
        swap_bits8(hi);
    };
    uint32_t lo0[8], hi0[8], lo1[8], hi1[8];
    steps(h0, (int)(a0 >> 16), lo0, hi0);
    steps(h1, (int)(a1 >> 16), lo1, hi1);
    if (!mine) return;
#pragma unroll
    for (int q = 0; q < 32; ++q) {
        const int k = q & 7, j = q >> 3;
        if (q) {
            a0 = __dp4a(lo0[k], 1u << (8 * j), a0);
            b0 = __dp4a(hi0[k], 1u << (8 * j), b0);
            a1 = __dp4a(lo1[k], 1u << (8 * j), a1);
            b1 = __dp4a(hi1[k], 1u << (8 * j), b1);
        }
        const uint32_t s0 = a0 + (b0 << 8), s1 = a1 + (b1 << 8);
        if (kEven) {
            *reinterpret_cast<uint32_t *>(o + q * X) = __byte_perm(s0, s1, 0x5410);
        } else {
            o[q * X] = (int16_t)s0;
            if (two) o[q * X + 1] = (int16_t)s1;
        }
    }
}

template <bool kEven>
__global__ void __launch_bounds__(kDecThreads, 5) unpack_kernel(const unsigned char *in, long long in_bytes, long long rows,
                                                             int X, long long nb, int16_t *pool_out, int *err)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const DecPlan pl(X);
    unsigned char *base = dsm + warp * pl.bytes(X);
    uint16_t *pos = reinterpret_cast<uint16_t *>(base + pl.pos_at());  // [G][X] word of each column's head
    int16_t *out = reinterpret_cast<int16_t *>(base + pl.out_at(X));   // [nsub][32][X]
    const long long head = 16 + 8 * (nb + 1);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const uint32_t *h = reinterpret_cast<const uint32_t *>(in);
        if (h[0] != kMagic || h[1] != (uint32_t)X || reinterpret_cast<const unsigned long long *>(in)[1] !=
                                                             (unsigned long long)rows)
            atomicOr(err, 1);
    }
    if (head > in_bytes) {  // the offsets table itself is cut short
        if (threadIdx.x == 0 && nb > 0) atomicOr(err, 2);
        return;
    }
    const unsigned long long *offs = reinterpret_cast<const unsigned long long *>(in + 16);
    const unsigned long long plen = (unsigned long long)(in_bytes - head);  // payload bytes there are
    const unsigned long long most = 72ull * X;                              // of one block
    const bool vec_out = (reinterpret_cast<uintptr_t>(pool_out) & 15) == 0;  // then every block is 16-byte aligned
    const int sub = lane / pl.np, pr = lane - sub * pl.np;
    const long long step = (long long)gridDim.x * kDecWarps * pl.G;
    long long b0 = ((long long)blockIdx.x * kDecWarps + warp) * pl.G;
    // the rows' last bulk copy has read them (the lanes that issued one wait): they may be rewritten
    auto bulk_read_done = [&] {
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
    };
    auto offset_of = [&](long long b) { return lane <= pl.G && b + lane <= nb ? offs[b + lane] : ~0ull; };
    unsigned long long next_off = b0 < nb ? offset_of(b0) : 0ull;
    for (; b0 < nb; b0 += step) {
        const int nblk = (int)min((long long)pl.G, nb - b0);
        const unsigned long long off = next_off;  // of block b0 + lane
        if (b0 + step < nb) next_off = offset_of(b0 + step);
        const unsigned long long end = __shfl_down_sync(kFull, off, 1);
        const bool ok = lane < nblk && off <= plen && !(off & 3ull);
        // regular: the next offset closes a block of a possible size
        const bool regular = ok && end <= plen && !(end & 3ull) && end > off && end - off <= most;
        const unsigned m_ok = __ballot_sync(kFull, ok), m_reg = __ballot_sync(kFull, regular);
        unsigned alone = 0;  // blocks whose words run past their regular end: staged again by themselves
        int i = 0;
        bool bad = lane < nblk && !ok;
        while (i < nblk || alone) {
            int g0, n;
            bool single = false;
            unsigned long long s0, s1;  // payload bytes staged
            if (alone) {
                g0 = __ffs(alone) - 1;
                alone &= alone - 1u;
                single = true;
            } else {
                g0 = i;
                if (!((m_ok >> g0) & 1u)) {
                    ++i;
                    continue;
                }
                single = !((m_reg >> g0) & 1u);
            }
            s0 = __shfl_sync(kFull, off, g0);
            if (single) {
                n = 1;
                s1 = min(s0 + most, plen);
            } else {
                const unsigned fit = __ballot_sync(kFull, regular && lane >= g0 && end - s0 <= (unsigned long long)pl.cap);
                n = __ffs(~(fit >> g0)) - 1;
                s1 = __shfl_sync(kFull, end, g0 + n - 1);
            }
            if (g0 == i) i += n;
            // stage [s0, s1): whole 16-byte units of the stream, then its last words
            const long long a = head + (long long)s0, e = head + (long long)s1;
            const long long a16 = a & ~15ll, e16 = min((e + 15) & ~15ll, in_bytes & ~15ll);
            const uint32_t dst = daq::smem_addr(base);
            for (long long u = a16 + 16 * lane; u < e16; u += 512)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)(u - a16)), "l"(in + u)
                             : "memory");
            uint32_t *words = reinterpret_cast<uint32_t *>(base);
            const long long t0 = max(a16, e16) + 4 * lane;
            if (t0 + 4 <= e) words[(t0 - a16) >> 2] = *reinterpret_cast<const uint32_t *>(in + t0);
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncwarp();
            if (i >= nblk && !alone && b0 + step < nb) {
                // the last run of this group: bring the next group's payload into L2 meanwhile
                const int nn = (int)min((long long)pl.G, nb - b0 - step);
                const unsigned long long f0 = __shfl_sync(kFull, next_off, 0), f1 = __shfl_sync(kFull, next_off, nn);
                if (lane == 0 && f0 < f1 && f1 <= plen && f1 - f0 <= most * pl.G) {
                    const long long q0 = (head + (long long)f0) & ~15ll, q1 = (head + (long long)f1) & ~15ll;
                    if (q1 > q0)
                        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(in + q0), "r"((uint32_t)(q1 - q0))
                                     : "memory");
                }
            }
            // walk the head words, one block a lane
            const int lim = (int)((e - a16) >> 2);  // words staged end here
            const unsigned long long my_off = __shfl_sync(kFull, off, (g0 + lane) & 31);
            bool good = false;
            if (lane < n && lim > 0) {
                // p only grows, so it ends within the staged words when it
                // always was (reads past them are held at the last one)
                int p = (int)((head + (long long)my_off - a16) >> 2), widest = 0;
                uint16_t *at = pos + lane * X;
#pragma unroll 6
                for (int x = 0; x < X; ++x) {
                    const int q = min(p, lim - 1);
                    const int w = (int)(words[q] >> 16);
                    at[x] = (uint16_t)q;
                    widest = max(widest, w);
                    p += 1 + w;
                }
                good = p <= lim && widest <= 17;
            }
            __syncwarp();
            const unsigned m_good = __ballot_sync(kFull, good);
            const unsigned m_rest = __ballot_sync(kFull, lane < n) & ~m_good;
            // staged alone, a block is cut short or has an impossible width;
            // staged with others it may run past its regular end and is tried again
            if (single) bad |= m_rest != 0u;
            else alone |= m_rest << g0;
            for (int r = 0; r < n; r += pl.nsub) {
                const int g = r + sub;
                const bool mine = sub < pl.nsub && g < n && ((m_good >> g) & 1u);
                const int x0 = 2 * pr;
                const bool two = mine && x0 + 1 < X;
                const uint32_t *h0 = words + (mine ? pos[g * X + x0] : 0);
                const uint32_t *h1 = words + (two ? pos[g * X + x0 + 1] : 0);
                const uint32_t v0 = mine ? h0[0] : 0u, v1 = two ? h1[0] : 0u;
                const int w0 = (int)(v0 >> 16), w1 = (int)(v1 >> 16);
                int16_t *o = out + (sub < pl.nsub ? sub : 0) * 32 * X + x0;
                if (__any_sync(kFull, max(w0, w1) > 8)) {
                    bulk_read_done();
                    decode_wide<kEven>(words, mine ? (int)(h0 - words) : -1, two ? (int)(h1 - words) : -1, o, X);
                } else {
                    uint32_t p0[8], p1[8];
                    column_steps(h0, w0, p0);
                    column_steps(h1, w1, p1);
                    bulk_read_done();
                    int32_t a0 = (int32_t)v0, a1 = (int32_t)v1;  // the low halves count
                    if (mine) {
#pragma unroll
                        for (int q = 0; q < 32; ++q) {
                            const int k = q & 7, j = q >> 3;
                            if (q) {
                                a0 = __dp4a((int)p0[k], 1 << (8 * j), a0);
                                a1 = __dp4a((int)p1[k], 1 << (8 * j), a1);
                            }
                            if (kEven) {
                                *reinterpret_cast<uint32_t *>(o + q * X) = __byte_perm((uint32_t)a0, (uint32_t)a1, 0x5410);
                            } else {
                                o[q * X] = (int16_t)a0;
                                if (two) o[q * X + 1] = (int16_t)a1;
                            }
                        }
                    }
                }
                __syncwarp();
                // rows of the good blocks to the pool: a bulk copy per whole block
                const bool whole = 32 * (b0 + g0 + r + pl.nsub) <= rows;
                if (vec_out && whole) {
                    if (pr == 0 && mine) {
                        daq::fence_proxy_async_smem();
                        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                                         pool_out + 32 * (b0 + g0 + g) * X),
                                     "r"(daq::smem_addr(out + sub * 32 * X)), "r"(64 * X)
                                     : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                } else {
                    for (int u = 0; u < pl.nsub && r + u < n; ++u) {
                        if (!((m_good >> (r + u)) & 1u)) continue;
                        const long long r0 = 32 * (b0 + g0 + r + u);
                        const int ne = (int)min(32ll, rows - r0) * X;
                        for (int q = lane; q < ne; q += 32) pool_out[r0 * X + q] = out[u * 32 * X + q];
                    }
                    __syncwarp();
                }
            }
        }
        if (bad) atomicOr(err, 2);
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Grid of a pipelined kernel: every CTA resident at once (its warps step
// through blocks), at most one warp per block.  The kernel's dynamic
// shared-memory limit is raised once per device to what the largest n_xtal
// needs (smem_max; a later call must never lower it), and the resident count
// is found once per (kernel slot, device, n_xtal) and kept.
constexpr int kGridDevices = 16;
int g_resident[4][kGridDevices][kMaxX + 1] = {};  // CTAs resident per GPU, 0 = not known yet
bool g_limit_set[4][kGridDevices] = {};

template <typename K>
int pipelined_grid(int slot, K kernel, int X, int threads, size_t smem, size_t smem_max, long long want)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    int resident = dev < kGridDevices ? g_resident[slot][dev][X] : 0;
    if (resident == 0) {
        int sms = 0, per = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 0;
        if (dev >= kGridDevices || !g_limit_set[slot][dev]) {
            if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max) != cudaSuccess)
                return 0;
            if (dev < kGridDevices) g_limit_set[slot][dev] = true;
        }
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess || per < 1)
            return 0;
        resident = per * sms;
        if (dev < kGridDevices) g_resident[slot][dev][X] = resident;
    }
    return (int)std::max<long long>(1, std::min<long long>(want, (long long)resident));
}

// The most shared memory a warp of a kernel takes, over the crystal counts.  Not the
// plan of the most crystals: 64 columns side by side are also 16 blocks of 4 crystals,
// and an encoder stage keeps a word for each block.
template <typename F> size_t most_bytes(F bytes_of)
{
    size_t most = 0;
    for (int X = 1; X <= kMaxX; ++X) most = std::max(most, bytes_of(X));
    return most;
}

// Workspace: one status word per chunk, then the ticket and the role counter.
long long enc_chunks(long long nb, int X) { return (nb + EncPlan(X).chunk_blocks() - 1) / EncPlan(X).chunk_blocks(); }
size_t pack_ws(long long nb, int X) { return (8 * (size_t)(enc_chunks(nb, X) + 2) + 255) & ~size_t(255); }

}  // namespace daq_pack

using namespace daq_pack;

extern "C" {

int64_t daq_pack_bound(int64_t rows, int n_xtal)
{
    if (rows < 0 || n_xtal < 1 || n_xtal > kMaxX) return -1;
    const int64_t nb = (rows + 31) / 32;
    return 16 + 8 * (nb + 1) + nb * (int64_t)n_xtal * 4 * 18;
}

int daq_pack_workspace_size(int64_t rows, int n_xtal, size_t *bytes)
{
    if (!bytes || rows < 0 || n_xtal < 1 || n_xtal > kMaxX) return DAQ_EINVAL;
    *bytes = pack_ws((rows + 31) / 32, n_xtal);
    return DAQ_OK;
}

int daq_pack_pool(const int16_t *pool, int64_t rows, int n_xtal, void *out, int64_t out_cap, int64_t *out_bytes,
                  void *workspace, size_t workspace_bytes, void *stream)
{
    if (rows < 0 || n_xtal < 1 || out_cap < 0 || !out_bytes || (rows > 0 && !pool)) return DAQ_EINVAL;
    if (n_xtal > kMaxX) return DAQ_EUNSUPPORTED;
    if ((out_cap > 0 && !out) || (reinterpret_cast<uintptr_t>(out) & 15) || (reinterpret_cast<uintptr_t>(out_bytes) & 7) ||
        (reinterpret_cast<uintptr_t>(pool) & 15))
        return DAQ_EINVAL;
    const long long nb = (rows + 31) / 32;
    if (!workspace || workspace_bytes < pack_ws(nb, n_xtal) || (reinterpret_cast<uintptr_t>(workspace) & 15)) return DAQ_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const long long n_chunks = enc_chunks(nb, n_xtal);
    const bool even = (n_xtal % 2) == 0;
    const auto kernel = even ? pack_kernel<true> : pack_kernel<false>;
    static const size_t warp_most = most_bytes([](int X) { return EncPlan(X).bytes(); });
    const size_t smem = kEncWarps * EncPlan(n_xtal).bytes(), most = kEncWarps * warp_most;
    const int grid = pipelined_grid(even ? 0 : 1, kernel, n_xtal, kEncThreads, smem, most, n_chunks + 1);
    if (grid < 1) return DAQ_ECUDA;
    if (cudaMemsetAsync(workspace, 0, 8 * (size_t)(n_chunks + 2), s) != cudaSuccess) return DAQ_ECUDA;
    kernel<<<grid, kEncThreads, smem, s>>>(pool, rows, n_xtal, nb, static_cast<unsigned long long *>(workspace), n_chunks,
                                           static_cast<unsigned char *>(out), out_cap, reinterpret_cast<long long *>(out_bytes));
    return cudaGetLastError() == cudaSuccess ? DAQ_OK : DAQ_ECUDA;
}

int daq_unpack_pool(const void *in, int64_t in_bytes, int64_t rows, int n_xtal, int16_t *pool_out, int32_t *err,
                    void *stream)
{
    if (!in || in_bytes < 16 || rows < 0 || n_xtal < 1 || !err || (rows > 0 && !pool_out) ||
        (reinterpret_cast<uintptr_t>(in) & 15))
        return DAQ_EINVAL;
    if (n_xtal > kMaxX) return DAQ_EUNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(err, 0, sizeof(int32_t), s) != cudaSuccess) return DAQ_ECUDA;
    const long long nb = (rows + 31) / 32;
    const bool even = (n_xtal % 2) == 0;
    const auto kernel = even ? unpack_kernel<true> : unpack_kernel<false>;
    const DecPlan pl(n_xtal);
    static const size_t warp_most = most_bytes([](int X) { return DecPlan(X).bytes(X); });
    const size_t most = kDecWarps * warp_most;
    const int grid = pipelined_grid(even ? 2 : 3, kernel, n_xtal, kDecThreads, kDecWarps * pl.bytes(n_xtal), most,
                                    (std::max<long long>(nb, 1) + kDecWarps * pl.G - 1) / (kDecWarps * pl.G));
    if (grid < 1) return DAQ_ECUDA;
    kernel<<<grid, kDecThreads, kDecWarps * pl.bytes(n_xtal), s>>>(static_cast<const unsigned char *>(in), in_bytes, rows,
                                                                    n_xtal, nb, pool_out, err);
    return cudaGetLastError() == cudaSuccess ? DAQ_OK : DAQ_ECUDA;
}

}  // extern "C"
