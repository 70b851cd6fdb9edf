// Decoding of binary32 streams: included by zccl_codec.cu inside its unnamed namespace.
//
// A CTA takes a tile at a time: four warps decode a round each, a lane a block of 32 elements, and a fifth warp fetches:
// it reads index and header a tile ahead, brings the blobs into one of three buffers by bulk copies, checks them and
// hands their facts over.  Sizes and signs are worked on four (or two) to a word: a block's planes are transposed into
// bytes, made two's complement with a bias of 128 in the same words and summed by byte dot products; the warps exchange
// their rounds' sums (one barrier per tile), and every lane then walks its elements.
//
// What bounds it: DRAM on large arrays (6.2 to 6.5 TB/s of blob reads and value writes at 2^27 elements, see TileDeal), the
// launch's ramps below that.  A warp per tile, four rounds in a row, with its own checks and 20 instructions per element
// took 18.1 us for 2^24 elements at code lengths around 4, 288 us for 2^28 at 8.5, 103 for 2^27 at 3 and 5.8 us for a few
// tiles; this form (17) takes 16.4, 233, 98 and 4.3 us.  Two buffers instead of three 18.0 us for 2^24, six CTAs per SM
// on two buffers 18.6, four on three 17.6.

// ------------------------------------------------------------------------------------------------ one block

// The payload of a block (sign word, planes) as biased deltas: element N h + i is field h of word i, stored as
// delta + 2^(N - 1).  Code lengths up to N - 1.  Words beyond the block's own planes are read too (the caller's buffer
// has room behind it) and masked away.  `sum`: the block's deltas added up.
template <int N>
__device__ __forceinline__ void load_deltas(const uint32_t* pay, uint32_t L, bool half, uint32_t (&w)[N], int32_t& sum)
{
    constexpr uint32_t ones = N == 8 ? 0x01010101u : 0x00010001u, bias = ones << (N - 1);
    const uint32_t sign = pay[0];
#pragma unroll
    for (int k = 0; k < N / 2; ++k) w[k] = pay[1 + k];
#pragma unroll
    for (int k = N / 2; k < N; ++k) w[k] = 0;
    if (!half) {              // (uniform) some block of the round has more than N / 2 planes
#pragma unroll
        for (int k = N / 2; k < N - 1; ++k) w[k] = pay[1 + k];
    }
    bit_transpose<N>(w);
    const uint32_t mask = ((1u << L) - 1u) * ones;
    uint32_t acc = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t s = (sign >> i) & ones;
        w[i] = ((w[i] & mask) ^ (bias - s)) + s;      // bias + magnitude, or bias - magnitude; no carry between fields
        if (N == 8) acc = __dp4a(w[i], 0x01010101u, acc);
        else acc = __dp2a_lo(w[i], 0x00000101u, acc);
    }
    sum = (int32_t)(acc - (32u << (N - 1)));
}

// Inclusive scan over the lanes.
__device__ __forceinline__ int32_t warp_incl_scan_s(int32_t v, int lane)
{
    return (int32_t)warp_incl_scan((uint32_t)v, lane);
}

// The lane's 32 values from the biased deltas (word i, field h = element N h + i): codes are exact in fp32 (the caller
// checked).  A delta under the exponent of 2^23 is a float, minus 2^23 and the bias it is the delta; the running code
// is a chain of additions; one multiplication makes the value.  Four values at a time go to `put(chunk, values)`.
template <int N, class Put>
__device__ __forceinline__ void expand_deltas(const uint32_t (&w)[N], int32_t code_in_front, float s, Put&& put)
{
    float run = (float)code_in_front;
    const float neg = -(8388608.0f + (float)(1u << (N - 1)));
    const float2 neg2 = make_float2(neg, neg), s2 = make_float2(s, s);
    // the bits of 2^23, in a way the compiler cannot see through: a byte permute has one immediate operand, the selector, and
    // a constant it knows it puts into a register anew for every element
    const uint32_t k23 = __float_as_uint(negative_zero(s)) ^ 0xCB000000u;
#pragma unroll
    for (int h = 0; h < 32 / N; ++h) {
        const uint32_t sel = N == 8 ? 0x7650u + (uint32_t)h : 0x7610u + 0x0022u * (uint32_t)h;
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            const float2 d01 = __fadd2_rn(make_float2(__uint_as_float(prmt(w[4 * q + 0], k23, sel)), __uint_as_float(prmt(w[4 * q + 1], k23, sel))), neg2);
            const float2 d23 = __fadd2_rn(make_float2(__uint_as_float(prmt(w[4 * q + 2], k23, sel)), __uint_as_float(prmt(w[4 * q + 3], k23, sel))), neg2);
            const float r0 = __fadd_rn(run, d01.x), r1 = __fadd_rn(r0, d01.y), r2 = __fadd_rn(r1, d23.x), r3 = __fadd_rn(r2, d23.y);
            run = r3;
            put((uint32_t)(h * (N / 4) + q), make_float2(r0, r1), make_float2(r2, r3), s2);
        }
    }
}

// ------------------------------------------------------------------------------------------------ a tile's blob

constexpr uint32_t kBlobWords = 1 + kLWords + 32 * 16 * kRoundsPerTile;   // a tile whose code lengths stay below 16
constexpr uint32_t kBlobBufWords = (kBlobWords + 4 + 16 + 3) / 4 * 4;     // slack of the 16-byte cover; what is read beyond a block's planes

// A tile as the fetching warp hands it to the coding warps.
enum : uint32_t { kTileNone = 0,     // no more tiles
                  kTileFast = 1,     // its blob is in the buffer, its codes are exact in fp32
                  kTileSlow = 2,     // to be read where it is, with integer arithmetic
                  kTileSkip = 3 };   // nothing to decode (reported)
struct alignas(16) DecodeWork {
    unsigned long long src;          // the blob's first word (global memory)
    unsigned long long start;        // the tile's first element
    uint32_t kind, job, len;         // len: elements of the tile
    float s;
    uint32_t words, lead;            // of the blob; words between the buffer's start and the blob
    int32_t outlier;
    uint32_t t;                      // number within the launch
    uint32_t before[kTileWarps];     // payload words in front of each round
    uint32_t bytes;                  // what the copy brings, from the boundary in front of the blob
    float eb_abs;
    uint32_t valid;                  // the stream's header agrees with the job
    uint32_t tiles;                  // of the stream
};

// What the code lengths of a tile say (the lane holds code-length word `lane`).
struct BlobFacts {
    bool ok;          // consistent with the blob's size
    bool exact;       // every code of the tile stays below 2^23 in magnitude: fp32 arithmetic is exact
    uint32_t before;  // lane 8 k: payload words in front of round k
};
__device__ __forceinline__ BlobFacts blob_facts(uint32_t lw, uint32_t words, uint32_t nb, int32_t outlier, int lane)
{
    BlobFacts f;
    const uint32_t any = __reduce_or_sync(kFull, lw);
    const uint32_t longest = (any | (any >> 8) | (any >> 16) | (any >> 24)) & 0xFFu;   // at least the longest code length's bits
    const uint32_t sizes = __dp4a(lw + (((lw + 0x7F7F7F7Fu) >> 7) & 0x01010101u), 0x01010101u, 0u);   // + 1 per block that has any (lengths up to 31)
    const uint32_t incl = warp_incl_scan(sizes, lane);
    const uint32_t padw = (nb + 3) >> 2;
    f.before = incl - sizes;
    f.ok = (any & 0xE0E0E0E0u) == 0u && 1u + padw + __shfl_sync(kFull, incl, 31) == words;
    if (nb & 3u) {    // padding of the code-length area must be zero
        const uint32_t last = __shfl_sync(kFull, lw, (int)(padw - 1u));
        if (last >> (8u * (nb & 3u))) f.ok = false;
    }
    const uint32_t ao = (uint32_t)(outlier < 0 ? -outlier : outlier);
    // every partial sum of deltas is below sum_b 32 * 2^L_b
    f.exact = ao < (1u << 22) && longest < 11u;
    if (!f.exact) {
        const uint32_t L0 = lw & 0xFFu, L1 = (lw >> 8) & 0xFFu, L2 = (lw >> 16) & 0xFFu, L3 = (lw >> 24) & 0xFFu;
        uint32_t spread = 1u << 24;
        if (max(max(L0, L1), max(L2, L3)) <= 18u) spread = min((32u << L0) + (32u << L1) + (32u << L2) + (32u << L3), 1u << 24);
        f.exact = ao < (1u << 23) && __reduce_add_sync(kFull, spread) < (1u << 23);
    }
    return f;
}

// Which tiles a CTA takes: its number and every gridDim.x-th from there, or (DEALT) its number and then whatever is next on
// a counter.  By number, CTAs that get on faster run ahead of the others, and the addresses a launch writes at a time
// spread until DRAM loses a tenth of its rate: 2^27 values at a code length of 3 took 110 us (5.5 TB/s; a warp per tile,
// in step by its slowness, 103) and take 98 from the counter (6.2), 2^28 220 and 191.  The counter's round trips cost
// a microsecond, mostly when all CTAs ask it for the first time at once, so launches of fewer than kDealtTiles tiles per
// CTA go by number: 2^24 values (5.5 tiles) 14.5 us and 15.6 from the counter, 2^25.6 (16.8) 42.6 and 40.4, at a code
// length of 0 38.1 and 38.9.
constexpr uint32_t kDealtTiles = 16;
template <bool DEALT>
struct TileDeal {
    uint32_t* next;
    uint32_t total, ticket = 0;
    bool over = false;          // the counter is through
    __device__ __forceinline__ TileDeal(uint32_t* counter, uint32_t total_tiles, int lane) : next(counter), total(total_tiles) { ask(lane); }
    // Every CTA takes one number beyond the last, so the counter goes around once in a launch and is back at 0 behind it.
    __device__ __forceinline__ void ask(int lane) { if (DEALT && lane == 0) ticket = atomicInc(next, total - 1u); }
    __device__ __forceinline__ uint32_t behind(uint32_t t, int lane)   // the tile behind t
    {
        if (!DEALT) return t + gridDim.x < t ? kNoTile : t + gridDim.x;
        if (over) return kNoTile;
        t = gridDim.x + __shfl_sync(kFull, ticket, 0);
        over = t >= total;
        if (over) return kNoTile;
        ask(lane);
        return t;
    }
    __device__ __forceinline__ void leave(int lane)                    // (where a wait ran out the counter is not through yet)
    {
        while (DEALT && !over) (void)behind(0, lane);
    }
};

// The warp that fetches blobs for its CTA: every tile's index entries and its stream's header are loaded (one word per
// lane) a tile before they are needed.
template <class JB>
struct BlobFetcher {
    uint32_t begin = 0, count = 0, raw_t = kNoTile, raw = 0, raw_begin = 0;
    int job = 0, raw_job = 0;
    __device__ __forceinline__ void locate(const JB& jb, uint32_t t)
    {
        if (t - begin < count) return;
        job = find_job(jb, t);
        begin = jb.job[job].tile_begin;
        count = (job + 1 < jb.count ? jb.job[job + 1].tile_begin : jb.total_tiles) - begin;
    }
    // asks for the header and index words of tile t
    __device__ __forceinline__ void ask(const JB& jb, uint32_t t, int lane)
    {
        raw_t = t < jb.total_tiles ? t : kNoTile;
        if (raw_t == kNoTile) return;
        locate(jb, t);
        raw_begin = begin; raw_job = job;
        const Job& q = jb.job[job];
        const uint32_t tile = t - begin;
        // lanes 0 .. 7: the header; 8, 9: the index entries of the tile in front and of the tile
        const uint32_t at = lane < kHeaderWords ? (uint32_t)lane : kHeaderWords + tile + (uint32_t)lane - 9u;
        const bool some = lane < kHeaderWords ? q.in_cap >= (unsigned)kHeaderBytes : lane == 9 || (lane == 8 && tile);
        raw = some && 4ull * ((unsigned long long)at + 1ull) <= q.in_cap ? ldg_u32(q.in_c + at) : 0u;
    }
    // what they say
    // (SAME_N: the stream has to have exactly the job's elements, not at most)
    // (F64: a binary64 stream, whose step is the binary64 in the header words of bound and step)
    template <bool SAME_N, bool F64>
    __device__ __forceinline__ DecodeWork resolve(const JB& jb, uint32_t& status, int lane) const
    {
        DecodeWork w;
        w.kind = kTileNone; w.src = 0; w.start = 0; w.words = 0; w.len = 0; w.s = 1.0f; w.job = (uint32_t)raw_job; w.lead = 0; w.outlier = 0; w.t = raw_t; w.bytes = 0; w.eb_abs = 0.0f; w.valid = 0; w.tiles = 0;
        if (raw_t == kNoTile) return w;
        w.kind = kTileSkip;
        const Job& q = jb.job[raw_job];
        const uint32_t tile = raw_t - raw_begin;
        const uint32_t magic = __shfl_sync(kFull, raw, 0), ver = __shfl_sync(kFull, raw, 1), T = __shfl_sync(kFull, raw, 6), nT = __shfl_sync(kFull, raw, 7);
        const unsigned long long n = (unsigned long long)__shfl_sync(kFull, raw, 2) | ((unsigned long long)__shfl_sync(kFull, raw, 3) << 32);
        const uint32_t raw_eb = __shfl_sync(kFull, raw, 4), raw_s = __shfl_sync(kFull, raw, 5);
        const float s = __uint_as_float(raw_s);
        const double s64 = __hiloint2double((int)raw_s, (int)raw_eb);
        const uint32_t w_beg = __shfl_sync(kFull, raw, 8), w_end = __shfl_sync(kFull, raw, 9);
        const bool ok = magic == kMagic && ver == (F64 ? kVersionF64 : kVersion) && T == (uint32_t)kTile && (n + kTile - 1) / kTile == nT &&
                        q.in_cap >= (unsigned long long)kHeaderBytes + 4ull * nT && (F64 ? s64 > 0.0 && isfinite(s64) : s > 0.0f && isfinite(s));
        if (!ok) { status |= kStBadStream; return w; }
        if (SAME_N && n != q.n) { status |= kStBadStream; return w; }
        if (n > q.n) { status |= kStCapacity; return w; }
        w.valid = 1;
        w.tiles = nT;
        w.s = s;
        w.eb_abs = __uint_as_float(raw_eb);
        if (tile >= nT) return w;
        w.start = (unsigned long long)tile * kTile;
        w.len = (uint32_t)(n - w.start < (unsigned long long)kTile ? n - w.start : kTile);
        const unsigned long long blob0 = (unsigned long long)kHeaderWords + nT;
        if (w_end <= w_beg || (blob0 + w_end) * 4ull > q.in_cap) { status |= kStBadStream; return w; }
        const uint32_t* p = q.in_c + blob0 + w_beg;
        w.src = (unsigned long long)(uintptr_t)p;
        w.words = w_end - w_beg;
        w.lead = (uint32_t)((uintptr_t)p & 15u) >> 2;
        w.kind = w.words <= kBlobWords ? kTileFast : kTileSlow;
        // the copy reads up to the 16-byte boundary behind the blob; where that is not readable (the last tile of a stream
        // that fills its buffer), up to the boundary in front, and the last words follow one by one
        const uintptr_t a_end = ((uintptr_t)(p + w.words) + 15) & ~(uintptr_t)15;
        w.bytes = (4u * (w.lead + w.words) + (a_end - (uintptr_t)q.in_c <= (uintptr_t)q.in_cap ? 15u : 0u)) & ~15u;
        return w;
    }
};
// Brings a tile's blob into `buf` (one lane).
__device__ __forceinline__ void fetch_blob(const DecodeWork& w, uint32_t* buf, unsigned long long* bar)
{
    if (w.kind == kTileFast && w.bytes) {
        mbar_expect_tx(bar, w.bytes);
        bulk_load(buf, (const void*)(uintptr_t)(w.src - 4u * w.lead), w.bytes, bar);
    } else mbar_arrive(bar);
}
// A decoding job with an output stream is a forwarded chunk: the tile's blob goes on, from the buffer it was brought to, to
// the same place in the receiver's slot, and what goes once per tile or stream with it (the fetching warp).
__device__ __forceinline__ void forward_blob(const Job& q, const DecodeWork& w, const uint32_t* buf, uint32_t tile, uint32_t& status, int lane)
{
    if (!q.out || !w.valid || (w.kind == kTileSkip && w.tiles)) return;
    const unsigned long long at = w.tiles ? (unsigned long long)((const uint32_t*)(uintptr_t)w.src - q.in_c) : (unsigned long long)kHeaderWords;
    if ((at + w.words) * 4ull > q.out_cap) { status |= kStCapacity; return; }
    if (w.tiles) {
        // slots start on the same kind of boundary, so the whole cover can go in one bulk store: the words of the neighbours at
        // its ends are those the neighbours' covers bring
        if (w.kind == kTileFast && (((uintptr_t)q.out ^ (uintptr_t)q.in_c) & 15u) == 0 && w.bytes >= 4u * (w.lead + w.words) &&
            (at - w.lead) * 4ull + w.bytes <= q.out_cap) {
            if (lane == 0) {
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(q.out + (at - w.lead)), "r"(smem_u32(buf)), "r"(w.bytes) : "memory");
            }
        } else copy_words(q.out + at, w.kind == kTileFast ? buf + w.lead : (const uint32_t*)(uintptr_t)w.src, w.words, lane);
        if (lane == 0) q.out[kHeaderWords + tile] = (uint32_t)(at - kHeaderWords - w.tiles) + w.words;
    }
    if (tile == 0 && lane < kHeaderWords) q.out[lane] = ldg_u32(q.in_c + lane);
    if (lane == 0 && tile + 1u >= w.tiles) *q.out_bytes = (size_t)((at + w.words) * 4ull);
}
// Reads the head of a tile's blob (in `buf` when it was brought there), completes its facts and hands them over.
template <bool F64>
__device__ __forceinline__ void check_blob(DecodeWork& w, uint32_t* buf, DecodeWork* to, uint32_t& status, int lane)
{
    uint32_t before = 0;
    if (w.kind == kTileFast || w.kind == kTileSlow) {
        const uint32_t nb = (w.len + kBlock - 1) / kBlock, padw = (nb + 3) >> 2;
        uint32_t lw = 0;
        const bool mine = (uint32_t)lane < padw && (uint32_t)lane + 1u < w.words;
        if (w.kind == kTileFast) {
            const uint32_t at = (w.bytes >> 2) + (uint32_t)lane;
            if (at < w.lead + w.words) buf[at] = ldg_u32((const uint32_t*)(uintptr_t)w.src + at - w.lead);   // at most three words
            __syncwarp();
            if (mine) lw = buf[w.lead + 1u + (uint32_t)lane];
            w.outlier = (int32_t)buf[w.lead];
        } else {
            const uint32_t* g = (const uint32_t*)(uintptr_t)w.src;
            if (mine) lw = ldg_u32(g + 1 + lane);
            w.outlier = (int32_t)ldg_u32(g);
        }
        const BlobFacts f = blob_facts(lw, w.words, nb, w.outlier, lane);
        before = f.before;
        if (!f.ok) { status |= kStBadStream; w.kind = kTileSkip; }
        else if (!F64 && !f.exact) w.kind = kTileSlow;   // (binary64 codes are summed as integers)
    }
    if (lane == 0) *to = w;
    __syncwarp();
    if ((lane & 7) == 0) to->before[lane >> 3] = before;
    __syncwarp();
}

// ------------------------------------------------------------------------------------------------ decompress

constexpr uint32_t kBlobBufs = 3;   // tiles' blobs of a CTA: being decoded, checked, on their way
struct alignas(1024) DecodeShared {
    float out[kTileWarps][kRound];
    alignas(16) uint32_t blob[kBlobBufs][kBlobBufWords];
    DecodeWork work[kBlobBufs];
    alignas(16) int32_t sums[kBlobBufs][kTileWarps];   // the rounds' sums of deltas, by parity of the CTA's tile count
    alignas(8) unsigned long long landed[kBlobBufs], ready[kBlobBufs], free[kBlobBufs];
};
static_assert(offsetof(DecodeShared, blob) % 16 == 0 && sizeof(uint32_t) * kBlobBufWords % 16 == 0, "targets of the copy engine");
constexpr int kDecodeThreads = kTileThreads + 32;

// The code in front of round rd: the tile's first code and the sums of the rounds in front, exchanged by the four coding
// warps (named barrier 1).
__device__ __forceinline__ int32_t code_in_front(int32_t* sums, int32_t mine, int32_t outlier, uint32_t rd, int lane)
{
    if (lane == 0) sums[rd] = mine;
    asm volatile("bar.sync 1, 128;" ::: "memory");
    const int4 s = *reinterpret_cast<const int4*>(sums);
    return outlier + (rd > 0 ? s.x : 0) + (rd > 1 ? s.y : 0) + (rd > 2 ? s.z : 0);
}

// The fetching warp's loop: the blob of tile i of the CTA (the first one is `first`; DEALT, next: see TileDeal) into
// buffer i mod NB, its facts as soon as it has landed.  `also` is called once per tile, in their order, for what else a
// tile needs (at once for the first two, for the others when the tile's facts have been handed over); false ends the
// loop.  FORWARD: see forward_blob.
template <uint32_t NB, bool SAME_N, bool FORWARD, bool F64, bool DEALT, class JB, class Also>
__device__ __forceinline__ void fetch_tiles(const JB& jb, uint32_t first, uint32_t* next, uint32_t (*blob)[kBlobBufWords], DecodeWork* work, unsigned long long* landed,
                                            unsigned long long* ready, unsigned long long* free_, uint32_t& status, int lane, Also&& also)
{
    BlobFetcher<JB> fetch;
    TileDeal<DEALT> deal(next, jb.total_tiles, lane);
    uint32_t t = first, out = 0;
    DecodeWork w[NB - 1];               // the tiles whose blobs are on their way
    auto send = [&](DecodeWork& to) {   // tile number `out` of the CTA
        to = fetch.template resolve<SAME_N, F64>(jb, status, lane);
        t = deal.behind(t, lane);
        fetch.ask(jb, t, lane);
        const uint32_t b = out % NB;
        const bool ok = out < NB || mbar_wait_resting(&free_[b], (out / NB - 1u) & 1u);
        if (!ok) status |= kStTimeout;
        else if (lane == 0) {
            // the blob forwarded from this buffer has left it (a group per tile; the newest is that of the tile handed over last,
            // in another buffer)
            if (FORWARD) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            fetch_blob(to, blob[b], &landed[b]);
        }
        __syncwarp();
        const bool more = out >= 2 || also(to, out);
        ++out;
        return ok && more;
    };
    fetch.ask(jb, t, lane);
#pragma unroll
    for (uint32_t k = 0; k + 1 < NB; ++k) (void)send(w[k]);
    for (uint32_t i = 0;; ++i) {
        const uint32_t b = i % NB;
        if (!mbar_wait(&landed[b], (i / NB) & 1u)) { status |= kStTimeout; break; }
        check_blob<F64>(w[0], blob[b], &work[b], status, lane);
        if (lane == 0) mbar_arrive(&ready[b]);
        __syncwarp();
        if (FORWARD && w[0].kind != kTileNone) {
            const Job& q = jb.job[w[0].job];
            forward_blob(q, w[0], blob[b], w[0].t - q.tile_begin, status, lane);
            if (lane == 0) asm volatile("cp.async.bulk.commit_group;" ::: "memory");   // (empty when nothing went in bulk)
            __syncwarp();
        }
        if (w[0].kind == kTileNone || (i >= 2 && !also(w[0], i))) break;
#pragma unroll
        for (uint32_t k = 0; k + 2 < NB; ++k) w[k] = w[k + 1];
        if (!send(w[NB - 2])) break;
    }
    deal.leave(lane);
    if (FORWARD && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Asks a tile's blob into L2, by one warp in front of the wait for the kernel in front on the stream.  Only a hint: what that
// kernel may still be writing is read past L1, looked at for nothing but the range to ask for, which lies within the stream's
// buffer, and read again behind the wait; L2 stays coherent with what it writes.  For streams that are mostly older than that:
// 2^24 values decompressed at 1e-4 18.3 -> 17.7 us, 2^22 smooth 7.1 -> 6.2, 2^20 4.4 -> 3.9, 2^14 3.22 -> 3.17; in launches of the collectives, whose streams the kernel in
// front writes, 8 x 2^21 Allreduce 68.4 -> 69.7.
__device__ __forceinline__ void hint_blob(const Job& q, uint32_t tile, int lane)
{
    const unsigned long long at = (unsigned long long)kHeaderWords + tile + (uint32_t)lane;   // behind the index entry of this lane
    uint32_t v = 0;
    if (lane < 2 && (lane || tile) && 4ull * at <= q.in_cap)
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(q.in_c + at - 1) : "memory");
    const uint32_t end = __shfl_sync(kFull, v, 1);
    if (lane == 0 && end > v && end - v <= kBlobWords) {
        const unsigned long long blobs = (unsigned long long)kHeaderWords + (q.n + kTile - 1) / kTile;
        const uintptr_t from = (uintptr_t)(q.in_c + blobs + v) & ~(uintptr_t)15, to = (uintptr_t)(q.in_c + blobs + end) & ~(uintptr_t)15;
        if (to > from && to <= (uintptr_t)q.in_c + q.in_cap) bulk_prefetch_l2((const void*)from, (uint32_t)(to - from));
    }
}

template <int CAP, bool DEALT>
__global__ void __launch_bounds__(kDecodeThreads, kDecodeCtas) decode_tiles_kernel(const __grid_constant__ JobBatchT<CAP> jb,
                                                                                  const __grid_constant__ TileMapsT<CAP> maps, Workspace ws)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DecodeShared& sh = *reinterpret_cast<DecodeShared*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t rd = (uint32_t)tid >> 5;
    if (tid == 0) {
#pragma unroll
        for (int k = 0; k < (int)kBlobBufs; ++k) { mbar_init(&sh.landed[k], 1); mbar_init(&sh.ready[k], 1); mbar_init(&sh.free[k], kTileWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (CAP == 1 && rd == kTileWarps) hint_blob(jb.job[0], blockIdx.x, lane);
    __syncthreads();
    pdl_enter();
    uint32_t status = 0;
    if (rd == kTileWarps) {
        fetch_tiles<kBlobBufs, false, (CAP > 1), false, DEALT>(jb, blockIdx.x, ws.next_decode, sh.blob, sh.work, sh.landed, sh.ready, sh.free, status, lane,
                                                   [&](const DecodeWork& w, uint32_t) {
                                                       if (CAP > 1 && lane == 0 && w.kind != kTileNone) prefetch_map(&maps.m[w.job]);
                                                       return true;
                                                   });
        if (status) atomicOr(ws.status, status);
        return;
    }
    const uint32_t e0 = rd * (uint32_t)kRound, sw = ((uint32_t)lane & 7u) << 4;
    float* stage = sh.out[rd];
    char* row = reinterpret_cast<char*>(stage) + 128 * lane;
    for (uint32_t i = 0;; ++i) {
        const uint32_t b = i % kBlobBufs;
        if (!mbar_wait(&sh.ready[b], (i / kBlobBufs) & 1u)) { status |= kStTimeout; break; }
        const DecodeWork& w = sh.work[b];
        const uint32_t kind = w.kind;
        if (kind == kTileNone) break;
        // the tile's facts are copied: the buffer is given back in the middle of the decoding
        const uint32_t len = w.len, job = CAP == 1 ? 0 : w.job;
        const unsigned long long start = w.start;
        const float s = w.s;
        auto give_back = [&]() {
            if (lane == 0) mbar_arrive(&sh.free[b]);
        };
        if (kind == kTileSkip) { __syncwarp(); give_back(); continue; }
        const uint32_t nb = (len + kBlock - 1) / kBlock, padw = (nb + 3) >> 2;
        // the stage was handed to a tensor store a tile ago, which by now has drained it
        auto drained = [&]() {
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
        };
        auto put = [&](uint32_t chunk, float2 r01, float2 r23, float2 s2) {
            const float2 a = __fmul2_rn(r01, s2), c = __fmul2_rn(r23, s2);
            *reinterpret_cast<float4*>(row + ((16u * chunk) ^ sw)) = make_float4(a.x, a.y, c.x, c.y);
        };
        const uint32_t bi = 32u * rd + (uint32_t)lane;
        const unsigned long long src = w.src;
        const int32_t outlier = w.outlier;
        const uint32_t before = w.before[rd];
        bool slow = kind == kTileSlow;
        uint32_t L;
        const uint32_t* blob = sh.blob[b] + w.lead;
        if (!slow) {
            L = bi < nb ? reinterpret_cast<const unsigned char*>(blob + 1)[bi] : 0u;
            slow = __any_sync(kFull, L > 15u);
        } else L = bi < nb ? (uint32_t)__ldg((const unsigned char*)(uintptr_t)src + 4u + bi) : 0u;
        if (!slow) {
            const uint32_t nw = L ? L + 1u : 0u;
            const uint32_t* pay = blob + 1 + padw + before + (warp_incl_scan(nw, lane) - nw);
            int32_t sum;
            if (!__any_sync(kFull, L > 7u)) {
                uint32_t v[8];
                load_deltas<8>(pay, L, !__any_sync(kFull, L > 4u), v, sum);
                const int32_t incl = warp_incl_scan_s(sum, lane);
                const int32_t code = code_in_front(sh.sums[b], __shfl_sync(kFull, incl, 31), outlier, rd, lane) + incl - sum;
                give_back();
                drained();
                expand_deltas<8>(v, code, s, put);
            } else {
                uint32_t v[16];
                load_deltas<16>(pay, L, !__any_sync(kFull, L > 8u), v, sum);
                const int32_t incl = warp_incl_scan_s(sum, lane);
                const int32_t code = code_in_front(sh.sums[b], __shfl_sync(kFull, incl, 31), outlier, rd, lane) + incl - sum;
                give_back();
                drained();
                expand_deltas<16>(v, code, s, put);
            }
        } else {   // read where it is
            const uint32_t* in_global = (const uint32_t*)(uintptr_t)src;
            uint32_t off = before;
            int32_t code = 0;
            skip_round(in_global, padw, L, &off, &code, lane);
            code = code_in_front(sh.sums[b], code, outlier, rd, lane);
            give_back();
            off = before;
            drained();
            decode_round_general(in_global, padw, L, &off, &code, s, stage, lane, nullptr, 0u);
        }
        __syncwarp();   // the stage's rows, written by all lanes, are visible
        float* __restrict__ y = jb.job[job].y;
        if (e0 + (uint32_t)kRound <= len && (((uintptr_t)y) & 15u) == 0) {
            if (lane == 0) tensor_store_round(&maps.m[job], (uint32_t)(start >> 5) + 32u * rd, stage);
        } else if (e0 < len) {
            store_round_ragged(y + start + e0, stage, len - e0 < (uint32_t)kRound ? len - e0 : (uint32_t)kRound, lane);
        }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (status) atomicOr(ws.status, status);
}
