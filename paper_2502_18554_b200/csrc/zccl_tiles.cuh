// Compression of binary32 in one launch: included by zccl_codec.cu inside its unnamed namespace.
//
// A CTA of four warps takes a tile, warp rd its round rd (32 blocks, one per lane).  A round comes in by one tensor copy,
// is encoded in place, and waits in its stage until the tile's place in the stream is known; then each warp stores its
// own piece.  The place is the sum of the sizes of the tiles in front, which every CTA finds by itself in ONE round
// trip: it keeps the sum up to the group of 32 tiles its last tile was in, so it adds the groups since (one
// accumulator per group, one lane each) and the tiles of the own group in front (one state per tile, one lane each).
// The trip runs while the CTA's next tile is encoded, so a launch of many tiles hardly ever waits for it.
//
// Tiles are handed out in the order in which CTAs ask for them (a ticket), so a CTA only ever waits for tiles that
// running CTAs hold; a launch of no more tiles than resident CTAs gives CTA b tile b (CTAs are dispatched in that
// order).  Every wait is bounded and reported.

// ------------------------------------------------------------------------------------------------ one block

// Two products, each rounded once.  Written as a fused multiply-add of minus zero, because the compiler contracts a
// packed product and a packed addition behind it into one packed fused multiply-add whatever --fmad says (30 % of the
// hop's sums were off by one unit in the last place); an addend that it cannot know (minus zero as the product
// of the positive step or reciprocal with -0.0f) leaves it nothing to contract.  x * y + (-0) is x * y, signs included.
__device__ __forceinline__ float2 product2(float2 x, float2 y, float2 neg_zero2) { return __ffma2_rn(x, y, neg_zero2); }
__device__ __forceinline__ float negative_zero(float positive) { return __fmul_rn(positive, -0.0f); }

// Deltas of the codes of the block in this lane's row of a stage against the element in front (xprev): magnitudes packed
// 32 / N to a word for the N-bit transpose (word i, field h = element N h + i), sign word, code length (more than
// 16 stands for anything this route does not cover).
//
// c = x r + 1.5 * 2^23 rounds x r to the nearest integer, ties to even, while |x r| < 2^22.  That needs a check only
// for the element in front: with |xprev r| < 2^21 and code lengths of at most 16 (found from the OR of the
// magnitudes, exponent bits included, so that a delta of 2^23 or more, or a NaN, shows up as a long code) no
// element of the block can be further away than 2^21 + 32 * 2^16 = 2^22.
template <int N>
struct BlockCode {
    uint32_t w[N];
    uint32_t sign, L;
    float t_front;    // xprev * r
    float t_max;      // N = 16: the largest |x r|; N = 8: not computed
};
template <int N>
__device__ __forceinline__ void block_codes(const char* row, uint32_t sw, float xprev, float r, float neg_zero, BlockCode<N>& o)
{
    const float tp = __fmul_rn(xprev, r);
    float cp = __fadd_rn(tp, kRoundMagic);
    const float2 r2 = make_float2(r, r), nz2 = make_float2(neg_zero, neg_zero), magic2 = make_float2(kRoundMagic, kRoundMagic);
    float tm = 0.0f;
    uint32_t orb = 0, sg = 0;
#pragma unroll
    for (int h = 0; h < 32 / N; ++h) {
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(row + ((16u * (uint32_t)(h * (N / 4) + q)) ^ sw));
            const float2 t01 = product2(make_float2(v.x, v.y), r2, nz2), t23 = product2(make_float2(v.z, v.w), r2, nz2);
            if (N == 16) tm = fmaxf(fmaxf(fmaxf(tm, fabsf(t01.x)), fabsf(t01.y)), fmaxf(fabsf(t23.x), fabsf(t23.y)));
            const float2 c01 = __fadd2_rn(t01, magic2), c23 = __fadd2_rn(t23, magic2);
            const float cs[4] = {c01.x, c01.y, c23.x, c23.y};
            uint32_t m[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float d = __fsub_rn(cs[e], cp);
                cp = cs[e];
                m[e] = __float_as_uint(__fadd_rn(fabsf(d), kTwo23));
                sg = __funnelshift_l(__float_as_uint(d), sg, 1);     // sign of element j ends up in bit 31 - j
            }
            orb |= m[0] | m[1];
            orb |= m[2] | m[3];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = 4 * q + e;
                if (h == 0) o.w[i] = m[e];
                else if (N == 16) o.w[i] = prmt(o.w[i], m[e], 0x5410u);
                else o.w[i] = prmt(o.w[i], m[e], h == 1 ? 0x0040u : h == 2 ? 0x0410u : 0x4210u);
            }
        }
    }
    o.sign = __brev(sg);
    o.L = 32u - (uint32_t)__clz((int)(orb ^ 0x4B000000u));
    if (!(fabsf(tp) < 2097152.0f)) o.L = 32u;
    o.t_front = tp;
    o.t_max = tm;
}

// The same with integers for a block of a round whose codes the fp32 pass does not cover: any code length, codes up to
// 2^30 (the definition itself).  The planes come back transposed.  Rare.
struct WideBlock {
    uint32_t w[32];
    uint32_t sign, L;
    float tmax;       // largest |x r|, that of the element in front included (the general route always looked at it too)
};
__device__ __forceinline__ void block_codes_wide(const char* row, uint32_t sw, float xprev, float r, WideBlock& o)
{
    const float tp = __fmul_rn(xprev, r);
    float tm = fabsf(tp);
    uint32_t qp = (uint32_t)__float2int_rn(tp), sg = 0, ob = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const float t = __fmul_rn(*reinterpret_cast<const float*>(row + ((16u * (uint32_t)(j >> 2)) ^ sw) + 4 * (j & 3)), r);
        tm = fmaxf(tm, fabsf(t));
        const uint32_t q = (uint32_t)__float2int_rn(t);
        const int32_t dd = (int32_t)(q - qp);
        qp = q;
        const uint32_t sm = (uint32_t)(dd >> 31);
        o.w[j] = (((uint32_t)dd ^ sm) - sm) & 0x7FFFFFFFu;   // |delta|; the mask only matters after a range error
        ob |= o.w[j];
        sg = __funnelshift_l((uint32_t)dd, sg, 1);
    }
    o.L = code_length(ob);
    o.sign = __brev(sg);
    o.tmax = tm;
    bit_transpose<32>(o.w);
}

// A round's payload: block b's sign word and planes behind those of the blocks in front (word 0 = sign word of the first
// block that has any), and one code-length byte per block beside it.  `refill` is called once by all lanes
// when the rows have been read for the last time.  (The last lane may write up to 16 words beyond the
// payload.)
// Out of line, without the hook (a closure handed to an out-of-line function puts what it captures into local memory).
struct RoundOut {
    uint32_t words;
    uint32_t status;
};
__device__ __noinline__ RoundOut encode_round_wide(const float* stage, float xprev, bool active, float r, unsigned char* lens, int lane, uint32_t* dst)
{
    RoundOut o;
    o.status = 0;
    const uint32_t sw = ((uint32_t)lane & 7u) << 4;
    WideBlock b;
    block_codes_wide(reinterpret_cast<const char*>(stage) + 128 * lane, sw, xprev, r, b);
    const uint32_t L = active ? b.L : 0u;
    if (active) {
        if (!(b.tmax < 1073741824.0f)) o.status = kStRange;
        else if (b.tmax > 32768.5f) o.status = kStPrecision;
    }
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    o.words = __shfl_sync(kFull, incl, 31);
    uint32_t* d = dst + (incl - nw);
    lens[lane] = (unsigned char)L;
    if (L) {
        d[0] = b.sign;
#pragma unroll
        for (int k = 0; k < 31; ++k)
            if ((uint32_t)k < L) d[1 + k] = b.w[k];
    }
    return o;
}

// The round's image: `w` the packed magnitudes, L the lane's code length, `longest` the round's.
template <int N, class Refill>
__device__ __forceinline__ uint32_t write_round(uint32_t (&w)[N], uint32_t sign, uint32_t L, uint32_t longest, uint32_t* payload, unsigned char* lens,
                                                int lane, Refill&& refill)
{
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    const uint32_t words = __shfl_sync(kFull, incl, 31);
    refill();       // (its warp barrier stands between the last reads of the rows and the first stores)
    volatile uint32_t* dst = payload + (incl - nw);   // volatile: the order of the stores matters, see below
    bit_transpose<N>(w);
    lens[lane] = (unsigned char)L;
    if (L) {   // from the last plane down: what a lane writes beyond its own code length is overwritten by the lane behind it
        if (N == 16 && longest > 12u) {
#pragma unroll
            for (int k = N - 1; k >= 12; --k) dst[1 + k] = w[k];
        }
        if (N == 16) {
#pragma unroll
            for (int k = (N == 16 ? 11 : 0); k >= 8; --k) dst[1 + k] = w[k];
        }
        if (longest > 4u) {
#pragma unroll
            for (int k = 7; k >= 4; --k) dst[1 + k] = w[k];
        }
#pragma unroll
        for (int k = 3; k >= 0; --k) dst[1 + k] = w[k];
        dst[0] = sign;
    }
    return words;
}
// One width class; ~0 with nothing stored and `refill` not called when a code is longer than N (or, N = 16, not covered).
template <int N, class Refill>
__device__ __forceinline__ uint32_t encode_round_class(const float* stage, float xprev, bool active, float r, float neg_zero, unsigned char* lens,
                                                       int lane, uint32_t& status, uint32_t& longest, uint32_t* payload, Refill&& refill)
{
    const char* row = reinterpret_cast<const char*>(stage) + 128 * lane;
    const uint32_t sw = ((uint32_t)lane & 7u) << 4;
    BlockCode<N> b;
    block_codes<N>(row, sw, xprev, r, neg_zero, b);
    const uint32_t L = active ? b.L : 0u;
    longest = __reduce_max_sync(kFull, L);
    if (longest > (uint32_t)N) return ~0u;
    // a code beyond 2^15 needs, at code lengths up to 8, an element in front beyond 2^15 - 32 * 2^8
    if (N == 16) {
        if (b.t_max > 32768.5f) status |= kStPrecision;
    } else if (__any_sync(kFull, fabsf(b.t_front) > 24000.0f) && block_tmax(row, sw, r) > 32768.5f) status |= kStPrecision;
    return write_round<N>(b.w, b.sign, L, longest, payload, lens, lane, refill);
}
// The narrow class first unless the warp's round before needed the wide one (`wide`).  A round with longer codes goes
// straight to its slot in global memory (bit 31 of the result).
template <class Refill>
__device__ __forceinline__ uint32_t encode_round_staged(float* stage, float xprev, bool active, float r, float neg_zero, unsigned char* lens,
                                                        int lane, bool& wide, uint32_t& status, float* image, uint32_t* slot, Refill&& refill)
{
    uint32_t* payload = reinterpret_cast<uint32_t*>(image) + 8;
    uint32_t words = ~0u, longest = 0;
    if (!wide) words = encode_round_class<8>(stage, xprev, active, r, neg_zero, lens, lane, status, longest, payload, refill);
    if (words == ~0u) {
        words = encode_round_class<16>(stage, xprev, active, r, neg_zero, lens, lane, status, longest, payload, refill);
        if (words == ~0u) {
            const RoundOut o = encode_round_wide(stage, xprev, active, r, reinterpret_cast<unsigned char*>(slot), lane, slot + 8);
            refill();
            status |= o.status;
            return o.words | 0x80000000u;
        }
        wide = longest > 8u;
    }
    __syncwarp();   // the words written by all lanes are visible to the one that stores them
    return words;
}

// ------------------------------------------------------------------------------------------------ places

// Where a tile belongs.
struct TileRef {
    uint32_t t;          // number within the launch (kNoTile: none)
    uint32_t begin;      // its job's first tile
    int job;
};
constexpr uint32_t kNoTile = 0xFFFFFFFFu;
template <class JB>
__device__ __forceinline__ uint32_t tile_length(const JB& jb, const TileRef& at, bool valid)
{
    const unsigned long long n = jb.job[at.job].n, start = (unsigned long long)(at.t - at.begin) * kTile;
    if (!n || !valid) return 0u;
    return (uint32_t)((n - start < (unsigned long long)kTile) ? (n - start) : kTile);
}

// What a CTA keeps between its tiles (in shared memory: a different warp of it may look up each tile).
struct PlaceBase {
    uint32_t job_begin;  // the job it belongs to
    uint32_t group;      // groups of that job that are summed
    uint32_t words;      // their words
};
// The loads of one look-up: the lane's share of the own group's tiles and of the groups since the base.
struct PlaceTrip {
    unsigned long long tile_st, group_st;
};
__device__ __forceinline__ uint32_t group_slot0(uint32_t begin, int job) { return (begin >> 5) + (uint32_t)job; }

__device__ __forceinline__ PlaceTrip place_issue(const Workspace& ws, const TileRef& at, uint32_t first_group, uint32_t epoch, int lane)
{
    PlaceTrip tr;
    const uint32_t rel = at.t - at.begin, g = rel >> 5;
    tr.tile_st = (uint32_t)lane < (rel & 31u) ? ld_state(ws.tile_state + at.begin + (g << 5) + (uint32_t)lane) : pack_state(epoch, 0u, 0u);
    tr.group_st = first_group + (uint32_t)lane < g ? ld_state(ws.group_acc + group_slot0(at.begin, at.job) + first_group + (uint32_t)lane) : (32ull << 40);
    return tr;
}
// The tile's first word within its job's blobs; false when a size in front of it was not published in time.  `tr` was
// issued with the base's group.
__device__ __forceinline__ bool place_finish(const Workspace& ws, const TileRef& at, PlaceBase& base, PlaceTrip tr, uint32_t epoch, int lane,
                                             uint32_t& words)
{
    const uint32_t g = (at.t - at.begin) >> 5;
    uint32_t first = base.job_begin == at.begin ? base.group : 0u, sum = base.job_begin == at.begin ? base.words : 0u;
    for (int polls = 0;;) {
        const bool groups_in = (uint32_t)(tr.group_st >> 40) == 32u, tile_in = (uint32_t)(tr.tile_st >> 33) == epoch;
        const bool all_groups = __all_sync(kFull, groups_in);
        if (all_groups && g - first > 32u) {          // more groups than lanes since the base: take these, then the next
            sum += __reduce_add_sync(kFull, (uint32_t)tr.group_st);
            first += 32u;
        } else if (all_groups && __all_sync(kFull, tile_in)) {
            sum += __reduce_add_sync(kFull, (uint32_t)tr.group_st);
            base.job_begin = at.begin; base.group = g; base.words = sum;
            words = sum + __reduce_add_sync(kFull, (uint32_t)tr.tile_st);
            return true;
        } else if (++polls > 4) {
            if (polls > (kSpinLimit >> 4)) return false;
            __nanosleep(polls < 64 ? 40u : 400u);
        }
        tr = place_issue(ws, at, first, epoch, lane);
    }
}

// ------------------------------------------------------------------------------------------------ shared front and back

constexpr int kTileWarps = kRoundsPerTile;
constexpr int kTileThreads = 32 * kTileWarps;

// Tells the launch the size of a tile (one thread).
__device__ __forceinline__ void publish_tile(const Workspace& ws, const TileRef& at, uint32_t words, uint32_t epoch)
{
    if (at.t == ws.skip_publish) return;
    st_state(ws.tile_state + at.t, pack_state(epoch, 0u, words));
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(ws.group_acc + group_slot0(at.begin, at.job) + ((at.t - at.begin) >> 5)),
                 "l"((1ull << 40) | (unsigned long long)words) : "memory");
}

// Called by one warp of a CTA when the CTA has looked up its last tile: the last CTA of the launch to get here re-arms
// the workspace, while others are still storing.
__device__ __forceinline__ void rearm_tiles(const Workspace& ws, uint32_t warps, uint32_t groups_used, uint32_t epoch, int lane)
{
    uint32_t last = 0;
    if (lane == 0) {
        __threadfence();
        last = atomicAdd(ws.done, 1u) == warps - 1u ? 1u : 0u;
    }
    if (!__shfl_sync(kFull, last, 0)) return;
    for (uint32_t k = (uint32_t)lane; k < groups_used; k += 32u) ws.group_acc[k] = 0ull;
    const uint32_t e = (epoch + 1u) & 0x7FFFFFFFu;
    if (e == 0) {   // the counter wraps (once in 2^31 launches): no state of an earlier launch may look current again
        for (uint32_t k = (uint32_t)lane; k < ws.max_tiles; k += 32u) st_state(ws.tile_state + k, 0ull);
        __threadfence();
    }
    __syncwarp();
    if (lane == 0) {
        *ws.done = 0;
        *ws.ticket = 0;
        *ws.epoch = e ? e : 1u;
    }
}

// For warps that mostly wait: rests between polls.
__device__ __forceinline__ bool mbar_wait_resting(unsigned long long* bar, uint32_t parity)
{
    for (int it = 0; it < kSpinLimit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        __nanosleep(300);
    }
    return false;
}

// ------------------------------------------------------------------------------------------------ compress, step 1
//
// A launch of many tiles: the CTA's four warps take the four rounds of a tile, the CTAs take the tiles in turn.  A round
// comes in by one tensor copy (kEncStages - 1 rounds ahead), is encoded in place and leaves by one bulk store to its
// slot, with its size; place_kernel turns the slots into the stream.  No warp waits for another.

template <int CAP>
struct RoundCursor {          // the walk over a launch's tiles, as the warp of round rd sees it
    uint32_t t;               // tile of the launch
    uint32_t u;               // the warp's round within the job
    uint32_t full, some;      // rounds of the job that are full, that have elements
    uint32_t begin, end;      // the job's tiles
    int job;
    const float* x;
};

template <int CAP>
__global__ void __launch_bounds__(kCodecThreads, kRoundCtas) encode_rounds_kernel(const __grid_constant__ JobBatchT<CAP> jb,
                                                                                 const __grid_constant__ TileMapsT<CAP> maps, Workspace ws,
                                                                                 Params hp, int use_dev_params)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    RoundWarpSharedT<kEncStages>& sh = reinterpret_cast<RoundWarpSharedT<kEncStages>*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u))[warp];
    const uint32_t rd = (uint32_t)warp;
    // Before the kernel in front on the stream is waited for: the warp's first two rounds are asked into L2.  (A prefetch
    // only moves lines into L2, which stays coherent with whatever that kernel still writes.)
    if (lane == 0) {
        for (uint32_t t = blockIdx.x, k = 0; k < 2 && t < jb.total_tiles; ++k, t += gridDim.x) {
            const Job& q = jb.job[CAP == 1 ? 0 : find_job(jb, t)];
            const unsigned long long e = (unsigned long long)(t - q.tile_begin) * kTile + (unsigned long long)rd * kRound;
            if (q.x && (((uintptr_t)q.x) & 15u) == 0 && e + kRound <= q.n) bulk_prefetch_l2(q.x + e, 4u * kRound);
        }
#pragma unroll
        for (int k = 0; k < kEncStages; ++k) mbar_init(&sh.bar[k], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    pdl_enter();
    Params prm = hp;
    if (use_dev_params) prm = *ws.params;
    const float r = prm.r, nz = negative_zero(prm.r);
    uint32_t status = 0;

    auto enter = [&](RoundCursor<CAP>& c) {      // the job of tile c.t
        c.job = CAP == 1 ? 0 : find_job(jb, c.t);
        const Job& q = jb.job[c.job];
        c.begin = q.tile_begin;
        c.end = CAP > 1 && c.job + 1 < jb.count ? jb.job[c.job + 1].tile_begin : jb.total_tiles;
        const bool bulk = (((uintptr_t)q.x) & 15u) == 0;
        c.some = prm.valid ? (uint32_t)((q.n + kRound - 1) / kRound) : 0u;
        c.full = bulk && prm.valid ? (uint32_t)(q.n / kRound) : 0u;
        c.x = q.x;
        c.u = 4u * (c.t - c.begin) + rd;
    };
    auto advance = [&](RoundCursor<CAP>& c) {
        c.t = c.t + gridDim.x < c.t ? kNoTile : c.t + gridDim.x;
        c.u += 4u * gridDim.x;
        if (CAP > 1 && c.t >= c.end && c.t < jb.total_tiles) enter(c);
    };
    // asks for the round under the cursor into stage st (rounds that the copy engine cannot bring: nothing)
    auto request = [&](const RoundCursor<CAP>& c, uint32_t st, float& front) {
        if (lane == 0) {
            if (c.t < jb.total_tiles && c.u < c.full) {
                tensor_load_round(sh.stage[st], &sh.bar[st], &maps.m[c.job], 32u * c.u);
                if (rd) front = __ldg(c.x + (size_t)c.u * kRound - 1);
            } else mbar_arrive(&sh.bar[st]);
        }
    };
    RoundCursor<CAP> cur, ahead;
    cur.t = blockIdx.x;
    enter(cur);
    ahead = cur;
    float front[kEncStages - 1];               // lane 0: the elements in front of the rounds on their way
#pragma unroll
    for (int k = 0; k + 1 < kEncStages; ++k) {
        front[k] = 0.0f;
        request(ahead, k, front[k]);
        advance(ahead);
    }
    uint32_t st = 0, phase = 0;
    bool wide = false;
    while (cur.t < jb.total_tiles) {
        const uint32_t ul = 4u * cur.t + rd;      // the round within the launch
        float* stage = sh.stage[st];
        if (!mbar_wait(&sh.bar[st], phase)) { status |= kStTimeout; break; }
        float front_new = 0.0f;
        // the stage the next request goes to was encoded in place and sent off one step ago: the copy engine has to be through
        // with reading it, which by the time this round's rows are read and sized it mostly is
        auto refill = [&]() {
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
            request(ahead, st == 0 ? kEncStages - 1u : st - 1u, front_new);
        };
        uint32_t words = 0;
        if (cur.u < cur.some) {
            bool active = true;
            float xprev0 = front[0];
            if (cur.u >= cur.full) {
                const unsigned long long e = (unsigned long long)cur.u * kRound, n = jb.job[cur.job].n;
                const uint32_t left = (uint32_t)(n - e < (unsigned long long)kRound ? n - e : kRound);
                load_round_ragged(stage, cur.x + e, 0, left, lane);
                if (rd) xprev0 = __ldg(cur.x + e - 1);
                active = 32u * (uint32_t)lane < left;
                __syncwarp();
            }
            uint32_t* slot = ws.slots + (size_t)ul * kRoundSlotWords;
            const float first = stage[0];
            const float xprev = lane ? read_last_of_row(stage, (uint32_t)lane - 1u) : (rd ? xprev0 : first);
            // in place: the stage becomes the round's slot image (code-length bytes, payload from word 8 on)
            words = encode_round_staged(stage, xprev, active, r, nz, reinterpret_cast<unsigned char*>(stage), lane, wide, status, stage, slot, refill);
            if (lane == 0) {
                if (!(words >> 31)) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(slot), "r"(smem_u32(stage)),
                                 "r"((32u + 4u * words + 15u) & ~15u) : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
                words &= 0x7FFFFFFFu;
                if (rd == 0) ws.outliers[cur.t] = __float2int_rn(__fmul_rn(first, r));
                asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(ws.group_acc + (cur.begin >> 5) + (uint32_t)cur.job + (cur.u >> 7)),
                             "l"((unsigned long long)words) : "memory");
            }
        } else refill();                          // a round beyond the end, or a job without elements
        if (lane == 0) ws.round_words[ul] = words;
#pragma unroll
        for (int k = 0; k + 2 < kEncStages; ++k) front[k] = front[k + 1];
        front[kEncStages - 2] = front_new;
        advance(cur);
        advance(ahead);
        st = st + 1 == kEncStages ? 0u : st + 1;
        if (st == 0) phase ^= 1u;
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // the stores have read shared memory and are complete
    if (status) atomicOr(ws.status, status);
}
