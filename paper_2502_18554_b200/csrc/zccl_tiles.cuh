// Compression of binary32: included by zccl_codec.cu inside its unnamed namespace.
//
// A CTA of four warps takes a tile, warp rd its round rd (32 blocks, one per lane).  A round comes in by one tensor copy
// and is encoded in place.  In a launch of few tiles (encode_tiles_kernel, a CTA per tile) it waits in its stage until
// the tile's place in the stream is known, which the CTAs find out by themselves (see "places"), and each warp stores its
// own piece; CTAs take their tiles in the order in which they start, so a CTA only ever waits for CTAs that run already.
// Every wait is bounded and reported.  Launches of many tiles: zccl_stream.cuh.

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
// (`get(k)`: elements 4 k .. 4 k + 3 of the block.)
template <int N, class Get>
__device__ __forceinline__ void block_codes(Get&& get, float xprev, float r, float neg_zero, BlockCode<N>& o)
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
            const float4 v = get((uint32_t)(h * (N / 4) + q));
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
    __syncwarp();   // every lane has read its row: dst may be the stage
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

// The round's image: `w` the packed magnitudes, L the lane's code length, `longest` the round's.  `where`, called once by
// all lanes with the payload's words, says where they go.
// ONE: the warps of the launch have one round each, see plain_scan.
template <int N, bool ONE, class Where>
__device__ __forceinline__ uint32_t write_round(uint32_t (&w)[N], uint32_t sign, uint32_t L, uint32_t longest, unsigned char* lens, int lane, Where&& where)
{
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = ONE ? plain_scan(nw, lane) : warp_incl_scan(nw, lane);
    const uint32_t words = __shfl_sync(kFull, incl, 31);
    uint32_t* payload = where(words);                 // (its warp barrier stands between the last reads of the rows and the first stores)
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
// One width class; ~0 with nothing stored and `where` not called when a code is longer than N (or, N = 16, not covered).
template <int N, bool ONE, class Where>
__device__ __forceinline__ uint32_t encode_round_class(const float* stage, float xprev, bool active, float r, float neg_zero, unsigned char* lens,
                                                       int lane, uint32_t& status, uint32_t& longest, Where&& where)
{
    const char* row = reinterpret_cast<const char*>(stage) + 128 * lane;
    const uint32_t sw = ((uint32_t)lane & 7u) << 4;
    BlockCode<N> b;
    const uint32_t at = smem_u32(row) + sw;
    block_codes<N>([&](uint32_t k) { return ONE ? *reinterpret_cast<const float4*>(row + ((16u * k) ^ sw)) : ld_shared4(at ^ (16u * k)); }, xprev, r, neg_zero, b);
    const uint32_t L = active ? b.L : 0u;
    longest = __reduce_max_sync(kFull, L);
    if (longest > (uint32_t)N) return ~0u;
    // a code beyond 2^15 needs, at code lengths up to 8, an element in front beyond 2^15 - 32 * 2^8
    if (N == 16) {
        if (b.t_max > 32768.5f) status |= kStPrecision;
    } else if (__any_sync(kFull, fabsf(b.t_front) > 24000.0f) && block_tmax(row, sw, r) > 32768.5f) status |= kStPrecision;
    return write_round<N, ONE>(b.w, b.sign, L, longest, lens, lane, where);
}
// The narrow class first unless the warp's round before needed the wide one (`wide`); ~0 when neither covers the round.
template <class Where>
__device__ __forceinline__ uint32_t encode_round_classes(const float* stage, float xprev, bool active, float r, float neg_zero, unsigned char* lens,
                                                         int lane, bool& wide, uint32_t& status, Where&& where)
{
    uint32_t words = ~0u, longest = 0;
    if (!wide) words = encode_round_class<8, false>(stage, xprev, active, r, neg_zero, lens, lane, status, longest, where);
    if (words == ~0u) {
        words = encode_round_class<16, false>(stage, xprev, active, r, neg_zero, lens, lane, status, longest, where);
        if (words != ~0u) wide = longest > 8u;
    }
    return words;
}
// The same with longer codes to wide_payload and wide_lens (bit 31 of the result), for which the stage itself will do.
template <bool ONE, class Refill>
__device__ __forceinline__ uint32_t encode_round_staged(float* stage, float xprev, bool active, float r, float neg_zero, unsigned char* lens,
                                                        int lane, bool& wide, uint32_t& status, uint32_t* payload, unsigned char* wide_lens, uint32_t* wide_payload,
                                                        Refill&& refill)
{
    auto where = [&](uint32_t) { refill(); return payload; };
    uint32_t words = ~0u, longest = 0;
    if (!wide) words = encode_round_class<8, ONE>(stage, xprev, active, r, neg_zero, lens, lane, status, longest, where);
    if (words == ~0u) {
        words = encode_round_class<16, ONE>(stage, xprev, active, r, neg_zero, lens, lane, status, longest, where);
        if (words == ~0u) {
            const RoundOut o = encode_round_wide(stage, xprev, active, r, wide_lens, lane, wide_payload);
            refill();
            status |= o.status;
            return o.words | 0x80000000u;
        }
        wide = longest > 8u;
    }
    __syncwarp();   // the words written by all lanes are visible to the one that stores them
    return words;
}

constexpr uint32_t kNoTile = 0xFFFFFFFFu;
constexpr int kTileWarps = kRoundsPerTile;
constexpr int kTileThreads = 32 * kTileWarps;


// ------------------------------------------------------------------------------------------------ places
//
// A tile's place in its stream is the sum of the sizes of the job's tiles in front.  A CTA of four coding warps that has
// one tile publishes its size twice, as the tile's state and added to the accumulator of its group of 32 tiles (which
// counts the tiles too), and finds its place with one load per lane: warp 0 looks at the states of the tiles in front
// within the group, warps 1 and 2 at the accumulators of the groups in front, back to a group whose inclusive sum warp 3
// looks at (a tile that closes a group publishes that in its state, which nobody else needs).  Inclusive sums are looked
// for kPlaceGroups groups back, more tiles than a GPU holds CTAs, so they are there long before: a place costs one
// round trip after the last size is there.  (Groups summed up by their last tile: one more round trip, 512 tiles placed
// after 5.4 us instead of 3.6.  Every tile's state looked at by everybody, up to eight per lane: 7.7 us, the polls get
// into each other's way.)  Launches of a CTA per tile have at most seven tiles per SM now, which is 33 groups on 148 SMs, so no tile
// looks that far back; the general form stays, since with what is not reached left out compressions took longer (256 tiles 5.4 us
// instead of 4.8, 888 tiles 8.4 instead of 8.0; hops of 256 tiles 6.8 instead of 7.15) and why was not found.
//
// A CTA only ever waits for the CTAs of lower tiles of its job.  CUDA promises no order in which the CTAs of a grid start,
// so a CTA takes the job's next tile when it starts (take_tile): those of lower tiles run by then, whatever share of the
// device the launch gets, and the one with the lowest unfinished tile waits for nobody.  Launches of one cluster, whose
// CTAs are scheduled together, take their tiles by their numbers.  Every wait is bounded and reported.

constexpr uint32_t kPlaceGroups = 40;

// The tile of this CTA within a job that has `tiles`, in a launch of a CTA per tile: one thread takes a number in front of
// the wait for the launch in front, which can cover the round trip.  Behind that wait one thread that is not in a hurry
// lets the launch behind start (tile_taken; no other thread does), when the counter is in order for that one: the CTA
// with the last number puts it back to 0.  By their numbers, as far as CTAs do start in that order, a hop of 25 tiles takes
// 6.8 us instead of 7.0, of 256 tiles 7.0 instead of 8.0, compressions of 16 and 256 tiles 3.7 and 5.3 instead of 4.0 and
// 5.1: less for the round trip than because a tile then stays on one SM from call to call.  Counters that go around by
// themselves, by atomicInc: 8 x 2^21 Allreduce 78.9 us instead of 74.3, 8 x 2^18 Allgather 36.6 instead of 35.2.  Put back
// in front of the wait: 75.8 and 36.2, compression of 16 tiles 3.3.
__device__ __forceinline__ uint32_t take_tile(const Workspace& ws, uint32_t job, uint32_t tiles)
{
    return tiles == 1 ? 0u : min(atomicAdd(ws.next_tile + job * kTileCounterStride, 1u), tiles - 1u);
}
__device__ __forceinline__ uint32_t taken_tile(const Workspace& ws, uint32_t tiles, uint32_t taken)
{
    const uint32_t t = taken + ws.first_tile;
    return t < tiles ? t : t - tiles;
}
__device__ __forceinline__ void tile_taken(const Workspace& ws, uint32_t job, uint32_t tiles, uint32_t taken)
{
    if (tiles > 1 && taken == tiles - 1u) {
        atomicExch(ws.next_tile + job * kTileCounterStride, 0u);
        __threadfence();
    }
    pdl_release();
}

struct PlaceShared {
    alignas(16) uint32_t words[kTileWarps];    // payload words of the four rounds
    alignas(16) uint32_t part[kTileWarps];     // the warps' shares of the sum
    uint32_t failed;                           // zero at the start
    uint32_t taken;                            // what take_tile gave
};

// Adds up what the lanes' states say (p = nullptr: nothing) once each is there: a tile's carries this launch's number (and,
// `incl`, an inclusive sum), a group's counts 32 tiles (`group`).
__device__ __forceinline__ bool sum_states(const unsigned long long* p, uint32_t epoch, bool group, bool incl, uint32_t& sum)
{
    unsigned long long st = p ? ld_state(p) : 0ull;
    bool ok = true;
    for (int polls = 0; p && (group ? (uint32_t)(st >> 40) != 32u : (uint32_t)(st >> 33) != epoch || (incl && !((st >> 32) & 1ull))); ++polls) {
        if (polls > (kSpinLimit >> 4)) { ok = false; break; }
        if (polls > 8) __nanosleep(polls < 64 ? 40u : 400u);
        st = ld_state(p);
    }
    sum = __reduce_add_sync(kFull, (uint32_t)st);
    return __all_sync(kFull, ok);
}

// The four coding warps of a CTA together (named barrier 1): their rounds' `words` give the tile's size, and the result is
// the tile's first word within the job's blobs.  `total`, `offset`: the tile's words, and the payload words in front of the
// warp's round; `placed`: false when a wait ran out.
__device__ __forceinline__ uint32_t find_place(const Workspace& ws, PlaceShared& sh, uint32_t begin, uint32_t job, uint32_t tile, uint32_t head_words,
                                               uint32_t words, uint32_t epoch, uint32_t rd, int lane, uint32_t& total, uint32_t& offset, bool& placed)
{
    if (lane == 0) sh.words[rd] = words;
    asm volatile("bar.sync 1, 128;" ::: "memory");
    const uint4 w4 = *reinterpret_cast<const uint4*>(sh.words);
    offset = (rd > 0 ? w4.x : 0u) + (rd > 1 ? w4.y : 0u) + (rd > 2 ? w4.z : 0u);
    total = head_words + w4.x + w4.y + w4.z + w4.w;
    unsigned long long* tiles = ws.tile_state + begin;
    unsigned long long* groups = ws.group_sums + (epoch & 1u) * (uint32_t)group_slots(ws.state_tiles) + (begin >> 5) + job;
    const uint32_t g = tile >> 5, in_group = tile & 31u, gb = g > kPlaceGroups ? g - kPlaceGroups : 0u, k = gb + (uint32_t)lane;
    const bool tell = begin + tile != ws.skip_publish, closes = in_group == 31u;
    if (rd == 0 && lane == 0 && tell) {
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(groups + g), "l"((1ull << 40) | (unsigned long long)total) : "memory");
        if (!closes) st_state(tiles + tile, pack_state(epoch, 0u, total));
    }
    const unsigned long long* p = nullptr;
    if (rd == 0) p = (uint32_t)lane < in_group ? tiles + 32u * g + (uint32_t)lane : nullptr;
    else if (rd == 1) p = k < g ? groups + k : nullptr;
    else if (rd == 2) p = k + 32u < g ? groups + k + 32u : nullptr;
    else p = lane == 0 && gb ? tiles + 32u * gb - 1u : nullptr;
    uint32_t sum;
    const bool ok = sum_states(p, epoch, rd == 1 || rd == 2, rd == 3, sum);
    if (lane == 0) {
        sh.part[rd] = sum;
        if (!ok) sh.failed = 1;
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    const uint4 p4 = *reinterpret_cast<const uint4*>(sh.part);
    const uint32_t place = p4.x + p4.y + p4.z + p4.w;
    placed = sh.failed == 0;
    if (rd == 0 && lane == 0 && closes && tell && placed) st_state(tiles + tile, pack_state(epoch, 1u, place + total));
    return place;
}

// At the end of the look-ups (one warp): the CTA of a job's last tile, which by their sizes has seen that every CTA of
// the job has read the launch counter, moves it on; with several jobs the last of them does.  The accumulators come in
// two sets, used in turn: the set of the next launch, which the launch before this one used, is cleared.  So no CTA has
// to be counted and nothing waits at the end of a launch (counting every CTA cost 1.5 us there).  Only when the counter
// wraps, once in 2^31 launches, every CTA is counted and the last one clears all states.
// `tiles`: calls of the launch at a wrap of the counter; `jobs`: those that have CTAs, without elements or not (a CTA without
// elements reads the counter and the bound like any other); `used`: accumulators the launch may have touched.
__device__ __forceinline__ void finish_places(const Workspace& ws, uint32_t epoch, bool last_of_job, uint32_t tiles, uint32_t jobs, uint32_t used_now,
                                              const Params& prm, int bound_source, int lane)
{
    uint32_t turn = 0;
    if (lane == 0) {
        if (epoch == 0x7FFFFFFFu) {
            __threadfence();
            turn = atomicAdd(ws.done, 1u) == tiles - 1u ? 1u : 0u;
        } else if (last_of_job) {
            turn = jobs == 1u || atomicAdd(ws.done, 1u) == jobs - 1u ? 1u : 0u;
        }
    }
    if (!__shfl_sync(kFull, turn, 0)) return;
    const uint32_t slots = (uint32_t)group_slots(ws.state_tiles);
    if (epoch == 0x7FFFFFFFu) {
        for (uint32_t k = (uint32_t)lane; k < ws.state_tiles; k += 32u) st_state(ws.tile_state + k, 0ull);
        for (uint32_t k = (uint32_t)lane; k < 2u * slots; k += 32u) ws.group_sums[k] = 0ull;
        if (lane < 2) ws.group_used[lane] = 0;
        __threadfence();
        epoch = 0;
    } else {
        const uint32_t next = (epoch + 1u) & 1u, used = ws.group_used[next];
        for (uint32_t k = (uint32_t)lane; k < used; k += 32u) ws.group_sums[next * slots + k] = 0ull;
        __syncwarp();
        if (lane == 0) {
            ws.group_used[next] = 0;
            ws.group_used[epoch & 1u] = used_now;
        }
    }
    if (lane == 0) {
        settle_bound(ws, prm, bound_source);
        *ws.done = 0;
        *ws.epoch = epoch + 1u;
    }
}

template <class JB>
__device__ __forceinline__ void finish_places(const JB& jb, const Workspace& ws, uint32_t epoch, bool last_of_job, const Params& prm, int bound_source, int lane)
{
    finish_places(ws, epoch, last_of_job, jb.total_tiles, (uint32_t)jb.count, (jb.total_tiles >> 5) + (uint32_t)jb.count + 1u, prm, bound_source, lane);
}

// `words` words from shared memory (or a slot) to anywhere: eight loads, then eight stores.
__device__ __forceinline__ void copy_words(uint32_t* __restrict__ dst, const uint32_t* src, uint32_t words, int lane)
{
    dst += lane;
    src += lane;
    for (uint32_t left = words; left; left = left > 256u ? left - 256u : 0u, src += 256, dst += 256) {
        uint32_t v[8];
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k)
            if (32u * k + (uint32_t)lane < left) v[k] = src[32u * k];
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k)
            if (32u * k + (uint32_t)lane < left) dst[32u * k] = v[k];
    }
}

// The payloads of a tile's four rounds, `words` of each, go to `dst` one behind the other (one warp): eight lanes per round, 16
// bytes per lane and store.  `src`: the payload of the lane's round, lane / 8, in shared memory.
__device__ __forceinline__ void store_payloads(uint32_t* __restrict__ dst, uint4 w4, const uint32_t* src, int lane)
{
    const uint32_t r = (uint32_t)lane >> 3, l = (uint32_t)lane & 7u, words = r == 0 ? w4.x : r == 1 ? w4.y : r == 2 ? w4.z : w4.w;
    dst += (r > 0 ? w4.x : 0u) + (r > 1 ? w4.y : 0u) + (r > 2 ? w4.z : 0u);
    uint32_t head = (uint32_t)(-(int32_t)((uintptr_t)dst >> 2)) & 3u;
    head = head < words ? head : words;
    const uint32_t quads = (words - head) >> 2, tail = (words - head) & 3u;
    if (l < head) dst[l] = src[l];
    if (l < tail) dst[head + 4u * quads + l] = src[head + 4u * quads + l];
    src += head + 4u * l;
    uint4* __restrict__ d4 = reinterpret_cast<uint4*>(dst + head) + l;
    const uint32_t most = __reduce_max_sync(kFull, quads);
    for (uint32_t k = 0; k < most; k += 32u, src += 128, d4 += 32) {
        uint4 v[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
            if (k + 8u * u + l < quads) v[u] = make_uint4(src[32u * u], src[32u * u + 1u], src[32u * u + 2u], src[32u * u + 3u]);
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u)
            if (k + 8u * u + l < quads) d4[8u * u] = v[u];
    }
}

// A warp's share of an encoded tile goes to its place: its payload and its round's code-length words, and (warp 0) what
// goes once per tile.
__device__ __forceinline__ void store_piece(const Job& job, uint32_t tile, uint32_t padw, uint32_t place, uint32_t offset, uint32_t words, uint32_t total,
                                            bool placed, int32_t first_code, const uint32_t* lens, const uint32_t* payload, float eb_abs, float s,
                                            uint32_t rd, int lane, uint32_t& status)
{
    const uint32_t nT = (uint32_t)((job.n + kTile - 1) / kTile);
    const unsigned long long word0 = (unsigned long long)kHeaderWords + nT + place;
    const bool fits = (word0 + total) * 4ull <= job.out_cap;
    if (!fits) status |= kStCapacity;
    if (!placed) status |= kStTimeout;
    if (fits && placed) {
        uint32_t* __restrict__ dst = job.out + word0;
        const uint32_t lw = 8u * rd + (uint32_t)lane;
        if (lane < 8 && lw < padw) dst[1 + lw] = lens[lane];
        if (rd == 0 && lane == 0) {
            dst[0] = (uint32_t)first_code;
            job.out[kHeaderWords + tile] = place + total;
        }
        copy_words(dst + 1 + padw + offset, payload, words, lane);
    }
    if (rd == 0) {
        if (lane == 0 && tile == nT - 1) *job.out_bytes = (size_t)((word0 + total) * 4ull);
        if (tile == 0) write_header(job.out, lane, job.n, eb_abs, s, nT);
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

// ------------------------------------------------------------------------------------------------ compress
//
// A CTA per tile, four warps, a round each: a round comes in by one tensor copy, is encoded in place and waits in its
// stage for the tile's place.
//
// RANGE: the bound is relative and the launch one cluster of at most kRangeTiles CTAs, which find the input's range
// themselves: every CTA looks through its tile in shared memory and leaves its extremes with all others (1024
// elements: 3.4 us in one launch, 5.8 with a range kernel in front).

constexpr uint32_t kRangeTiles = 8;   // the portable size of a cluster
struct alignas(1024) EncodeShared {
    float stage[kTileWarps][kRound];           // a round; then its payload, in place
    uint32_t lens[kTileWarps][8];              // its code-length bytes
    alignas(8) unsigned long long bar[kTileWarps];
    PlaceShared place;
    float2 warp_range[kTileWarps], cta_range[kRangeTiles];   // (min, max)
};

template <int CAP, bool RANGE>
__global__ void __launch_bounds__(kTileThreads, kEncodeCtas) encode_tiles_kernel(const __grid_constant__ JobBatchT<CAP> jb,
                                                                                const __grid_constant__ TileMapsT<CAP> maps, Workspace ws, Params hp,
                                                                                int bound_source)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    EncodeShared& sh = *reinterpret_cast<EncodeShared*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t rd = (uint32_t)tid >> 5;
    const uint32_t j = CAP == 1 ? 0u : (uint32_t)find_job(jb, blockIdx.x);
    const Job& job = jb.job[j];
    const uint32_t begin = job.tile_begin, tiles = (CAP > 1 && j + 1 < (uint32_t)jb.count ? jb.job[j + 1].tile_begin : jb.total_tiles) - begin;
    if (tid == 0) {
        if (!RANGE) sh.place.taken = take_tile(ws, j, tiles);
        sh.place.failed = 0;
    }
    __syncthreads();
    const uint32_t tile = RANGE ? blockIdx.x : taken_tile(ws, tiles, sh.place.taken);
    const unsigned long long n = job.n, start = (unsigned long long)tile * kTile, e = start + (unsigned long long)rd * kRound;
    const bool bulk = (((uintptr_t)job.x) & 15u) == 0 && e + kRound <= n;
    // before the kernel in front on the stream is waited for: the round is asked into L2 (a prefetch only moves lines there;
    // L2 stays coherent with whatever that kernel still writes)
    if (lane == 0) {
        if (bulk) bulk_prefetch_l2(job.x + e, 4u * kRound);
        mbar_init(&sh.bar[rd], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    pdl_wait();
    float* stage = sh.stage[rd];
    if (bulk && lane == 0) tensor_load_round(stage, &sh.bar[rd], &maps.m[j], (uint32_t)(e >> 5));
    if (RANGE) pdl_release();
    else if (tid == kTileThreads - 32) tile_taken(ws, j, tiles, sh.place.taken);
    if (CAP > 1 && n == 0)
        for (uint32_t k = 0; k < ws.store_pause; ++k) __nanosleep(1000);
    const uint32_t epoch = *reinterpret_cast<volatile uint32_t*>(ws.epoch);
    Params prm = hp;
    if (!RANGE) prm = bound_of(ws, hp, bound_source);
    uint32_t status = 0;
    bool there = false;                          // the round is in its stage
    auto arrive = [&]() {
        if (there) return;
        there = true;
        if (!bulk) {
            load_round_ragged(stage, job.x + e, 0, n - e < (unsigned long long)kRound ? (uint32_t)(n - e) : (uint32_t)kRound, lane);
            __syncwarp();
        } else if (!mbar_wait(&sh.bar[rd], 0u)) status |= kStTimeout;
    };
    if (RANGE) {
        float lo = __int_as_float(0x7F800000), hi = __int_as_float(0xFF800000);
        if (e < n) {
            arrive();
            const float4* row = reinterpret_cast<const float4*>(stage) + 8 * lane;   // any order will do
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float4 v = row[k ^ (lane & 7)];
                lo = fminf(fminf(lo, v.x), fminf(v.y, fminf(v.z, v.w)));
                hi = fmaxf(fmaxf(hi, v.x), fmaxf(v.y, fmaxf(v.z, v.w)));
            }
#pragma unroll
            for (int d = 16; d; d >>= 1) {
                lo = fminf(lo, __shfl_xor_sync(kFull, lo, d));
                hi = fmaxf(hi, __shfl_xor_sync(kFull, hi, d));
            }
        }
        if (lane == 0) sh.warp_range[rd] = make_float2(lo, hi);
        __syncthreads();
        if ((uint32_t)tid < gridDim.x) {
            float2 m = sh.warp_range[0];
#pragma unroll
            for (int k = 1; k < kTileWarps; ++k) m = make_float2(fminf(m.x, sh.warp_range[k].x), fmaxf(m.y, sh.warp_range[k].y));
            uint32_t to;                         // this CTA's place in CTA tid's table
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(smem_u32(&sh.cta_range[blockIdx.x])), "r"(tid));
            asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(to), "f"(m.x), "f"(m.y) : "memory");
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
        float2 m = sh.cta_range[0];
        for (uint32_t k = 1; k < gridDim.x; ++k) m = make_float2(fminf(m.x, sh.cta_range[k].x), fmaxf(m.y, sh.cta_range[k].y));
        prm = params_of(hp.eb_abs, m.x <= m.y ? __fsub_rn(m.y, m.x) : 0.0f);
        if (blockIdx.x == 0 && tid == 0) {
            *ws.params = prm;
            if (!prm.valid) status |= kStDegenerate;
        }
    }
    const float r = prm.r, nz = negative_zero(prm.r);
    const uint32_t len = n && prm.valid ? (uint32_t)(n - start < (unsigned long long)kTile ? n - start : kTile) : 0u;
    const uint32_t e0 = rd * (uint32_t)kRound;
    uint32_t words = 0;
    int32_t first_code = 0;
    uint32_t* payload = reinterpret_cast<uint32_t*>(stage);
    unsigned char* lens = reinterpret_cast<unsigned char*>(sh.lens[rd]);
    if (lane < 8) sh.lens[rd][lane] = 0;
    __syncwarp();
    if (e0 < len) {
        const float front = rd ? __ldg(job.x + e - 1) : 0.0f;
        arrive();
        if (job.y) {                             // an uncompressed copy of the input goes along (an Allgather's own contribution)
            store_round_ragged(job.y + e, stage, len - e0 < (uint32_t)kRound ? len - e0 : (uint32_t)kRound, lane);
            __syncwarp();
        }
        const float first = stage[0];
        const float xprev = lane ? read_last_of_row(stage, (uint32_t)lane - 1u) : (rd ? front : first);
        first_code = __float2int_rn(__fmul_rn(first, r));
        bool wide = false;
        words = encode_round_staged<true>(stage, xprev, e0 + 32u * (uint32_t)lane < len, r, nz, lens, lane, wide, status, payload, lens, payload,
                                    [] { __syncwarp(); }) & 0x7FFFFFFFu;
    } else {
        if (bulk) arrive();      // no valid bound: a copy on its way into shared memory has to land before the CTA ends
        if (job.y && e < n) copy_round_plain(job.y + e, job.x + e, n - e, lane);   // a contribution of one's own needs no bound
    }
    if (len) {
        const uint32_t padw = (((len + kBlock - 1) / kBlock) + 3) >> 2;
        uint32_t total, offset;
        bool placed;
        const uint32_t place = find_place(ws, sh.place, begin, j, tile, 1u + padw, words, epoch, rd, lane, total, offset, placed);
        if (rd == kTileWarps - 1) finish_places(jb, ws, epoch, tile + 1u == tiles, prm, bound_source, lane);
        store_piece(job, tile, padw, place, offset, words, total, placed, first_code, sh.lens[rd], payload, prm.eb_abs, prm.s, rd, lane, status);
    } else if (rd == 0) {   // a job without elements, or no valid bound: header and length only
        const bool hdr = prm.valid && job.out_cap >= (unsigned)kHeaderBytes;
        if (lane == 0) *job.out_bytes = hdr ? kHeaderBytes : 0;
        if (prm.valid || epoch == 0x7FFFFFFFu) finish_places(jb, ws, epoch, prm.valid != 0, prm, bound_source, lane);
        else if (lane == 0 && blockIdx.x == 0) settle_bound(ws, prm, bound_source);
        if (hdr) write_header(job.out, lane, 0, prm.eb_abs, prm.s, 0);
    }
    if (status) atomicOr(ws.status, status);
}
