// Compression of many tiles of binary32 in one launch: included by zccl_codec.cu inside its unnamed namespace.
//
// A CTA takes tiles one after the other: four warps encode a round each, a lane a block of 32 elements.  A fifth warp deals
// out the tiles (from a counter, so that a CTA only ever waits for tiles which CTAs hold that run already), asks for each
// with one tensor copy into one of kStreamStages stages, and finds the places of encoded tiles.  A sixth stores them.  A
// coding warp puts its round's payload into a ring of its own, so the tile's stage is free as soon as its rows have been
// read, and the warp that completes a tile publishes its size at once: no coding warp waits for a place but one whose ring is
// full.
//
// What bounds it: from 2^26 values on DRAM (5.8 TB/s of reads and writes at code lengths around 4) and, at code lengths of 10
// and more, how long tiles wait for their places; below that the ramps, and a last tile per CTA that others cannot share.  The
// issue slots are what the two serving warps compete for with the sixteen coding ones of an SM, so what counts there is how few
// instructions a tile costs them.  us, rounds sent to slots of their own in global memory and placed by a second launch / this:
// 2^24 field values at 1e-3 20.4 / 18.6, with a relative bound 33.9 / 32.8; 2^26 smooth 68 / 57; 2^28 field 286 / 207, gradients
// (code lengths 7 to 15; the slots alone moved 660 MB) 352 / 269.
// Tried: serving and storing by one warp 2^28 gradients 325, pieces stored by the coding warps themselves 311; places by two
// tiles' sums at a time and group sums from inclusive ones 48 groups back 333 (273 a tile at a time, 260 with the sum kept from
// the CTA's tile before); five CTAs with rings of 576 words 2^24 27.9 and 2^28 1690 (rings run dry), five or four with one stage
// 26.4 and 28.3; blocks read into registers at once, to free the stage earlier, 22.9.

constexpr int kStreamCtas = 4;
constexpr int kStreamThreads = kTileThreads + 64;
constexpr uint32_t kStreamStages = 2;      // tiles on their way in, or being encoded
constexpr uint32_t kStreamQueue = 8;       // tiles on their way in, being encoded or not yet stored
constexpr uint32_t kStreamRing = 1328;     // payload words of a warp that wait for their places: one round at least, with what write_round writes behind it
constexpr uint32_t kStreamEnd = 3;         // tiles per CTA left to be dealt out from which on numbers are taken late (8 the same; always late: 2^28 field 217 us)
constexpr uint32_t kInStage = 0x80000000u;

struct alignas(16) StreamEntry {
    uint32_t words[kTileWarps];            // payload words of the rounds
    uint32_t at[kTileWarps];               // where they are in the warps' rings (kInStage: in the tile's stage)
    uint32_t lens[kTileWarps][8];          // code-length bytes
    unsigned long long start;              // the tile's first element
    uint32_t tile, job, len;               // within the job; len: its elements
    uint32_t begin;                        // the job's first tile within the launch
    uint32_t kind;                         // kTileNone: no more tiles
    int32_t first_code;
    uint32_t sum;                          // {rounds that are through:8 | their words:24}
    uint32_t bulk;                         // the copy engine brings the tile
    uint32_t total;                        // the tile's words
    uint32_t place;                        // when it is known: the words of the job's tiles in front
    uint32_t late;                         // ... and when the wait for them ran out
};
struct alignas(1024) StreamShared {
    float stage[kStreamStages][kTileWarps][kRound];
    uint32_t ring[kTileWarps][kStreamRing];
    StreamEntry entry[kStreamQueue];
    Params bound;                          // what the serving warp has read, for the storing one
    alignas(8) unsigned long long full[kStreamStages], seen[kStreamStages], empty[kStreamStages], coded[kStreamQueue], known[kStreamQueue], gone[kStreamQueue];
};
static_assert(sizeof(StreamShared) + 2048 <= 228 * 1024 / kStreamCtas, "resident together");

// Has the phase ended?  The same answer to all lanes (a lane by itself may see the end of a phase that its neighbour does not yet).
__device__ __forceinline__ bool mbar_test_warp(unsigned long long* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return __all_sync(kFull, ok != 0);
}

// For the coding and the storing warps, which wait for the serving one, whose own waits have a limit: theirs is beyond that (a few
// seconds against at most 2 kStreamQueue + 1 times a tenth of one), so that a CTA whose places do not come still goes through all its tiles.
__device__ __forceinline__ bool mbar_wait_long(unsigned long long* bar, uint32_t parity)
{
    for (int it = 0; it < 2 * kSpinLimit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (it > kSpinLimit) __nanosleep(4000);
    }
    return false;
}

// The places of a CTA's tiles, by one warp.  A tile's place is the sum of the sizes of its job's tiles in front, published as
// in zccl_tiles.cuh: the states of the tiles in front within its group of 32, and the accumulators of the groups in front, of
// which the warp keeps the sum up to its last look-up, so that a look at what is new is two loads per lane.
struct PlaceFinder {
    uint32_t job = ~0u, groups = 0, base = 0;        // of that job, `groups` groups are in the sum `base`
    uint32_t g = 0, tile_sum = 0, group_sum = 0;     // the tile looked for: its group; what the lane has found
    const unsigned long long *tile = nullptr, *group = nullptr;   // what the lane still waits for
    __device__ __forceinline__ void ask(const unsigned long long* acc, int lane) { group = groups + (uint32_t)lane < g ? acc + groups + (uint32_t)lane : nullptr; }
    __device__ __forceinline__ const unsigned long long* accumulators(const Workspace& ws, uint32_t begin, uint32_t epoch) const
    {
        return ws.group_sums + (epoch & 1u) * (uint32_t)group_slots(ws.state_tiles) + (begin >> 5) + job;
    }
    __device__ __forceinline__ void start(const Workspace& ws, uint32_t begin, uint32_t j, uint32_t t, uint32_t epoch, int lane)
    {
        if (j != job) { job = j; groups = 0; base = 0; }
        g = t >> 5;
        tile_sum = group_sum = 0;
        tile = (uint32_t)lane < (t & 31u) ? ws.tile_state + begin + 32u * g + (uint32_t)lane : nullptr;
        ask(accumulators(ws, begin, epoch), lane);
    }
    // one look at what is missing; true when all is there
    __device__ __forceinline__ bool look(const Workspace& ws, uint32_t begin, uint32_t epoch, int lane, uint32_t& place)
    {
        const unsigned long long a = tile ? ld_state(tile) : 0ull, b = group ? ld_state(group) : 0ull;
        if (tile && (uint32_t)(a >> 33) == epoch) { tile_sum = (uint32_t)a; tile = nullptr; }
        if (group && (uint32_t)(b >> 40) == 32u) { group_sum = (uint32_t)b; group = nullptr; }
        if (!__all_sync(kFull, !tile && !group)) return false;
        base += __reduce_add_sync(kFull, group_sum);
        group_sum = 0;
        groups = g - groups > 32u ? groups + 32u : g;
        if (groups < g) {                            // 32 groups at a time
            ask(accumulators(ws, begin, epoch), lane);
            return false;
        }
        place = base + __reduce_add_sync(kFull, tile_sum);
        return true;
    }
};

// An encoded tile goes to its place (one warp).
__device__ __forceinline__ void store_tile(const Job& q, const StreamEntry& e, const Params& bound, const float* stage, const uint32_t (*ring)[kStreamRing],
                                           uint32_t& status, int lane)
{
    const uint32_t padw = (((e.len + kBlock - 1) / kBlock) + 3) >> 2, r = (uint32_t)lane >> 3, l = (uint32_t)lane & 7u;
    const uint32_t nT = (uint32_t)((q.n + kTile - 1) / kTile), tile = e.tile, end = e.place + e.total;
    const unsigned long long word0 = (unsigned long long)kHeaderWords + nT + e.place;
    if (tile == 0) write_header(q.out, lane, q.n, bound.eb_abs, bound.s, nT);
    if (lane == 0 && tile == nT - 1u) *q.out_bytes = (size_t)((word0 + e.total) * 4ull);
    if (e.late) { status |= kStTimeout; return; }
    if ((word0 + e.total) * 4ull > q.out_cap) { status |= kStCapacity; return; }
    uint32_t* __restrict__ dst = q.out + word0;
    if (lane == 0) {
        dst[0] = (uint32_t)e.first_code;
        q.out[kHeaderWords + tile] = end;
    }
    if ((uint32_t)lane < padw) dst[1 + lane] = e.lens[r][l];
    store_payloads(dst + 1u + padw, *reinterpret_cast<const uint4*>(e.words), e.at[r] & kInStage ? reinterpret_cast<const uint32_t*>(stage + r * kRound) : ring[r] + e.at[r], lane);
}

template <int CAP>
__global__ void __launch_bounds__(kStreamThreads, kStreamCtas) encode_stream_kernel(const __grid_constant__ JobBatchT<CAP> jb,
                                                                                      const __grid_constant__ TileMapsT<CAP> maps, Workspace ws,
                                                                                      Params hp, int bound_source)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StreamShared& sh = *reinterpret_cast<StreamShared*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t rd = (uint32_t)tid >> 5;
    // Before the kernel in front on the stream is waited for: a share of the tiles that are dealt out first is asked into L2.  (A
    // prefetch only moves lines into L2, which stays coherent with whatever that kernel still writes.)
    if (rd < kTileWarps && lane == 0) {
        for (uint32_t t = blockIdx.x, k = 0; k < kStreamStages && t < jb.total_tiles; ++k, t += gridDim.x) {
            const Job& q = jb.job[CAP == 1 ? 0 : find_job(jb, t)];
            const unsigned long long e = (unsigned long long)(t - q.tile_begin) * kTile + (unsigned long long)rd * kRound;
            if (q.x && (((uintptr_t)q.x) & 15u) == 0 && e + kRound <= q.n) bulk_prefetch_l2(q.x + e, 4u * kRound);
        }
    }
    if (tid < (int)kStreamQueue) sh.entry[tid].sum = 0;
    if (tid == 0) {
#pragma unroll
        for (int k = 0; k < (int)kStreamStages; ++k) { mbar_init(&sh.full[k], 1); mbar_init(&sh.seen[k], kTileWarps); mbar_init(&sh.empty[k], kTileWarps); }
#pragma unroll
        for (int k = 0; k < (int)kStreamQueue; ++k) { mbar_init(&sh.coded[k], kTileWarps); mbar_init(&sh.known[k], 1); mbar_init(&sh.gone[k], 1); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // The CTA's first number is taken here too: the launch behind, which may be one of this kernel, is let in when every CTA has
    // found that there is no more, or has left, and finds the counter at 0.  (With a relative bound, where a range pass is what
    // comes behind, only when they have left.  us, inputs in turn, let in when there is no more / when left: absolute bounds one
    // behind the other, field at 1e-3, 1037 tiles 9.2 / 10.8, 2048 12.1 / 14.0, 2^24 values 18.6 / 20.2, gradients 2^25 40.3 / 41.8;
    // relative, 2^25 values 59.6 / 56.8.  A decompression let in early: one of each in turn, 2^24 values, 41.1 / 38.3.)
    uint32_t ticket = 0;
    // every CTA takes one number beyond the last tile's, so the counter is back at 0 behind the launch
    auto ask = [&] { if (lane == 0) ticket = atomicInc(ws.next_stream, jb.total_tiles + gridDim.x - 1u); };
    if (rd == kTileWarps) {
        ask();
        if (CAP == 1 && lane == 0) prefetch_map(&maps.m[0]);
    }
    __syncthreads();
    pdl_wait();
    const uint32_t epoch = *reinterpret_cast<volatile uint32_t*>(ws.epoch);
    // The range keys go back to their start once every tile's size is published (finish_places).  The coding warps' sizes come
    // from the bound and the serving warp hands out tiles by it, so they have read it by then; the storing warp of a tile has nothing
    // to do with its size and takes the bound from the serving one.  (A CTA that starts when the launch's last tile has been
    // placed may find the launch counter moved on and the keys back at their start.  It gets no tile.)
    Params prm = hp;
    if (rd != kTileWarps + 1) prm = bound_of(ws, hp, bound_source);
    uint32_t status = 0;

    if (rd == kTileWarps) {                // ---- the warp that brings tiles in and finds their places
        if (lane == 0) sh.bound = prm;     // (seen by the storing warp behind `known`)
        uint32_t asked = 0, placed = 0, coded = 0;    // tiles of the CTA so far: taken, with a known place, encoded (as seen here)
        bool over = false, late = false;
        uint32_t idle = 0;
        PlaceFinder find;
        // every tile of the launch comes by here: the CTA of a job's last one, see finish_places
        auto through = [&](uint32_t j, uint32_t t) {
            const bool last = t + 1u == (CAP > 1 && j + 1u < (uint32_t)jb.count ? jb.job[j + 1u].tile_begin : jb.total_tiles) && prm.valid;
            if (last || epoch == 0x7FFFFFFFu) finish_places(jb, ws, epoch, last, prm, bound_source, lane);
        };
        // Towards the end of a launch a number is taken when the tile can be asked for, not earlier: every number that a CTA holds
        // is then a tile that others, who have none, cannot take.  Its round trip and a look at the places go side by side.
        bool asking = true, taking = true;   // the next number is on its way, or there; its tile's stage and entry are free
        while (!over || placed < asked) {
            bool moved = false;
            if (!over && !taking && (asked < kStreamStages || mbar_test_warp(&sh.empty[asked % kStreamStages], (asked / kStreamStages - 1u) & 1u)) &&
                (asked < kStreamQueue || mbar_test_warp(&sh.gone[asked % kStreamQueue], (asked / kStreamQueue - 1u) & 1u))) {
                if (!asking) ask();
                asking = taking = true;
            }
            if (placed < asked) {
                StreamEntry& e = sh.entry[placed % kStreamQueue];
                if (coded == placed && mbar_test_warp(&sh.coded[placed % kStreamQueue], (placed / kStreamQueue) & 1u)) {
                    moved = true;
                    ++coded;
                    if (e.len) find.start(ws, e.begin, e.job, e.tile, epoch, lane);
                }
                if (coded > placed) {
                    uint32_t place = 0;
                    const bool known = !e.len || find.look(ws, e.begin, epoch, lane, place);
                    if (known || late) {
                        moved = true;
                        through(e.job, e.begin + e.tile);
                        if (lane == 0) {
                            e.place = place; e.late = known ? 0u : 1u;
                            mbar_arrive(&sh.known[placed % kStreamQueue]);
                        }
                        __syncwarp();
                        ++placed;
                    }
                }
            }
            if (taking) {
                asking = taking = false;
                moved = true;
                const uint32_t t = __shfl_sync(kFull, ticket, 0), st = asked % kStreamStages;
                StreamEntry& e = sh.entry[asked % kStreamQueue];
                over = t >= jb.total_tiles;
                if (over) {
                    if (bound_source != kBoundKeys) pdl_release();
                    if (lane == 0) { e.kind = kTileNone; mbar_arrive(&sh.full[st]); }
                    __syncwarp();
                } else {
                    const int j = CAP == 1 ? 0 : find_job(jb, t);
                    const Job& q = jb.job[j];
                    const uint32_t tile = t - q.tile_begin;
                    const unsigned long long start = (unsigned long long)tile * kTile;
                    const uint32_t len = q.n && prm.valid ? (uint32_t)(q.n - start < (unsigned long long)kTile ? q.n - start : kTile) : 0u;
                    const bool bulk = len == (uint32_t)kTile && (((uintptr_t)q.x) & 15u) == 0;
                    if (lane == 0) {
                        e.kind = kTileFast; e.tile = tile; e.job = (uint32_t)j; e.begin = q.tile_begin; e.len = len; e.start = start; e.bulk = bulk ? 1u : 0u;
                        if (bulk) {
                            mbar_expect_tx(&sh.full[st], kTile * 4);
                            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                            asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                         ::"r"(smem_u32(sh.stage[st])), "l"(&maps.m[j]), "r"(0), "r"((int)(start >> 5)), "r"(smem_u32(&sh.full[st])) : "memory");
                        } else mbar_arrive(&sh.full[st]);   // the coding warps load their rounds themselves
                    }
                    __syncwarp();
                    ++asked;
                    if (t + kStreamEnd * gridDim.x < jb.total_tiles) { ask(); asking = true; }
                }
            }
            if (moved) idle = 0;
            else if (++idle > 2u) {
                __nanosleep(idle < 256u ? 20u : 400u);
                if (idle > (uint32_t)(kSpinLimit >> 4)) {
                    if (late) { status |= kStTimeout; break; }
                    late = true;           // no more waiting for places in this launch
                    idle = 0;
                }
            }
        }
        // A wait for the CTA's own warps ran out.  Copies land before the CTA ends, the counter still goes around, and the end of the
        // launch is seen to for the tiles that are left out: the next launch is in order.
        if (!over || placed < asked) {
            const uint32_t newer = asked + (over ? 1u : 0u);              // (what says that there is no more has taken the stage of an older tile, which is through)
            for (uint32_t k = newer > kStreamStages ? newer - kStreamStages : 0u; k < asked; ++k) (void)mbar_wait(&sh.full[k % kStreamStages], (k / kStreamStages) & 1u);
            if (!over && !asking) ask();
            for (uint32_t k = placed; k < asked || !over; ++k) {          // tiles that have been asked for, then further numbers
                const StreamEntry& e = sh.entry[k % kStreamQueue];
                const uint32_t t = k < asked ? e.begin + e.tile : __shfl_sync(kFull, ticket, 0);
                over = over || t >= jb.total_tiles;
                if (t < jb.total_tiles) through(CAP == 1 ? 0u : (uint32_t)find_job(jb, t), t);
                if (k >= asked && !over) ask();
            }
        }
        if (lane == 0) {                   // no more (the last tile's entry is another one: the queue has room for it)
            sh.entry[placed % kStreamQueue].kind = kTileNone;
            mbar_arrive(&sh.known[placed % kStreamQueue]);
        }
        if (status) atomicOr(ws.status, status);
        return;
    }
    if (rd == kTileWarps + 1) {            // ---- the warp that stores them
        for (uint32_t k = 0; k < ws.store_pause; ++k) __nanosleep(1000);
        const Params& bound = sh.bound;
        for (uint32_t i = 0;; ++i) {
            if (!mbar_wait_long(&sh.known[i % kStreamQueue], (i / kStreamQueue) & 1u)) { status |= kStTimeout; break; }
            const StreamEntry& e = sh.entry[i % kStreamQueue];
            if (e.kind == kTileNone) break;
            const Job& q = jb.job[CAP == 1 ? 0 : e.job];
            if (e.len) store_tile(q, e, bound, sh.stage[i % kStreamStages][0], sh.ring, status, lane);
            else if (e.tile == 0) {        // a job without elements, or no valid bound: header and length only
                const bool hdr = bound.valid && q.out_cap >= (unsigned)kHeaderBytes;
                if (lane == 0) *q.out_bytes = hdr ? kHeaderBytes : 0;
                if (hdr) write_header(q.out, lane, 0, bound.eb_abs, bound.s, 0);
                if (lane == 0 && !bound.valid && e.begin == 0) settle_bound(ws, bound, bound_source);
            }
            __syncwarp();
            if (lane == 0) {
                if (e.len) {
#pragma unroll
                    for (int k = 0; k < kTileWarps; ++k)
                        if (e.at[k] & kInStage) mbar_arrive(&sh.empty[i % kStreamStages]);
                }
                mbar_arrive(&sh.gone[i % kStreamQueue]);
            }
            __syncwarp();
        }
        if (status) atomicOr(ws.status, status);
        return;
    }

    // ---- the coding warps
    const float r = prm.r, nz = negative_zero(prm.r);
    const uint32_t e0 = rd * (uint32_t)kRound;
    bool wide = false;
    uint32_t pos = 0, used = 0, stored = 0;  // the ring: where the next payload goes, words that wait (with what is left out at the end), tiles that do not
    uint32_t hold = 0;                       // lane q: what the tile in entry q holds of it
    for (uint32_t i = 0;; ++i) {
        const uint32_t st = i % kStreamStages, q = i % kStreamQueue;
        if (!mbar_wait_long(&sh.full[st], (i / kStreamStages) & 1u) || i + 1u == ws.leave_before) { status |= kStTimeout; break; }
        StreamEntry& e = sh.entry[q];
        if (e.kind == kTileNone) break;
        const uint32_t len = e.len;
        uint32_t words = 0, at = 0, holds = 0;
        int32_t first_code = 0;
        float* stage = sh.stage[st][rd];
        unsigned char* lens = reinterpret_cast<unsigned char*>(e.lens[rd]);
        if (e0 < len) {
            float front = 0.0f;
            if (!e.bulk) {
                const float* x = jb.job[CAP == 1 ? 0 : e.job].x + e.start + e0;
                load_round_ragged(stage, x, 0, len - e0 < (uint32_t)kRound ? len - e0 : (uint32_t)kRound, lane);
                if (rd) front = __ldg(x - 1);
                __syncwarp();
            } else if (rd) front = read_last_of_row(sh.stage[st][rd - 1], 31u);
            const float first = stage[0];
            const float xprev = lane ? read_last_of_row(stage, (uint32_t)lane - 1u) : (rd ? front : first);
            first_code = __float2int_rn(__fmul_rn(first, r));
            if (float* y = jb.job[CAP == 1 ? 0 : e.job].y)   // an uncompressed copy of the input goes along (an Allgather's own contribution)
                store_round_ragged(y + e.start + e0, stage, len - e0 < (uint32_t)kRound ? len - e0 : (uint32_t)kRound, lane);
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.seen[st]);
            words = encode_round_classes(stage, xprev, 32u * (uint32_t)lane < len - e0, r, nz, lens, lane, wide, status, [&](uint32_t need) {
                __syncwarp();                                             // every lane has read its row
                if (lane == 0) mbar_arrive(&sh.empty[st]);
                // room in the ring for the round's payload, and for what write_round may write behind it
                const uint32_t skip = pos + need + 16u > kStreamRing ? kStreamRing - pos : 0u;
                while (used + skip + need + 16u > kStreamRing && stored < i) {
                    if (!mbar_wait_long(&sh.gone[stored % kStreamQueue], (stored / kStreamQueue) & 1u)) { status |= kStTimeout; break; }
                    used -= __shfl_sync(kFull, hold, stored % kStreamQueue);
                    ++stored;
                }
                at = skip ? 0u : pos;
                pos = at + need;
                holds = skip + need;
                used += holds;
                return sh.ring[rd] + at;
            });
            if (words == ~0u) {            // code lengths above 16: in place, where it waits
                if (!mbar_wait_long(&sh.seen[st], (i / kStreamStages) & 1u)) status |= kStTimeout;   // the warp behind has read this round's last value
                const RoundOut o = encode_round_wide(stage, xprev, 32u * (uint32_t)lane < len - e0, r, lens, lane, reinterpret_cast<uint32_t*>(stage));
                status |= o.status;
                words = o.words;
                at = kInStage;
            }
            __syncwarp();
        } else {
            if (lane < 8) e.lens[rd][lane] = 0;
            const Job& job = jb.job[CAP == 1 ? 0 : e.job];
            if (job.y && e.start + e0 < job.n) copy_round_plain(job.y + e.start + e0, job.x + e.start + e0, job.n - e.start - e0, lane);   // no valid bound
            __syncwarp();
            if (lane == 0) { mbar_arrive(&sh.seen[st]); mbar_arrive(&sh.empty[st]); }
        }
        for (; stored + kStreamQueue <= i; ++stored) used -= __shfl_sync(kFull, hold, stored % kStreamQueue);   // (entry q was free, so that tile is stored)
        if ((uint32_t)lane == q) hold = holds;
        if (lane == 0) {
            e.words[rd] = words; e.at[rd] = at;
            if (rd == 0) e.first_code = first_code;
            const uint32_t old = atomicAdd(&e.sum, (1u << 24) | words);
            if (old >> 24 == kTileWarps - 1) {                            // the tile is complete: its size is published
                e.sum = 0;
                const uint32_t tile = e.tile, begin = e.begin, total = 1u + ((((len + kBlock - 1) / kBlock) + 3) >> 2) + (old & 0xFFFFFFu) + words;
                e.total = total;
                if (len && begin + tile != ws.skip_publish) {
                    unsigned long long* groups = ws.group_sums + (epoch & 1u) * (uint32_t)group_slots(ws.state_tiles) + (begin >> 5) + e.job;
                    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(groups + (tile >> 5)), "l"((1ull << 40) | (unsigned long long)total) : "memory");
                    if ((tile & 31u) != 31u) st_state(ws.tile_state + begin + tile, pack_state(epoch, 0u, total));
                }
            }
            mbar_arrive(&sh.coded[q]);
        }
        __syncwarp();
    }
    if (status) atomicOr(ws.status, status);
}
