// The emulated ring reduce-scatter in one launch: included by zccl_codec.cu inside its unnamed namespace.
//
// Chunk c is compressed by its first rank and then passes N - 1 fused hops, each a launch whose CTAs read the index, fetch
// the blob, decode, add, encode, look up a place, store: about 10 us per hop on short chunks, most of it round trips.  A
// tile of a hop's stream depends on nothing but the same tile of the stream before, so a CTA takes a tile through ALL
// steps: it decodes the image the step before has left in shared memory, and every step's stream is still written, in
// full, to a slot of its own, by a fifth warp that publishes the tile's sizes, finds its places and stores it while the
// coding warps are a step further.  No coding warp waits for another: the code in front of its round is that of the
// value in front, which it quantised itself.  An 8-rank
// Allreduce of 2^21 values each takes 74.3 us in all; with a launch or two per step, and the hop of that time, 154.
//
// A CTA waits for the places of lower tiles of its chunk, as in zccl_tiles.cuh (take_tile), and keeps its operands in three
// stages of 16 KiB.  Used while all tiles are resident together: a later wave would go through all its steps alone.

constexpr int kRingRanks = 16;
struct RingArgs {
    const float* send[kRingRanks];
    float* recv[kRingRanks];         // where rank r's uncompressed result of the last step goes
    unsigned long long n, m;         // elements of a rank's array, of a chunk
    unsigned char* mid;              // slots of the streams of steps 0 .. N - 2: step k, rank r at [k N + r]
    unsigned char* last;             // slots of the last step's: rank r at [r]
    unsigned long long slot_bytes;
    size_t* sizes;                   // [N][N]: step, rank
    uint32_t tile_begin[kRingRanks + 1];
    int N, shift;                    // chunk c starts at rank c + shift
    uint32_t flags;
    int whole;                       // recv[r] is an array of n elements (the chunk goes to its place in it), otherwise the chunk
};
struct alignas(64) RingMaps {
    CUtensorMap in[kRingRanks], out[kRingRanks];   // rank r's array, in tiles of 128 rows; its result, in tiles of 32 rows
};

struct alignas(1024) RingShared {
    float stage[3][kTileWarps][kRound];     // a step's operand, its combined values, its image
    uint32_t lens[3][kTileWarps][8];
    uint32_t words[3][kTileWarps];
    int32_t first_code[3];
    uint32_t sum[3];                        // {rounds that are through:8 | their words:24}
    uint32_t taken;                         // what take_tile gave
    alignas(8) unsigned long long full[3], coded[3], used[3];
};

// The place of a tile by one warp: as find_place, for jobs of at most 1024 tiles, both kinds of sizes with one look.  The
// tile's own size has been published (publish_tile).
__device__ __forceinline__ void publish_tile(unsigned long long* tiles, unsigned long long* groups, uint32_t tile, uint32_t total, uint32_t epoch)
{
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(groups + (tile >> 5)), "l"((1ull << 40) | (unsigned long long)total) : "memory");
    if ((tile & 31u) != 31u) st_state(tiles + tile, pack_state(epoch, 0u, total));
}
__device__ __forceinline__ bool find_place_warp(const unsigned long long* tiles, const unsigned long long* groups, uint32_t tile, uint32_t epoch, int lane, uint32_t& place)
{
    const uint32_t g = tile >> 5, in_group = tile & 31u;
    const unsigned long long* pg = (uint32_t)lane < g ? groups + lane : nullptr;
    const unsigned long long* pt = (uint32_t)lane < in_group ? tiles + 32u * g + (uint32_t)lane : nullptr;
    uint32_t sum = 0;
    bool ok = true;
    for (int polls = 0; pg || pt; ++polls) {
        if (polls > (kSpinLimit >> 4)) { ok = false; break; }
        if (polls > 8) __nanosleep(polls < 64 ? 40u : 400u);
        const unsigned long long a = pg ? ld_state(pg) : 0ull, b = pt ? ld_state(pt) : 0ull;
        if (pg && (uint32_t)(a >> 40) == 32u) { sum += (uint32_t)a; pg = nullptr; }
        if (pt && (uint32_t)(b >> 33) == epoch) { sum += (uint32_t)b; pt = nullptr; }
    }
    place = __reduce_add_sync(kFull, sum);
    return __all_sync(kFull, ok);
}

template <int OP>
__global__ void __launch_bounds__(kDecodeThreads, 4) ring_tiles_kernel(const __grid_constant__ RingArgs ra, const __grid_constant__ RingMaps maps, Workspace ws,
                                                                      Params hp, int bound_source)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RingShared& sh = *reinterpret_cast<RingShared*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const int tid = threadIdx.x, lane = tid & 31, N = ra.N;
    const uint32_t rd = (uint32_t)tid >> 5;
    int c = 0;                           // the CTA's chunk
    while (c + 1 < N && ra.tile_begin[c + 1] <= blockIdx.x) ++c;
    const uint32_t tiles = ra.tile_begin[c + 1] - ra.tile_begin[c];
    if (tid == 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) { mbar_init(&sh.full[k], 1); mbar_init(&sh.coded[k], kTileWarps); mbar_init(&sh.used[k], kTileWarps); sh.sum[k] = 0; }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid == 32 * kTileWarps) sh.taken = take_tile(ws, (uint32_t)c, tiles);
    if (rd == 0 && lane < N) prefetch_map(&maps.in[lane]);
    __syncthreads();
    const uint32_t tile = __shfl_sync(kFull, taken_tile(ws, tiles, sh.taken), 0);   // uniform, and known to be: addresses and coordinates stay in uniform registers
    const unsigned long long off = (unsigned long long)c * ra.m;                 // the chunk within a rank's array
    const unsigned long long clen = ra.n - off < ra.m ? ra.n - off : ra.m, start = (unsigned long long)tile * kTile;
    const uint32_t len = (uint32_t)(clen - start < (unsigned long long)kTile ? clen - start : kTile);
    auto rank_at = [&](int k) { const int r = c + ra.shift + k; return r < N ? r : r - N; };   // (below 2 N)
    auto bulk_from = [&](const float* p) {                                       // rank's tile by one tensor copy
        return len == (uint32_t)kTile && (((uintptr_t)p) & 15u) == 0 && ((off + start) & 31ull) == 0;
    };
    if (rd == kTileWarps && lane == rank_at(N - 1)) prefetch_map(&maps.out[lane]);
    pdl_wait();
    if (tid == 0) tile_taken(ws, (uint32_t)c, tiles, sh.taken);
    const Params prm = bound_of(ws, hp, bound_source);
    const uint32_t epoch = *reinterpret_cast<volatile uint32_t*>(ws.epoch);
    uint32_t status = 0;
    if (!prm.valid) {                    // no bound: empty streams
        if (tid == 0 && tile == 0)
            for (int k = 0; k < N; ++k) ra.sizes[k * N + rank_at(k)] = 0;
        if (tid == 0 && blockIdx.x == 0) settle_bound(ws, prm, bound_source);
        return;
    }
    const uint32_t padw = (((len + kBlock - 1) / kBlock) + 3) >> 2;
    const uint32_t all_tiles = ra.tile_begin[N], all_groups = (all_tiles >> 5) + (uint32_t)N + 1u;   // of a step
    unsigned long long* tiles0 = ws.tile_state + ra.tile_begin[c];
    unsigned long long* groups0 = ws.group_sums + (epoch & 1u) * (uint32_t)group_slots(ws.state_tiles) + (ra.tile_begin[c] >> 5) + (uint32_t)c;

    if (rd == kTileWarps) {              // ---- the warp that brings operands and stores streams
        auto request = [&](int k) {
            if (k >= N) return;
            const int r = rank_at(k), s = k % 3;
            if (lane == 0) {
                if (bulk_from(ra.send[r])) {
                    mbar_expect_tx(&sh.full[s], kTile * 4);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 ::"r"(smem_u32(sh.stage[s])), "l"(&maps.in[r]), "r"(0), "r"((int)((off + start) >> 5)), "r"(smem_u32(&sh.full[s])) : "memory");
                } else mbar_arrive(&sh.full[s]);   // the coding warps load their rounds themselves
            }
            __syncwarp();
        };
        for (int k = 0; k < 3; ++k) request(k);
        const uint32_t nT = (uint32_t)((clen + kTile - 1) / kTile);
        bool ok = true;
        for (int k = 0; k < N; ++k) {
            const int s = k % 3, r = rank_at(k);
            const uint32_t phase = (uint32_t)(k / 3) & 1u;
            if (!mbar_wait_resting(&sh.coded[s], phase)) { status |= kStTimeout; ok = false; break; }
            const uint4 w4 = *reinterpret_cast<const uint4*>(sh.words[s]);
            const uint32_t total = 1u + padw + w4.x + w4.y + w4.z + w4.w;
            uint32_t place = 0;
            if (ok) ok = find_place_warp(tiles0 + (size_t)k * all_tiles, groups0 + (uint32_t)k * all_groups, tile, epoch, lane, place);
            if (!ok) status |= kStTimeout;
            uint32_t* out = reinterpret_cast<uint32_t*>(k + 1 < N ? ra.mid + ((size_t)k * N + r) * ra.slot_bytes : ra.last + (size_t)r * ra.slot_bytes);
            const unsigned long long word0 = (unsigned long long)kHeaderWords + nT + place;
            const bool fits = (word0 + total) * 4ull <= ra.slot_bytes;
            if (!fits) status |= kStCapacity;
            if (fits && ok) {
                uint32_t* __restrict__ dst = out + word0;
                if ((uint32_t)lane < padw) dst[1 + lane] = sh.lens[s][lane >> 3][lane & 7];
                if (lane == 0) {
                    dst[0] = (uint32_t)sh.first_code[s];
                    out[kHeaderWords + tile] = place + total;
                }
                store_payloads(dst + 1 + padw, w4, reinterpret_cast<const uint32_t*>(sh.stage[s][lane >> 3]), lane);
            }
            if (lane == 0 && tile == nT - 1) ra.sizes[k * N + r] = (size_t)((word0 + total) * 4ull);
            if (tile == 0) write_header(out, lane, clen, prm.eb_abs, prm.s, nT);
            __syncwarp();
            if (k + 3 < N) {             // the stage takes another operand when the image is stored and decoded
                if (!mbar_wait_resting(&sh.used[s], phase)) { status |= kStTimeout; break; }
                request(k + 3);
            }
        }
        uint32_t jobs = 0;
        for (int k = 0; k < N; ++k) jobs += ra.tile_begin[k + 1] > ra.tile_begin[k] ? 1u : 0u;
        finish_places(ws, epoch, tile + 1u == tiles, all_tiles, jobs, (uint32_t)N * all_groups, prm, bound_source, lane);
        if (status) atomicOr(ws.status, status);
        return;
    }

    // ---- the coding warps
    const float s = prm.s, r = prm.r, nz = negative_zero(prm.s);
    const uint32_t e0 = rd * (uint32_t)kRound, sw = ((uint32_t)lane & 7u) << 4, op = (ra.flags >> 1) & 3u, flip = op == 2u ? 0x80000000u : 0u;
    const uint32_t mine = e0 < len ? (len - e0 < (uint32_t)kRound ? len - e0 : (uint32_t)kRound) : 0u;   // elements of the round
    const bool active = 32u * (uint32_t)lane < mine;
    int32_t code_round = 0;              // the code in front of the round, in the stream of the step before
    bool wide = false, general = false;  // general: that stream's round is beyond the fp32 route
    // the element in front of the round in the next step's operand: asked for a step ahead
    auto in_front = [&](int k) { return rd && mine && k < N ? __ldg(ra.send[rank_at(k)] + off + start + e0 - 1) : 0.0f; };
    float front_next = in_front(0);
    for (int k = 0; k < N; ++k) {
        const int st = k % 3, pst = (k + 2) % 3;
        if (!mbar_wait(&sh.full[st], (uint32_t)(k / 3) & 1u)) { status |= kStTimeout; break; }
        const int rank = rank_at(k);
        const float* x = ra.send[rank] + off + start + e0;
        float* stage = sh.stage[st][rd];
        uint32_t* payload = reinterpret_cast<uint32_t*>(stage);
        unsigned char* lens = reinterpret_cast<unsigned char*>(sh.lens[st][rd]);
        uint32_t words = 0;
        int32_t first_code = 0;
        const float front_x = front_next;
        front_next = in_front(k + 1);
        // the image of the step before has been read for the last time
        auto used = [&] {
            __syncwarp();
            if (k && lane == 0) mbar_arrive(&sh.used[pst]);
        };
        if (mine) {
            if (!bulk_from(ra.send[rank])) {
                load_round_ragged(stage, x, 0, mine, lane);
                __syncwarp();
            }
            const float y0_raw = stage[0];
            float front = front_x;       // the value in front of the round
            if (k == 0) {
                const float xprev = lane ? read_last_of_row(stage, (uint32_t)lane - 1u) : (rd ? front_x : y0_raw);
                first_code = __float2int_rn(__fmul_rn(y0_raw, r));
                words = encode_round_staged<false>(stage, xprev, active, r, nz, lens, lane, wide, status, payload, lens, payload, [] { __syncwarp(); });
                general = (words >> 31) != 0;
                words &= 0x7FFFFFFFu;
            } else {
                front = __fmul_rn(__int2float_rn(code_round), s);
                front = OP == 0 ? __fadd_rn(front, front_x) : choose(front, front_x, flip);
                const uint32_t* pay = reinterpret_cast<const uint32_t*>(sh.stage[pst][rd]);
                const uint32_t L = reinterpret_cast<const unsigned char*>(sh.lens[pst][rd])[lane];
                const uint32_t nw = L ? L + 1u : 0u, at = warp_incl_scan(nw, lane) - nw;
                char* row = reinterpret_cast<char*>(stage) + 128 * lane;
                uint32_t longest = 0;
                auto in_place = [&](uint32_t) { __syncwarp(); return payload; };
                words = ~0u;
                // the combined values replace the operand's in the stage: what the narrow class does not cover is encoded from there
                auto recode = [&](auto& v, auto& o) {
                    constexpr int W = sizeof(v) / 4;
                    int32_t sum;
                    load_deltas<W>(pay + at, L, !__any_sync(kFull, L > (uint32_t)W / 2), v, sum);
                    const int32_t code = code_round + warp_incl_scan_s(sum, lane) - sum;
                    float c0;
                    recode_block<W, OP, true, false>(v, code, s, r, nz, row, sw, rd != 0, front, flip, lane, o, c0);
                    first_code = (int32_t)(__float_as_uint(c0) - kRoundMagicBits);
                    if (!active) o.L = 0;
                    longest = __reduce_max_sync(kFull, o.L);
                };
                auto copy_out = [&]() {  // the uncompressed copy of the last step leaves before the image is written over it
                    float* y = ra.recv[rank];
                    if (k + 1 < N || !y) return;
                    y += start + e0 + (ra.whole ? off : 0ull);
                    __syncwarp();
                    if (ra.flags & 1u) store_round_dequantised(y, stage, mine, r, s, lane);
                    else if (mine == (uint32_t)kRound && (((uintptr_t)ra.recv[rank]) & 15u) == 0 && ((start + (ra.whole ? off : 0ull)) & 31ull) == 0) {
                        if (lane == 0) {
                            tensor_store_round(&maps.out[rank], (uint32_t)((start + e0 + (ra.whole ? off : 0ull)) >> 5), stage);
                            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        }
                    } else store_round_ragged(y, stage, mine, lane);
                    __syncwarp();
                };
                if (!general && !__any_sync(kFull, L > 15u)) {
                    if (!wide && !__any_sync(kFull, L > 7u)) {
                        uint32_t v[8];
                        BlockCode<8> o;
                        recode(v, o);
                        used();
                        copy_out();
                        if (longest <= 8u && !__any_sync(kFull, fabsf(o.t_front) > 24000.0f))
                            words = write_round<8, false>(o.w, o.sign, o.L, longest, lens, lane, in_place);
                    } else {
                        uint32_t v[16];
                        BlockCode<16> o;
                        recode(v, o);
                        used();
                        copy_out();
                        if (longest <= 16u) {
                            if (o.t_max > 32768.5f) status |= kStPrecision;
                            words = write_round<16, false>(o.w, o.sign, o.L, longest, lens, lane, in_place);
                        }
                        wide = longest > 8u || __any_sync(kFull, L > 7u);
                    }
                } else {
                    uint32_t zero = 0;
                    int32_t code = code_round;
                    decode_round_general(pay - 1, 0, L, &zero, &code, s, stage, lane, stage, op);
                    used();
                    copy_out();
                }
                general = false;
                if (words == ~0u) {
                    __syncwarp();
                    const float y0 = stage[0];
                    const float xprev = lane ? read_last_of_row(stage, (uint32_t)lane - 1u) : (rd ? front : y0);
                    first_code = __float2int_rn(__fmul_rn(y0, r));
                    wide = true;
                    words = encode_round_staged<false>(stage, xprev, active, r, nz, lens, lane, wide, status, payload, lens, payload, [] { __syncwarp(); });
                    general = (words >> 31) != 0;
                    words &= 0x7FFFFFFFu;
                    wide = true;
                }
            }
            code_round = rd ? __float2int_rn(__fmul_rn(front, r)) : __shfl_sync(kFull, first_code, 0);
        } else {
            if (lane < 8) sh.lens[st][rd][lane] = 0;
            used();
        }
        __syncwarp();
        if (lane == 0) {
            sh.words[st][rd] = words;
            if (rd == 0) sh.first_code[st] = first_code;
            const uint32_t old = atomicAdd(&sh.sum[st], (1u << 24) | words);
            if (old >> 24 == kTileWarps - 1) {   // the tile is complete: its size is published
                sh.sum[st] = 0;
                publish_tile(tiles0 + (size_t)k * all_tiles, groups0 + (uint32_t)k * all_groups, tile, 1u + padw + (old & 0xFFFFFFu) + words, epoch);
            }
            mbar_arrive(&sh.coded[st]);
        }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (status) atomicOr(ws.status, status);
}
