// The fused hop of binary32, out = compress(decompress(in) (+) local): included by zccl_codec.cu inside its unnamed
// namespace.
//
// The decoder's CTA (zccl_decode.cuh: four coding warps, one fetching warp) with the encoder's back end: a lane takes its
// block from planes to planes in registers.  Every delta is expanded, summed into the running code, multiplied, combined
// with the operand's value from the stage and at once quantised, differenced and packed again; only the operand's row
// and the two blobs pass through shared memory.  The first delta of a block needs the last value of the block in
// front: it is added at the end, from the lane in front (a round's first lane recomputes the value in front of the
// round from the code there, which is known).  place_kernel turns the rounds' slots into the stream.
//
// What bounds it: instruction issue (30 instructions per element at 60 % of the slots).  A decoder that left the sums in
// the stage and an encoder that read them back, a warp per tile, executed 42.8 and took 42.3 us per 2^24 values with
// its placement (code lengths around 4; 54 us at 7, 196 us per 2^26 gradients); this form takes 32.2, 42.5 and 159.
// Three CTAs per SM, with two or three blob buffers, take 36.3 and 35.1.

struct alignas(1024) HopShared {
    float loc[2][kTileWarps][kRound];      // the operand's tiles; a round's image replaces its operand and leaves from here
    alignas(16) uint32_t blob[kHopBlobs][kBlobBufWords];
    DecodeWork work[kHopBlobs];
    alignas(16) int32_t sums[kHopBlobs][kTileWarps];
    PlaceShared place;
    alignas(8) unsigned long long landed[kHopBlobs], ready[kHopBlobs], free[kHopBlobs], full[2], gone[2];
};
static_assert(offsetof(HopShared, blob) % 16 == 0, "targets of the copy engine");

__device__ __forceinline__ float choose(float a, float b, uint32_t flip)
{
    return __uint_as_float(__float_as_uint(a) ^ flip) < __uint_as_float(__float_as_uint(b) ^ flip) ? b : a;
}

// From biased deltas to packed magnitudes.  `loc`: the operand's row; OP 0: sum, 1: max (flip = 0) or min
// (flip = the sign bit), of two that compare equal the decoded one; Y: the combined values
// replace the operand's in the row.  front_value: the value in front of the block, for lane 0 (has_front: there is one).
// (ONE: the launch's warps have one block each.  Chosen by measurement: with the values written back, loads and stores whose order
// the compiler may choose, 2^19 gradients 8.2 us instead of 8.6 (in the order as written a chunk's load stands behind the store of
// the chunk in front); without, loads as written, which need an instruction less, 100 003 values 6.0 instead of 6.5.)
template <int N, int OP, bool Y, bool ONE>
__device__ __forceinline__ void recode_block(const uint32_t (&v)[N], int32_t code_before, float s, float r, float nz, char* row, uint32_t sw,
                                             bool has_front, float front_value, uint32_t flip, int lane, BlockCode<N>& o, float& first_c)
{
    const float2 r2 = make_float2(r, r), nz2 = make_float2(nz, nz), magic2 = make_float2(kRoundMagic, kRoundMagic);
    const uint32_t row0 = smem_u32(row) + sw;
    float cp = 0.0f, c0 = 0.0f, tm = 0.0f;
    uint32_t orb = 0x4B000000u, sg = 0;
    expand_deltas<N>(v, code_before, s, [&](uint32_t chunk, float2 r01, float2 r23, float2 s2) {
        const uint32_t at = row0 ^ (16u * chunk);
        float4* const p = reinterpret_cast<float4*>(row + ((16u * chunk) ^ sw));
        const float4 l = Y && ONE ? *p : ld_shared4(at);
        const float2 p01 = product2(r01, s2, nz2), p23 = product2(r23, s2, nz2);
        float2 y01, y23;
        if (OP == 0) {
            y01 = __fadd2_rn(p01, make_float2(l.x, l.y));
            y23 = __fadd2_rn(p23, make_float2(l.z, l.w));
        } else {
            y01 = make_float2(choose(p01.x, l.x, flip), choose(p01.y, l.y, flip));
            y23 = make_float2(choose(p23.x, l.z, flip), choose(p23.y, l.w, flip));
        }
        if (Y && ONE) *p = make_float4(y01.x, y01.y, y23.x, y23.y);
        else if (Y) st_shared4(at, make_float4(y01.x, y01.y, y23.x, y23.y));
        const float2 t01 = product2(y01, r2, nz2), t23 = product2(y23, r2, nz2);
        if (N == 16) tm = fmaxf(fmaxf(fmaxf(tm, fabsf(t01.x)), fabsf(t01.y)), fmaxf(fabsf(t23.x), fabsf(t23.y)));
        const float2 c01 = __fadd2_rn(t01, magic2), c23 = __fadd2_rn(t23, magic2);
        const float cs[4] = {c01.x, c01.y, c23.x, c23.y};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t h = (4u * chunk + e) / N;
            const int i = (4 * (int)chunk + e) % N;
            if (h == 0 && i == 0) { c0 = cs[0]; cp = cs[0]; o.w[0] = 0x4B000000u; continue; }   // the first delta: at the end
            const float d = __fsub_rn(cs[e], cp);
            cp = cs[e];
            const uint32_t m = __float_as_uint(__fadd_rn(fabsf(d), kTwo23));
            orb |= m;
            sg = __funnelshift_l(__float_as_uint(d), sg, 1);
            if (h == 0) o.w[i] = m;
            else if (N == 16) o.w[i] = prmt(o.w[i], m, 0x5410u);
            else o.w[i] = prmt(o.w[i], m, h == 1 ? 0x0040u : h == 2 ? 0x0410u : 0x4210u);
        }
    });
    float front = __shfl_up_sync(kFull, cp, 1);
    if (lane == 0) front = has_front ? __fadd_rn(__fmul_rn(front_value, r), kRoundMagic) : c0;
    const float d = __fsub_rn(c0, front);
    const uint32_t m = __float_as_uint(__fadd_rn(fabsf(d), kTwo23));
    orb |= m;
    o.w[0] = prmt(o.w[0], m, N == 16 ? 0x3254u : 0x3214u);
    o.sign = __brev(sg | (__float_as_uint(d) & 0x80000000u));
    o.L = 32u - (uint32_t)__clz((int)(orb ^ 0x4B000000u));
    o.t_front = __fsub_rn(front, kRoundMagic);
    if (!(fabsf(o.t_front) < 2097152.0f)) o.L = 32u;
    o.t_max = tm;
    first_c = c0;
}

// A round by the slow route: the incoming round from global memory with integer arithmetic onto the stage.
// Then the encoder's general classes.  Out of line; bit 31 of the result: the image went straight to the slot.
__device__ __noinline__ RoundOut encode_round_from_stage(float* stage, float xprev, bool active, float r, uint32_t* slot, int lane)
{
    RoundOut o;
    o.status = 0;
    uint32_t longest = 0;
    o.words = encode_round_class<16, false>(stage, xprev, active, r, negative_zero(r), reinterpret_cast<unsigned char*>(stage), lane, o.status, longest,
                                     [&](uint32_t) { __syncwarp(); return reinterpret_cast<uint32_t*>(stage) + 8; });
    if (o.words == ~0u) {
        o = encode_round_wide(stage, xprev, active, r, reinterpret_cast<unsigned char*>(slot), lane, slot + 8);
        o.words |= 0x80000000u;
    }
    __syncwarp();
    return o;
}

// One launch's hops.  OP 0: sums (and averages), 1: the reduce operation is max or min, by the job's flags.  Y: some job
// wants an uncompressed copy of its result.  ONCE: a CTA per tile, which finds its place itself; otherwise the rounds go
// to their slots for place_kernel.  maps: job j's operand (in tiles of 128 rows) at [j]; of its uncompressed
// result (32 rows) at [CAP / 2 + j] in launches of at most CAP / 2 jobs, at [1] for CAP = 1.
template <int CAP, int OP, bool Y, bool ONCE>
__global__ void __launch_bounds__(kDecodeThreads, kHopCtas) hop_tiles_kernel(const __grid_constant__ JobBatchT<CAP> jb,
                                                                            const __grid_constant__ TileMapsT<CAP == 1 ? 2 : CAP> maps, Workspace ws)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    HopShared& sh = *reinterpret_cast<HopShared*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t rd = (uint32_t)tid >> 5;
    if (tid == 0) {
#pragma unroll
        for (int k = 0; k < (int)kHopBlobs; ++k) { mbar_init(&sh.landed[k], 1); mbar_init(&sh.ready[k], 1); mbar_init(&sh.free[k], kTileWarps); }
#pragma unroll
        for (int k = 0; k < 2; ++k) { mbar_init(&sh.full[k], 1); mbar_init(&sh.gone[k], kTileWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (ONCE) sh.place.failed = 0;
    }
    uint32_t from = 0, first = 0, of = 0;     // ONCE: the CTA's job, its first tile, its tiles
    if (ONCE) {
        from = CAP == 1 ? 0u : (uint32_t)find_job(jb, blockIdx.x);
        first = jb.job[from].tile_begin;
        of = (from + 1u < (uint32_t)jb.count ? jb.job[from + 1u].tile_begin : jb.total_tiles) - first;
        if (tid == 32 * kTileWarps) sh.place.taken = take_tile(ws, from, of);
    }
    // In front of the wait for the kernel in front on the stream: the operand's tile is asked into L2, and the blob.  (With a tile
    // per CTA, whose number is not the CTA's, 2^19 values 7.2 us instead of 6.9.)
    if (!ONCE && rd == 0 && lane == 0) {
        const Job& q = jb.job[CAP == 1 ? 0 : find_job(jb, blockIdx.x)];
        const unsigned long long e = (unsigned long long)(blockIdx.x - q.tile_begin) * kTile;
        if (q.x && (((uintptr_t)q.x) & 15u) == 0 && e + kTile <= q.n) bulk_prefetch_l2(q.x + e, 4u * kTile);
    }
    if (!ONCE && CAP == 1 && rd == 1) hint_blob(jb.job[0], blockIdx.x, lane);
    __syncthreads();
    if (ONCE) {
        pdl_wait();
        if (tid == 0) tile_taken(ws, from, of, sh.place.taken);
    } else pdl_enter();
    const uint32_t epoch = ONCE ? *reinterpret_cast<volatile uint32_t*>(ws.epoch) : 0u;
    uint32_t status = 0;
    if (rd == kTileWarps) {
        // the operand's tile goes into its stage when the image that was there has left
        auto operand = [&](const DecodeWork& w, uint32_t i) {
            const uint32_t st = i & 1u;
            if (i >= 2 && !mbar_wait_resting(&sh.gone[st], ((i >> 1) - 1u) & 1u)) { status |= kStTimeout; return false; }
            if (lane == 0) {
                const float* x = jb.job[CAP == 1 ? 0 : w.job].x;
                if ((w.kind == kTileFast || w.kind == kTileSlow) && w.len == (uint32_t)kTile && (((uintptr_t)x) & 15u) == 0) {
                    mbar_expect_tx(&sh.full[st], kTile * 4);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 ::"r"(smem_u32(sh.loc[st])), "l"(&maps.m[CAP == 1 ? 0 : w.job]), "r"(0), "r"((int)(w.start >> 5)),
                                   "r"(smem_u32(&sh.full[st])) : "memory");
                } else mbar_arrive(&sh.full[st]);   // the coding warps load their rounds themselves
            }
            __syncwarp();
            return true;
        };
        fetch_tiles<kHopBlobs, true, false, false, false>(jb, ONCE ? first + taken_tile(ws, of, sh.place.taken) : blockIdx.x, nullptr, sh.blob, sh.work, sh.landed, sh.ready, sh.free, status, lane, operand);
        if (status) atomicOr(ws.status, status);
        return;
    }
    const uint32_t e0 = rd * (uint32_t)kRound, sw = ((uint32_t)lane & 7u) << 4;
    bool wide = false;
    for (uint32_t i = 0;; ++i) {
        const uint32_t b = i % kHopBlobs, st = i & 1u;
        if (!mbar_wait(&sh.ready[b], (i / kHopBlobs) & 1u)) { status |= kStTimeout; break; }
        const DecodeWork& w = sh.work[b];
        const uint32_t kind = w.kind;
        if (kind == kTileNone) break;
        const uint32_t len = w.len, job = CAP == 1 ? 0 : w.job, ul = 4u * w.t + rd;
        const unsigned long long start = w.start;
        const float s = w.s, r = __fdiv_rn(1.0f, s), nz = negative_zero(s);
        const Job& q = jb.job[job];
        float* stage = sh.loc[st][rd];
        // the image of the tile in front has left its stage once the copy engine is through with reading it
        auto left = [&]() {
            if (i == 0) return;
            if (lane == 0) {
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                mbar_arrive(&sh.gone[st ^ 1u]);
            }
        };
        auto give_back = [&]() {
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.free[b]);
        };
        if (!mbar_wait(&sh.full[st], (i >> 1) & 1u)) { status |= kStTimeout; break; }
        const float eb_abs = w.eb_abs;
        const bool with_header = w.valid != 0;
        // the tile is encoded (first_code: warp 0's): its place, and the warp's piece of it goes there
        auto finish = [&](uint32_t words, int32_t first_code, const uint32_t* lens, const uint32_t* payload) {
            const uint32_t tile = (uint32_t)(start >> 12), begin = (ul >> 2) - tile, padw = (((len + kBlock - 1) / kBlock) + 3) >> 2;
            uint32_t total, offset;
            bool placed;
            const uint32_t place = find_place(ws, sh.place, begin, job, tile, 1u + padw, words, epoch, rd, lane, total, offset, placed);
            if (rd == kTileWarps - 1) finish_places(jb, ws, epoch, start + len == q.n, Params{}, kBoundHost, lane);
            store_piece(q, tile, padw, place, offset, words, total, placed, first_code, lens, payload, eb_abs, s, rd, lane, status);
        };
        if (kind == kTileSkip || e0 >= len) {
            if (kind != kTileSkip) (void)code_in_front(sh.sums[b], 0, 0, rd, lane);   // the exchange needs all four
            left();
            give_back();
            if (!ONCE) {
                if (lane == 0) ws.round_words[ul] = 0;
            } else if (len) {                        // (a damaged tile, reported, counts as one of constant blocks)
                if (lane < 8) reinterpret_cast<uint32_t*>(stage)[lane] = 0;
                __syncwarp();
                finish(0, 0, reinterpret_cast<const uint32_t*>(stage), nullptr);
            } else if (rd == 0) {                    // a job without elements, or streams that do not agree with it: header and length only
                const bool hdr = with_header && q.out_cap >= (unsigned)kHeaderBytes;
                if (lane == 0) *q.out_bytes = hdr ? kHeaderBytes : 0;
                const uint32_t end = CAP > 1 && job + 1 < (uint32_t)jb.count ? jb.job[job + 1].tile_begin : jb.total_tiles;
                finish_places(jb, ws, epoch, (ul >> 2) + 1u == end, Params{}, kBoundHost, lane);
                if (hdr) write_header(q.out, lane, 0, eb_abs, s, 0);
            }
            continue;
        }
        const uint32_t nb = (len + kBlock - 1) / kBlock, padw = (nb + 3) >> 2, bi = 32u * rd + (uint32_t)lane;
        const float front_x = rd && lane == 0 ? __ldg(q.x + start + e0 - 1u) : 0.0f;
        const uint32_t op = OP == 0 ? 0u : (q.flags >> 1) & 3u, flip = op == 2u ? 0x80000000u : 0u;
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
        if (len != (uint32_t)kTile || (((uintptr_t)q.x) & 15u) != 0) {
            load_round_ragged(stage, q.x + start + e0, 0, len - e0 < (uint32_t)kRound ? len - e0 : (uint32_t)kRound, lane);
            __syncwarp();
        }
        char* row = reinterpret_cast<char*>(stage) + 128 * lane;
        uint32_t* slot = ws.slots + (size_t)ul * kRoundSlotWords;
        uint32_t* payload = reinterpret_cast<uint32_t*>(stage) + 8;
        unsigned char* lens = reinterpret_cast<unsigned char*>(stage);
        auto in_place = [&](uint32_t) { __syncwarp(); return payload; };
        uint32_t words = ~0u, longest = 0;
        int32_t first_code = 0;
        bool told = false, staged = true;      // `left` has been called; the image is in the stage
        const bool active = bi < nb;
        // the uncompressed copy leaves the stage before the image is written over it
        auto copy_out = [&]() {
            if (!Y || !q.y) return;
            const uint32_t count = len - e0 < (uint32_t)kRound ? len - e0 : (uint32_t)kRound;
            __syncwarp();
            if (q.flags & 1u) store_round_dequantised(q.y + start + e0, stage, count, r, s, lane);
            else if ((CAP == 1 || jb.count <= CAP / 2) && (((uintptr_t)q.y) & 15u) == 0 && count == (uint32_t)kRound) {
                if (lane == 0) {
                    tensor_store_round(&maps.m[CAP == 1 ? 1 : CAP / 2 + job], (uint32_t)(start >> 5) + 32u * rd, stage);
                    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                }
            } else store_round_ragged(q.y + start + e0, stage, count, lane);
            __syncwarp();
        };
        int32_t code_round = 0;                // the code in front of the round
        auto code_of = [&](const uint32_t* pay, auto& v) {
            int32_t sum;
            constexpr int N = sizeof(v) / 4;
            load_deltas<N>(pay, L, !__any_sync(kFull, L > (uint32_t)N / 2), v, sum);
            const int32_t incl = ONCE ? plain_scan(sum, lane) : warp_incl_scan_s(sum, lane);
            if (!told) {
                code_round = code_in_front(sh.sums[b], __shfl_sync(kFull, incl, 31), outlier, rd, lane);
                left();
                told = true;
            }
            return code_round + incl - sum;
        };
        auto recode = [&](auto& v, int32_t code, auto& o) {
            constexpr int N = sizeof(v) / 4;
            float c0;
            float fv = __fmul_rn((float)code_round, s);
            fv = OP == 0 ? __fadd_rn(fv, front_x) : choose(fv, front_x, flip);
            recode_block<N, OP, Y, ONCE>(v, code, s, r, nz, row, sw, rd != 0, fv, flip, lane, o, c0);
            first_code = (int32_t)(__float_as_uint(c0) - kRoundMagicBits);
            if (!active) o.L = 0;
            longest = __reduce_max_sync(kFull, o.L);
        };
        if (!slow) {
            const uint32_t nw = L ? L + 1u : 0u;
            const uint32_t* pay = blob + 1 + padw + before + ((ONCE ? plain_scan(nw, lane) : warp_incl_scan(nw, lane)) - nw);
            bool narrow = !wide && !__any_sync(kFull, L > 7u);
            if (narrow) {
                uint32_t v[8];
                const int32_t code = code_of(pay, v);
                BlockCode<8> o;
                recode(v, code, o);
                // (Y: the stage holds the combined values by now, and there is no second try from the operand)
                narrow = longest <= 8u && !__any_sync(kFull, fabsf(o.t_front) > 24000.0f);
                if (narrow) {
                    give_back();
                    copy_out();
                    words = write_round<8, ONCE>(o.w, o.sign, o.L, longest, lens, lane, in_place);
                } else if (Y) slow = true;
            }
            if (!narrow && !slow) {
                uint32_t v[16];
                const int32_t code = code_of(pay, v);
                BlockCode<16> o;
                recode(v, code, o);
                if (longest <= 16u) {
                    give_back();
                    copy_out();
                    if (o.t_max > 32768.5f) status |= kStPrecision;
                    words = write_round<16, ONCE>(o.w, o.sign, o.L, longest, lens, lane, in_place);
                    wide = longest > 8u || __any_sync(kFull, L > 7u);
                } else slow = true;
            }
        }
        if (words == ~0u) {                    // the slow route: decode onto the stage, then encode from it
            const uint32_t* in_global = (const uint32_t*)(uintptr_t)src;
            uint32_t off = before;
            int32_t code = code_round;
            if (!told) {
                int32_t sum = 0;
                skip_round(in_global, padw, L, &off, &sum, lane);
                code = code_in_front(sh.sums[b], sum, outlier, rd, lane);
                code_round = code;
                left();
                off = before;
            }
            if (!(Y && told)) decode_round_general(in_global, padw, L, &off, &code, s, stage, lane, stage, op);
            give_back();
            copy_out();
            __syncwarp();
            const float y0 = stage[0];
            const float xprev = lane ? read_last_of_row(stage, (uint32_t)lane - 1u) : (rd ? combine(op, __fmul_rn(__int2float_rn(code_round), s), front_x) : y0);
            first_code = __float2int_rn(__fmul_rn(y0, r));
            const RoundOut o = encode_round_from_stage(stage, xprev, active, r, slot, lane);
            status |= o.status;
            staged = !(o.words >> 31);
            words = o.words & 0x7FFFFFFFu;
            wide = true;
        }
        __syncwarp();
        if (ONCE) {
            const uint32_t* image = staged ? reinterpret_cast<const uint32_t*>(stage) : slot;
            finish(words, first_code, image, image + 8);
            continue;
        }
        if (lane == 0) {
            if (staged) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(slot), "r"(smem_u32(stage)),
                             "r"((32u + 4u * words + 15u) & ~15u) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
            ws.round_words[ul] = words;
            const uint32_t tile = (uint32_t)(start >> 12), begin = (ul >> 2) - tile;
            if (rd == 0) ws.outliers[ul >> 2] = first_code;
            asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(ws.group_acc + (begin >> 5) + job + (tile >> 5)),
                         "l"((unsigned long long)words) : "memory");
        }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (status) atomicOr(ws.status, status);
}
