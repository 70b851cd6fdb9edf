// Binary64 input on the lane-per-block decomposition: included by zccl_codec.cu inside its unnamed namespace, after
// the binary32 kernels whose back ends (bit-matrix transposes, plane loads, blob windows, the placement) it shares.
//
// What differs from binary32 is the way in and the way out.  In: q = rint(fl64(x * r)) comes from one multiplication and
// one addition of 1.5 * 2^52, whose sum carries q in two's complement in its low mantissa word for every |x r| < 2^51;
// deltas, magnitudes and signs are 32-bit integer work from there on (no precision caveat: the codes are exact over
// the whole range |q| < 2^30, which is checked on the exponent bits of x r).  Out: x' = fl64(q * s) with q made a
// binary64 by the same device backwards (the word q ^ 2^31 under the exponent of 2^52, minus 2^52 + 2^31).
//
// A round is still 32 blocks = 1024 elements, now 8 KiB.  The output array is described to the copy engine as rows of 16
// doubles (128 bytes, the widest row the 128-byte swizzle takes), a round is a box of 64 rows, and lane l owns rows
// 2 l and 2 l + 1.  Chunk c (16 bytes = two doubles) of row t sits at chunk c ^ (t & 7) of that row.  Kernels here
// take one array per launch; one that does not start on a 16-byte boundary is accessed with 8-byte loads and stores.

constexpr double kMagic52 = 6755399441055744.0;         // 1.5 * 2^52
constexpr double kIntBias = 4503601774854144.0;         // 2^52 + 2^31
constexpr uint32_t kRangeHi = 0x41D00000u;              // high word of 2^30: |t| < 2^30 <=> (hi(t) & 0x7FFFFFFF) < kRangeHi
constexpr int kRowsPerRound64 = 64;                     // rows of 16 doubles

// Byte offset, inside a lane's pair of rows, of the lane's 16-byte chunk k (k = 0 .. 15: elements 2 k and 2 k + 1 of its
// block); sw0 = (2 lane) & 7 is the swizzle of the first row, sw0 | 1 that of the second.
__device__ __forceinline__ uint32_t pair_chunk_byte(uint32_t k, uint32_t sw0) { return (16u * k) ^ ((sw0 | (k >> 3)) << 4); }

// A warp's round as codes: 32 rows of 32 words, chunk c of row l at c ^ (l & 7), so that both the elements' order (a row
// per half warp) and the blocks' (a row per lane) are free of bank conflicts.  Its image (code-length bytes, payload
// from word 8) is made in the same place, whatever the code lengths; what write_round may write behind the
// payload fits too.
struct alignas(128) Round64Shared {
    uint32_t image[kRound + 8 + 24];
};
static_assert(sizeof(Round64Shared) == 33 * 128, "a warp's share of the shared memory");
constexpr int kEnc64Ctas = 5;

// Deltas of the block in this lane's row of codes against the code in front: magnitudes packed 32 / N to a word for the
// N-bit transpose (word i, field h = element N h + i; more than N bits: the caller looks at the OR), sign word.
template <int N>
__device__ __forceinline__ void block_deltas(const uint32_t* row, uint32_t sw, uint32_t q_front, uint32_t (&w)[N], uint32_t& sign, uint32_t& orb_out)
{
    uint32_t qp = q_front, orb = 0, sg = 0;
#pragma unroll
    for (int h = 0; h < 32 / N; ++h) {
#pragma unroll
        for (int k = 0; k < N / 4; ++k) {
            const uint4 v = *reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(row) + ((16u * (uint32_t)(h * (N / 4) + k)) ^ sw));
            const uint32_t q[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = 4 * k + e;
                const int32_t d = (int32_t)(q[e] - qp);
                qp = q[e];
                const uint32_t m = (uint32_t)abs(d);
                orb |= m;
                sg = __funnelshift_l((uint32_t)d, sg, 1);     // sign of element j ends up in bit 31 - j
                if (h == 0) w[i] = m;
                else if (N == 16) w[i] = prmt(w[i], m, 0x5410u);
                else w[i] = prmt(w[i], m, h == 1 ? 0x0040u : h == 2 ? 0x0410u : 0x4210u);
            }
        }
    }
    sign = __brev(sg);
    orb_out = orb;
}
// One width class; ~0 with nothing stored when a lane's code is longer than N.
template <int N>
__device__ __forceinline__ uint32_t encode_codes_class(uint32_t* image, uint32_t q_front, int lane)
{
    uint32_t w[N], sign, orb;
    block_deltas<N>(image + 32 * lane, ((uint32_t)lane & 7u) << 4, q_front, w, sign, orb);
    const uint32_t L = code_length(orb);
    const uint32_t longest = __reduce_max_sync(kFull, L);
    if (longest > (uint32_t)N) return ~0u;
    return write_round<N, false>(w, sign, L, longest, reinterpret_cast<unsigned char*>(image), lane, [&](uint32_t) { __syncwarp(); return image + 8; });
}
// Codes of any length (out of line: its 32 words would set the kernel's register count).
__device__ __noinline__ uint32_t encode_codes_wide(uint32_t* image, uint32_t q_front, int lane)
{
    uint32_t w[32], qp = q_front, sg = 0, orb = 0;
    const char* row = reinterpret_cast<const char*>(image + 32 * lane);
    const uint32_t sw = ((uint32_t)lane & 7u) << 4;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const uint32_t q = *reinterpret_cast<const uint32_t*>(row + ((16u * (uint32_t)(j >> 2)) ^ sw) + 4 * (j & 3));
        const int32_t d = (int32_t)(q - qp);
        qp = q;
        w[j] = (uint32_t)abs(d);
        orb |= w[j];
        sg = __funnelshift_l((uint32_t)d, sg, 1);
    }
    const uint32_t L = code_length(orb), nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    bit_transpose<32>(w);
    __syncwarp();   // every lane has read its row
    uint32_t* dst = image + 8 + (incl - nw);
    reinterpret_cast<unsigned char*>(image)[lane] = (unsigned char)L;
    if (L) {
        dst[0] = __brev(sg);
#pragma unroll
        for (int k = 0; k < 31; ++k)
            if ((uint32_t)k < L) dst[1 + k] = w[k];
    }
    return __shfl_sync(kFull, incl, 31);
}

// General route for one round of a binary64 tile: any code length, ragged ends, straight from global memory into the
// round's slot, conversions by the definition itself.  Compact rather than fast.
__device__ __noinline__ uint32_t encode_round_general_f64(const double* __restrict__ xt, uint32_t len, uint32_t rd, double r, uint32_t* __restrict__ slot,
                                                          uint32_t* round_words, int32_t* outlier, unsigned long long* group_words, int lane)
{
    uint32_t status = 0;
    const uint32_t nb = (len + kBlock - 1) / kBlock;
    const uint32_t bi = 32u * rd + (uint32_t)lane;
    const uint32_t last = len - 1;
    uint32_t L = 0, sgw = 0;
    uint32_t m[32];
    if (bi < nb) {
        const uint32_t e0 = 32u * bi;
        const uint32_t ep = e0 ? e0 - 1u : 0u;
        const double tp = __dmul_rn(__ldg(xt + (ep < last ? ep : last)), r);
        bool out_of_range = !(fabs(tp) < 1073741824.0);   // also true for a NaN
        uint32_t qp = (uint32_t)__double2int_rn(tp);
        uint32_t sg = 0, ob = 0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const uint32_t e = e0 + (uint32_t)j;
            const double t = __dmul_rn(__ldg(xt + (e < last ? e : last)), r);
            out_of_range = out_of_range || !(fabs(t) < 1073741824.0);
            const uint32_t q = (uint32_t)__double2int_rn(t);
            const int32_t dd = (int32_t)(q - qp);
            qp = q;
            const uint32_t sm = (uint32_t)(dd >> 31);
            m[j] = (((uint32_t)dd ^ sm) - sm) & 0x7FFFFFFFu;   // |delta|; the mask only matters after a range error
            ob |= m[j];
            sg = __funnelshift_l((uint32_t)dd, sg, 1);
        }
        if (out_of_range) status |= kStRange;
        L = code_length(ob);
        sgw = __brev(sg);
        bit_transpose<32>(m);
    }
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    reinterpret_cast<unsigned char*>(slot)[lane] = (unsigned char)L;
    if (L) {
        uint32_t* d = slot + 8 + (incl - nw);
        d[0] = sgw;
#pragma unroll
        for (int k = 0; k < 31; ++k)
            if ((uint32_t)k < L) d[1 + k] = m[k];
    }
    if (lane == 31) { *round_words = incl; atomicAdd(group_words, (unsigned long long)incl); }
    if (rd == 0 && lane == 0) *outlier = __double2int_rn(__dmul_rn(__ldg(xt), r));
    return status;
}

// Step 1 of a binary64 compression (step 2 is place_kernel): a CTA of four warps takes a tile, a warp a round.  A round's
// 1024 elements come straight into registers, 16 bytes per lane and load and all loads in flight at once, and are made
// codes there, in the order of memory (a code does not depend on its neighbours); the codes go through 4 KiB of shared
// memory to their blocks' lanes, and the image leaves from the same place by one bulk store.  Partial rounds (the end
// of the array) take the general route.
//
// What bounds it: latency (one round per warp: load, pass, transposes, store), so what counts is how many warps an SM
// holds.  Rounds brought as 8-KiB stages by the copy engine, three to a warp, left room for eight: 23.9 us with the
// placement for 2^23 elements at code lengths around 5; this form, twenty warps (five CTAs, 100 registers), takes 20.7
// (10.3 is what the reads take).  Four CTAs 21.9, six (spills) 23.9, persistent CTAs 22.2, with the next tile asked into L2
// 24.4, the first tile not asked for in advance 21.5.
template <bool ALIGNED>
__device__ __forceinline__ void load_codes_f64(uint32_t* image, const double* __restrict__ xr, double r, uint32_t& hi_max, int lane)
{
    constexpr int kLoads = ALIGNED ? 16 : 32;
    double v[32];
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
        if (ALIGNED) {
            const double2 d = __ldg(reinterpret_cast<const double2*>(xr) + 32 * k + lane);
            v[2 * k] = d.x; v[2 * k + 1] = d.y;
        } else v[k] = __ldg(xr + 32 * k + lane);
    }
    uint32_t q[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const double t = __dmul_rn(v[k], r);
        hi_max = max(hi_max, (uint32_t)__double2hiint(t) & 0x7FFFFFFFu);
        q[k] = (uint32_t)__double2loint(__dadd_rn(t, kMagic52));
    }
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
        if (ALIGNED) {
            const uint32_t row = 2u * (uint32_t)k + ((uint32_t)lane >> 4), chunk = ((uint32_t)lane & 15u) >> 1;
            *reinterpret_cast<uint2*>(reinterpret_cast<char*>(image) + 128u * row + ((16u * chunk) ^ ((row & 7u) << 4)) + 8u * ((uint32_t)lane & 1u)) =
                make_uint2(q[2 * k], q[2 * k + 1]);
        } else
            *reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(image) + stage_chunk_byte((uint32_t)k, (uint32_t)lane >> 2) + 4u * ((uint32_t)lane & 3u)) = q[k];
    }
}
__global__ void __launch_bounds__(kCodecThreads, kEnc64Ctas) encode_rounds_f64_kernel(const double* __restrict__ x, unsigned long long n,
                                                                                     Workspace ws, ParamsF64 hp, int bound_source, unsigned early)
{
    __shared__ Round64Shared shared[kCodecWarps];
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t rd = (uint32_t)tid >> 5, e0 = rd * (uint32_t)kRound;
    const bool aligned = (((uintptr_t)x) & 15u) == 0;
    const unsigned long long t = blockIdx.x;
    // before the kernel in front is waited for: the warp's round is asked into L2 (a prefetch only moves lines there; L2 stays
    // coherent with what that kernel still writes).  `early`: the CTAs that may be there by then, one full load of the device
    if (aligned && lane == 0 && t < early && t * kTile + e0 + (unsigned)kRound <= n) bulk_prefetch_l2(x + t * kTile + e0, kRound * 8u);
    pdl_enter();
    uint32_t* image = shared[rd].image;
    uint32_t status = 0;
    const ParamsF64 prm = bound_of_f64(ws, hp, bound_source);
    const double r = prm.r;
    const uint32_t u = 4u * (uint32_t)t + rd;
    uint32_t len = 0;
    if (prm.valid && n) len = (uint32_t)(n - t * kTile < (unsigned long long)kTile ? n - t * kTile : (unsigned long long)kTile);
    if (e0 >= len) {      // a round beyond the tile's last block, or a tile without elements
        if (lane == 0) ws.round_words[u] = 0;
        return;
    }
    uint32_t* slot = ws.slots + (size_t)u * kRoundSlotWords;
    unsigned long long* group = ws.group_acc + (uint32_t)(t >> 5);
    const double* xr = x + t * kTile + e0;
    bool general = e0 + (uint32_t)kRound > len;
    if (!general) {
        const double front = __dmul_rn(rd ? __ldg(xr - 1) : 0.0, r);
        uint32_t hi_max = (uint32_t)__double2hiint(front) & 0x7FFFFFFFu;
        if (aligned) load_codes_f64<true>(image, xr, r, hi_max, lane);
        else load_codes_f64<false>(image, xr, r, hi_max, lane);
        __syncwarp();
        general = __any_sync(kFull, hi_max >= kRangeHi);
        if (!general) {
            const uint32_t first = image[0];
            const uint32_t q_front = lane ? *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(image) +
                                                                               stage_chunk_byte((uint32_t)lane - 1u, 7u) + 12u)
                                          : (rd ? (uint32_t)__double2loint(__dadd_rn(front, kMagic52)) : first);
            uint32_t words = encode_codes_class<8>(image, q_front, lane);
            if (words == ~0u) words = encode_codes_class<16>(image, q_front, lane);
            if (words == ~0u) words = encode_codes_wide(image, q_front, lane);
            __syncwarp();   // the words written by all lanes are visible to lane 0's store
            if (lane == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(slot), "r"(smem_u32(image)),
                             "r"((32u + 4u * words + 15u) & ~15u) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                ws.round_words[u] = words;
                asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(group), "l"((unsigned long long)words) : "memory");
                if (rd == 0) ws.outliers[t] = (int32_t)first;
            }
        }
    }
    if (general) status |= encode_round_general_f64(x + t * kTile, len, rd, r, slot, ws.round_words + u, ws.outliers + t, group, lane);
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // the stores have read shared memory and are complete
    if (status) atomicOr(ws.status, status);
}

// ------------------------------------------------------------------------------------------------ binary64, decompress

// A code as a binary64, exactly: the word q ^ 2^31 under the exponent of 2^52 is 2^52 + 2^31 + q.
__device__ __forceinline__ double code_to_double(int32_t q)
{
    return __dsub_rn(__hiloint2double(0x43300000, (int)((uint32_t)q ^ 0x80000000u)), kIntBias);
}

// The lane's 32 elements from the biased deltas (word i, field h = element N h + i) as values in the lane's two rows of a
// stage: running code (32-bit integers), one conversion and one multiplication.
template <int N>
__device__ __forceinline__ void expand_block_f64(const uint32_t (&w)[N], int32_t code_in_front, double s, char* rows, uint32_t sw0)
{
    uint32_t run = (uint32_t)code_in_front;
#pragma unroll
    for (int h = 0; h < 32 / N; ++h) {
        const uint32_t sel = N == 8 ? 0x4440u + (uint32_t)h : 0x4410u + 0x0022u * (uint32_t)h;   // byte (pair) h of a word, zero above it
#pragma unroll
        for (int q = 0; q < N / 2; ++q) {
            double o[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                run = run + prmt(w[2 * q + e], 0u, sel) - (1u << (N - 1));
                o[e] = __dmul_rn(code_to_double((int32_t)run), s);
            }
            *reinterpret_cast<double2*>(rows + pair_chunk_byte((uint32_t)(h * (N / 2) + q), sw0)) = make_double2(o[0], o[1]);
        }
    }
}

// One round of a binary64 tile by the general route: any code length.  blob: the tile's words,
// pay_off: payload words of the rounds before, code: the code in front of the round.
__device__ __noinline__ void decode_round_general_f64(const uint32_t* blob, uint32_t padw, uint32_t L, uint32_t* pay_off_io, int32_t* code_io,
                                                      double s, double* stage, int lane)
{
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    const uint32_t* pay = blob + 1 + padw + *pay_off_io + (incl - nw);
    *pay_off_io += __shfl_sync(kFull, incl, 31);
    const uint32_t sign = L ? pay[0] : 0u;
    uint32_t w[32];
    int32_t total = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        w[k] = (uint32_t)k < L ? pay[1 + k] : 0u;
        total += (__popc(w[k]) - 2 * __popc(w[k] & sign)) << k;
    }
    int32_t inc = total;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t v = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += v;
    }
    bit_transpose<32>(w);
    int32_t run = *code_io + inc - total;
    *code_io += __shfl_sync(kFull, inc, 31);
    char* rows = reinterpret_cast<char*>(stage) + 256 * lane;
    const uint32_t sw0 = (2u * (uint32_t)lane) & 7u;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        run += ((sign >> j) & 1u) ? -(int32_t)w[j] : (int32_t)w[j];
        *reinterpret_cast<double*>(rows + pair_chunk_byte((uint32_t)j >> 1, sw0) + 8u * (j & 1)) = __dmul_rn(__int2double_rn(run), s);
    }
}

// `count` elements of a stage to global memory, coalesced (ragged ends).
__device__ __noinline__ void store_round_ragged_f64(double* __restrict__ y, const double* stage, uint32_t count, int lane)
{
#pragma unroll 4
    for (uint32_t k = 0; k < 32u; ++k) {
        const uint32_t e = 32u * k + (uint32_t)lane;
        const uint32_t row = e >> 4, chunk = (e & 15u) >> 1;
        if (e < count) y[e] = *reinterpret_cast<const double*>(reinterpret_cast<const char*>(stage) + stage_chunk_byte(row, chunk) + 8u * (e & 1u));
    }
}

constexpr uint32_t kBlob64Bufs = 3;
constexpr int kDecode64Ctas = 3;
// binary64 streams carry the step as one binary64 in the words where binary32 streams have bound and step
__device__ __forceinline__ double step_of_f64(const DecodeWork& w) { return __hiloint2double(__float_as_int(w.s), __float_as_int(w.eb_abs)); }
struct alignas(1024) Decode64Shared {
    double out[kTileWarps][kRound];
    alignas(16) uint32_t blob[kBlob64Bufs][kBlobBufWords];
    DecodeWork work[kBlob64Bufs];
    alignas(16) int32_t sums[kBlob64Bufs][kTileWarps];
    alignas(8) unsigned long long landed[kBlob64Bufs], ready[kBlob64Bufs], free[kBlob64Bufs];
};

// The decomposition of decode_tiles_kernel (a tile per CTA, a round per warp, a fifth warp that fetches) with 8-KiB
// stages.  What bounds it: the stores (10.3 us for 2^23 elements), then the ramps of the launch.  A warp per tile, its four
// rounds in a row, took 16.7 us for 2^23 elements at code lengths around 5 and 31.2 for 2^24 at 8.5; this form takes 15.7 and
// 28.5.  Two buffers and four CTAs per SM 17.5 and 29.2.
// Full rounds leave by one tensor store when y starts on a 16-byte boundary (and has a map), by plain coalesced stores
// otherwise.
__global__ void __launch_bounds__(kDecodeThreads, kDecode64Ctas) decode_tiles_f64_kernel(const __grid_constant__ JobBatchT<1> jb, const __grid_constant__ CUtensorMap map, Workspace ws)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Decode64Shared& sh = *reinterpret_cast<Decode64Shared*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t rd = (uint32_t)tid >> 5;
    if (tid == 0) {
#pragma unroll
        for (int k = 0; k < (int)kBlob64Bufs; ++k) { mbar_init(&sh.landed[k], 1); mbar_init(&sh.ready[k], 1); mbar_init(&sh.free[k], kTileWarps); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_enter();
    uint32_t status = 0;
    if (rd == kTileWarps) {
        fetch_tiles<kBlob64Bufs, false, false, true, false>(jb, blockIdx.x, nullptr, sh.blob, sh.work, sh.landed, sh.ready, sh.free, status, lane, [](const DecodeWork&, uint32_t) { return true; });
        if (status) atomicOr(ws.status, status);
        return;
    }
    const uint32_t e0 = rd * (uint32_t)kRound, sw0 = (2u * (uint32_t)lane) & 7u;
    double* stage = sh.out[rd];
    char* rows = reinterpret_cast<char*>(stage) + 256 * lane;
    double* __restrict__ y = reinterpret_cast<double*>(jb.job[0].y);
    const bool mapped = (((uintptr_t)y) & 15u) == 0;
    for (uint32_t i = 0;; ++i) {
        const uint32_t b = i % kBlob64Bufs;
        if (!mbar_wait(&sh.ready[b], (i / kBlob64Bufs) & 1u)) { status |= kStTimeout; break; }
        const DecodeWork& w = sh.work[b];
        const uint32_t kind = w.kind;
        if (kind == kTileNone) break;
        // the tile's facts are copied: the buffer is given back in the middle of the decoding
        const uint32_t len = w.len, before = w.before[rd];
        const unsigned long long start = w.start;
        const double s = step_of_f64(w);
        const int32_t outlier = w.outlier;
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
        const uint32_t bi = 32u * rd + (uint32_t)lane;
        // a blob larger than the buffer is read where it is
        const uint32_t* blob = kind == kTileFast ? sh.blob[b] + w.lead : (const uint32_t*)(uintptr_t)w.src;
        const uint32_t L = bi < nb ? (uint32_t) reinterpret_cast<const unsigned char*>(blob + 1)[bi] : 0u;
        if (kind == kTileFast && !__any_sync(kFull, L > 15u)) {
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
                expand_block_f64<8>(v, code, s, rows, sw0);
            } else {
                uint32_t v[16];
                load_deltas<16>(pay, L, !__any_sync(kFull, L > 8u), v, sum);
                const int32_t incl = warp_incl_scan_s(sum, lane);
                const int32_t code = code_in_front(sh.sums[b], __shfl_sync(kFull, incl, 31), outlier, rd, lane) + incl - sum;
                give_back();
                drained();
                expand_block_f64<16>(v, code, s, rows, sw0);
            }
        } else {
            uint32_t off = before;
            int32_t code = 0;
            skip_round(blob, padw, L, &off, &code, lane);
            code = code_in_front(sh.sums[b], code, outlier, rd, lane);
            off = before;
            drained();
            decode_round_general_f64(blob, padw, L, &off, &code, s, stage, lane);
            __syncwarp();
            give_back();
        }
        __syncwarp();   // the stage's rows, written by all lanes, are visible
        if (mapped && e0 + (uint32_t)kRound <= len) {
            if (lane == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                             ::"l"(&map), "r"(0), "r"((int)(uint32_t)((start + e0) >> 4)), "r"(smem_u32(stage)) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        } else if (e0 < len) {
            store_round_ragged_f64(y + start + e0, stage, len - e0 < (uint32_t)kRound ? len - e0 : (uint32_t)kRound, lane);
            __syncwarp();   // the stage is read before the next round overwrites it
        }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (status) atomicOr(ws.status, status);
}
