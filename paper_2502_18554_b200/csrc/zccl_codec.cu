// fZ-light codec kernels for sm_100a: encoder, decoder and the fused decode + reduce + encode hop.
//
// Work decomposition: ONE LANE OWNS ONE 32-ELEMENT BLOCK.  A warp works on a round of 32 blocks (1024 elements,
// a quarter of a tile); lane l holds the 32 consecutive elements of block l in registers.  Everything the format
// asks of a block then happens inside one thread, with no shuffle, vote or barrier:
//   * quantise and 1-D Lorenzo delta: fp32 on the FMA pipe (t + 1.5 * 2^23 rounds to nearest even, deltas of two
//     such values are exact, |delta| + 2^23 has the magnitude in its mantissa);
//   * code length: OR of the 32 magnitudes, one count-leading-zeros;
//   * bit planes: the magnitudes are packed four (code lengths up to 8), two (up to 16) or one to a word by byte
//     permutes and an in-register bit-matrix transpose (3, 4 or 5 stages of shift + bit-select pairs) turns them
//     into plane words; the decoder runs the same transpose backwards and gets the block's delta sum from byte dot
//     products of the deltas (other tile sizes, two compressed operands: population counts of the planes);
//   * sign word: one funnel shift per element.
// A warp needs its neighbours only for the prefix sum of the blocks' sizes and, when it decodes, of the blocks'
// delta sums (one shuffle scan per round each).
//
// Memory.  A lane wants 128 consecutive bytes per block while global accesses must be contiguous across the warp,
// so rounds go through shared memory.  The array is described to the copy engine as rows of 32 floats (one tensor
// map per chunk-operation, built on the host); one tiled tensor copy brings a round's 32 rows into a 4 KiB stage
// in the 128-byte swizzle (16-byte chunk c of row t at c ^ (t & 7)), completion on an mbarrier; the lanes' 128-bit row
// reads and (decoder) row writes are free of bank conflicts; decoded rounds leave by a tensor store.  Ragged or
// misaligned rounds take plain loads and stores into the same layout.  Compressed bytes move with untiled bulk
// copies.
//
// The kernels of binary32 streams of 4096-element tiles are in files of their own, included below:
//   zccl_tiles.cuh   compression of few tiles: encode_tiles_kernel (a tile per CTA, which finds its place itself)
//   zccl_stream.cuh  compression of many: encode_stream_kernel (CTAs take tile after tile and find their places)
//   zccl_decode.cuh  decompression
//   zccl_hop.cuh     the fused hop, with its placement inside or by place_kernel
//   zccl_ring.cuh    the emulated ring reduce-scatter in one launch
// This file has what they share, place_kernel (one CTA per group of 32 tiles turns the group sums in front of it and its
// own rounds' sizes into stream positions and moves the payloads from the slots), the hop with two compressed
// operands, which has a decomposition of its own (a warp per tile or part of one), and the launch functions.
// zccl_codec_f64.cuh has the kernels for binary64, zccl_codec_tiled.cuh those for other tile sizes.
#include "zccl_device.cuh"

#include <cuda.h>
#include <cstring>
#include <mutex>

namespace zccl {
namespace {

constexpr int kCodecWarps = 4;                        // warps per CTA, each with tiles of its own
constexpr int kCodecThreads = 32 * kCodecWarps;
constexpr int kRound = 32 * kBlock;                   // elements per round: one block per lane
constexpr int kRoundsPerTile = kTile / kRound;
constexpr int kLWords = kBlocksPerTile / 4;           // code-length words of a full tile

// ------------------------------------------------------------------------------------------------ small pieces

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, int lane)
{
    (void)lane;
    // The shuffle itself says which lanes have one in front: a comparison less per step.  With ld_shared4: decoder 541 -> 505
    // instructions per round, hop 963 -> 924; us: 2^24 field values 15.96 -> 15.9 and 30.8 -> 30.1, 2^27 decompressed 97.3 -> 96.6,
    // 2^28 gradients compressed 268 -> 265, 8 x 2^21 Allreduce 69.3 -> 67.9.
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tshfl.sync.up.b32 t|p, %0, %1, 0, 0xffffffff;\n\t@p add.u32 %0, %0, t;\n\t}" : "+r"(v) : "r"(d));
    return v;
}

// The scan as the compiler schedules it among its neighbours, for launches whose warps have one round each (latency, not issue):
// hop of 25 tiles 6.35 us, with warp_incl_scan, which saves instructions but keeps its place, 6.5; compression of 256 tiles
// 5.1 and 5.45.
template <class V>
__device__ __forceinline__ V plain_scan(V v, int lane)
{
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const V t = __shfl_up_sync(kFull, v, d);
        if (lane >= d) v += t;
    }
    return v;
}

// In-register bit-matrix transpose of N words (N = 8, 16, 32).  Word i holds 32 / N values of N bits each: value
// number N * h + i sits in bits [N h, N h + N).  Afterwards word k holds plane k: bit N * h + i = bit k of that value.
// Each stage exchanges, between words i and i + d, the bits whose in-value position has bit d set against those that
// have it clear: two shifts and two bit-selects per pair.  The transpose is its own inverse.
// (The stages are separate instantiations rather than a loop over d: left to the unroller, the 16-word form kept its
// words in local memory, indexed at run time.)
template <int N, int D>
__device__ __forceinline__ void bit_transpose_stage(uint32_t (&w)[N])
{
    constexpr uint32_t m = D == 16 ? 0x0000FFFFu : D == 8 ? 0x00FF00FFu : D == 4 ? 0x0F0F0F0Fu : D == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (i & D) continue;
        const uint32_t a = w[i], b = w[i + D];
        w[i] = (a & m) | ((b << D) & ~m);
        w[i + D] = ((a >> D) & m) | (b & ~m);
    }
}
template <int N>
__device__ __forceinline__ void bit_transpose(uint32_t (&w)[N])
{
    if constexpr (N >= 32) bit_transpose_stage<N, 16>(w);
    if constexpr (N >= 16) bit_transpose_stage<N, 8>(w);
    bit_transpose_stage<N, 4>(w);
    bit_transpose_stage<N, 2>(w);
    bit_transpose_stage<N, 1>(w);
}

// ------------------------------------------------------------------------------------------------ stages

// A stage holds one round: row t = the 32 floats of block t (128 bytes), its 16-byte chunk c stored at chunk
// position c ^ (t & 7) of the row, so that the lanes' 128-bit reads of their own rows fall into different banks.
// That is the 128-byte swizzle of the tensor copy engine: a full round of an array that starts on a 16-byte boundary
// is brought in by ONE tiled tensor copy (32 rows x 32 floats of the array seen as rows of 32 floats; issued by one
// lane, completion on the stage's mbarrier).  Besides costing no instructions, this keeps the load/store path free:
// with the input streamed through it (16-byte asynchronous copies were tried first), every latency-critical load
// of the placement (the states of other tiles) queued up behind kilobytes of input and took microseconds.  Stages
// must start on a 1024-byte boundary (the swizzle works on address bits).  Other rounds (ragged ends, unaligned
// arrays) are loaded element by element, positions beyond the tile's end repeating its last element (so that the
// padding of the last block has zero deltas).
__device__ __forceinline__ uint32_t stage_chunk_byte(uint32_t row, uint32_t chunk) { return row * 128u + ((chunk ^ (row & 7u)) << 4); }

__device__ __noinline__ void load_round_ragged(float* stage, const float* __restrict__ xt, uint32_t e0, uint32_t len, int lane)
{
    // all loads in flight at once: four at a time, the one ragged tile of an array was what a launch ended with (1332 tiles, the
    // last one five elements short: 13.6 us, 10.3 so; hop of 25 tiles, 100 003 elements, 7.0 and 6.0)
    const uint32_t last = len - 1;
    float v[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const uint32_t e = e0 + 32u * k + (uint32_t)lane;
        v[k] = __ldg(xt + (e < last ? e : last));
    }
#pragma unroll
    for (int k = 0; k < 32; ++k)
        *reinterpret_cast<float*>(reinterpret_cast<char*>(stage) + stage_chunk_byte(k, (uint32_t)lane >> 2) + 4 * (lane & 3)) = v[k];
}
// Tiled tensor copy of rows [row0, row0 + 32) of the array behind `map` into a stage (one thread).
__device__ __forceinline__ void tensor_load_round(float* stage, unsigned long long* bar, const CUtensorMap* map, uint32_t row0)
{
    mbar_expect_tx(bar, kRound * 4);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(smem_u32(stage)), "l"(map), "r"(0), "r"((int)row0), "r"(smem_u32(bar)) : "memory");
}

// The last element of a row of a stage (the element in front of the next row's block).
__device__ __forceinline__ float read_last_of_row(const float* stage, uint32_t row)
{
    return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(stage) + stage_chunk_byte(row, 7) + 12);
}

// ------------------------------------------------------------------------------------------------ one block, encode

// fp32 pass over the block in this lane's row of a stage: deltas against the element in front (xprev), magnitudes
// packed 32 / N to a word for the N-bit transpose (word i, field h = element N h + i), OR of the magnitude words, sign
// word, and the sum of squares of x * r that tells whether fp32 was exact (below 2^43: every |x r| < 2^21.5).  N = 8
// serves code lengths up to 8, N = 16 up to 16.  The loop over groups of N elements is kept rolled: every word shifts
// down by one field and takes the new magnitude on top, so the body is the same for every group and stays small
// enough for the instruction cache of a scheduler (unrolled, the kernel stalled on instruction fetch).
template <int N>
struct BlockPack {
    uint32_t w[N];
    uint32_t sign, orb;
    float guard;
};
template <int N>
__device__ __forceinline__ void block_pass(const char* row, uint32_t sw, float xprev, float r, BlockPack<N>& o)
{
    const float tp = __fmul_rn(xprev, r);
    float cp = __fadd_rn(tp, kRoundMagic);
    // the multiplications, the additions of the rounding constant and the guard's sums go two elements to an instruction
    // (sm_100's packed fp32: each half rounds as the scalar operation does; 23.3 -> 23.0 us per 64 MiB)
    float2 acc2 = make_float2(__fmul_rn(tp, tp), 0.0f);
    const float2 r2 = make_float2(r, r), magic2 = make_float2(kRoundMagic, kRoundMagic);
    uint32_t orb = 0, sg = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) o.w[i] = 0;
#pragma unroll 1
    for (uint32_t g = 0; g < 32u / N; ++g) {
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(row + ((16u * (g * (N / 4) + q)) ^ sw));
            const float2 t01 = __fmul2_rn(make_float2(v.x, v.y), r2), t23 = __fmul2_rn(make_float2(v.z, v.w), r2);
            acc2 = __ffma2_rn(t01, t01, acc2);
            acc2 = __ffma2_rn(t23, t23, acc2);
            // (the products are used twice, by the guard and here; the compiler was seen to contract a packed product with
            // ONE use and the packed addition behind it into a packed fused multiply-add whatever --fmad says, which the
            // full-size parity tests would show as codes that differ at ties)
            const float2 c01 = __fadd2_rn(t01, magic2), c23 = __fadd2_rn(t23, magic2);
            const float cs[4] = {c01.x, c01.y, c23.x, c23.y};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float c = cs[e];
                const float d = __fsub_rn(c, cp);
                cp = c;
                const uint32_t m = __float_as_uint(__fadd_rn(fabsf(d), kTwo23));   // bits 0..22: |delta|
                orb |= m;
                sg = __funnelshift_l(__float_as_uint(d), sg, 1);                  // sign of element j ends up in bit 31 - j
                o.w[4 * q + e] = prmt(o.w[4 * q + e], m, N == 8 ? 0x4321u : 0x5432u);
            }
        }
    }
    o.sign = __brev(sg);
    o.orb = orb & 0x007FFFFFu;
    o.guard = __fadd_rn(acc2.x, acc2.y);
}

__device__ __forceinline__ uint32_t code_length(uint32_t orb) { return 32u - (uint32_t)__clz((int)orb); }

// Largest |x r| of a block (the rare recheck behind the precision warning).
__device__ __forceinline__ float block_tmax(const char* row, uint32_t sw, float r)
{
    float tm = 0.0f;
#pragma unroll 1
    for (uint32_t q = 0; q < 8; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(row + ((16u * q) ^ sw));
        tm = fmaxf(fmaxf(tm, fabsf(__fmul_rn(v.x, r))), fmaxf(fabsf(__fmul_rn(v.y, r)), fmaxf(fabsf(__fmul_rn(v.z, r)), fabsf(__fmul_rn(v.w, r)))));
    }
    return tm;
}

// What the lanes carry from round to round of a tile they encode.
struct EncodeCarry {
    uint32_t pay_used;   // payload words of the rounds so far
    bool wide;           // the round before had a code length above 8: start with the 16-bit pass
};

// One round of the encoder's back end, for the block in this lane's row of a stage (row: its first byte, sw: the
// lane's chunk swizzle; xprev: the element in front of the block).
// Appends the round's payload to the tile's blob in shared memory (word i of the blob at blob[org + sgn * i]) and
// sets the lane's code-length byte.  `active`: the block exists (ragged tiles have fewer than 128).  Returns 0 when
// done; otherwise nothing was stored: 1 when the round is beyond what this path covers (a code length above 16, or
// codes for which fp32 is not exact) and the whole tile has to take the general route, 2 when the blob would
// outgrow `pay_cap` payload words.  `mid` is called once, by all lanes, when the rows have been read and the sizes are
// known, before anything is stored.
// This is one width class (N = 8 or 16 bits per packed magnitude); it returns 3, with nothing stored and `mid` not
// called, when a lane's code is longer than N.
template <int N, class Mid>
__device__ __forceinline__ int encode_round_n(const char* row, uint32_t sw, float xprev, float r, bool active, uint32_t block_in_tile,
                                              uint32_t lbytes, uint32_t* __restrict__ blob, uint32_t org, int sgn, uint32_t pay_base,
                                              uint32_t pay_cap, EncodeCarry& cy, int lane, uint32_t& status, Mid&& mid)
{
    BlockPack<N> a;
    block_pass<N>(row, sw, xprev, r, a);
    uint32_t L = active ? code_length(a.orb) : 0u;
    if (N == 8 && __any_sync(kFull, L > 8u)) return 3;
    const bool beyond = !(a.guard < kGuardExact) || L > 16u;
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    const uint32_t round_total = __shfl_sync(kFull, incl, 31);
    mid();   // the caller's business between the two halves (all lanes, once per round)
    if (__any_sync(kFull, beyond)) return 1;
    if (cy.pay_used + round_total > pay_cap) return 2;
    if (a.guard >= kGuardSmall && block_tmax(row, sw, r) > 32768.5f) status |= kStPrecision;
    __syncwarp();   // every lane has read its row for the last time: the blob may lie over the stage
    if (L) {
        uint32_t* dst = blob + ((int)org + sgn * (int)(pay_base + cy.pay_used + (incl - nw)));
        dst[0] = a.sign;
        bit_transpose<N>(a.w);
#pragma unroll
        for (int k = 0; k < N; ++k)
            if ((uint32_t)k < L) dst[sgn * (1 + k)] = a.w[k];
    }
    if (block_in_tile < lbytes) {
        const uint32_t wi = 1u + (block_in_tile >> 2);
        reinterpret_cast<unsigned char*>(blob + (sgn > 0 ? org + wi : org - wi))[block_in_tile & 3u] = (unsigned char)L;
    }
    cy.pay_used += round_total;
    cy.wide = __any_sync(kFull, L > 8u);
    return 0;
}

// One width class for the whole warp: a pass at 8 bits first unless the round before was wide; if any lane then has a
// longer code, every lane repeats the pass at 16 bits (the warp would execute those instructions anyway, and with
// one class at a time only one set of packed words is alive).
template <class Mid>
__device__ __forceinline__ int encode_round(const char* row, uint32_t sw, float xprev, float r, bool active, uint32_t block_in_tile,
                                            uint32_t lbytes, uint32_t* __restrict__ blob, uint32_t org, int sgn, uint32_t pay_base,
                                            uint32_t pay_cap, EncodeCarry& cy, int lane, uint32_t& status, Mid&& mid)
{
    if (!cy.wide) {
        const int rc = encode_round_n<8>(row, sw, xprev, r, active, block_in_tile, lbytes, blob, org, sgn, pay_base, pay_cap, cy, lane, status, mid);
        if (rc != 3) return rc;
    }
    return encode_round_n<16>(row, sw, xprev, r, active, block_in_tile, lbytes, blob, org, sgn, pay_base, pay_cap, cy, lane, status, mid);
}

// ---- general route: any code length, any alignment, codes up to 2^30, blobs of any size; straight from and to
// global memory, integer conversion (the definition itself).  Compact rather than fast.

// Sign word and planes of block `bi` of a tile (len elements at xt) into out[0 .. 32] (out[0] = sign word, out[1 + k]
// = plane k); returns the code length.  Positions beyond the tile's end repeat its last element.
__device__ __noinline__ uint32_t general_block(const float* __restrict__ xt, uint32_t bi, uint32_t len, float r, uint32_t* out, float* tmax)
{
    const uint32_t last = len - 1;
    const uint32_t e0 = 32u * bi;
    const uint32_t ep = e0 ? e0 - 1u : 0u;
    const float tp = __fmul_rn(__ldg(xt + (ep < last ? ep : last)), r);
    float tm = fmaxf(*tmax, fabsf(tp));
    uint32_t qp = (uint32_t)__float2int_rn(tp);
    uint32_t m[32];
    uint32_t sg = 0, ob = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const uint32_t e = e0 + (uint32_t)j;
        const float t = __fmul_rn(__ldg(xt + (e < last ? e : last)), r);
        tm = fmaxf(tm, fabsf(t));
        const uint32_t q = (uint32_t)__float2int_rn(t);
        const int32_t dd = (int32_t)(q - qp);
        qp = q;
        const uint32_t sm = (uint32_t)(dd >> 31);
        m[j] = (((uint32_t)dd ^ sm) - sm) & 0x7FFFFFFFu;   // |delta|; the mask only matters after a range error
        ob |= m[j];
        sg = __funnelshift_l((uint32_t)dd, sg, 1);
    }
    *tmax = tm;
    bit_transpose<32>(m);
    out[0] = __brev(sg);
#pragma unroll
    for (int k = 0; k < 32; ++k) out[1 + k] = m[k];
    return code_length(ob);
}

// One tensor map per job of a launch: the job's input seen as rows of 32 floats.
template <int CAP>
struct alignas(64) TileMapsT {
    CUtensorMap m[CAP];
};
using TileMaps = TileMapsT<kMaxJobs>;

// ------------------------------------------------------------------------------------------------ two steps: slots, places
//
// Hops of more tiles than are resident together, compressions of binary64 and of other tile sizes.  Step 1: rounds (32 blocks
// of a tile, one per lane) go to their fixed slots in the workspace (code-length bytes, then payload), with their sizes and,
// for a tile's first round, the tile's first quantised value; nobody waits for anybody.  Step 2 (place_kernel) turns the slots
// into the stream.

constexpr int kRoundBufWords = 8 + 32 * 17;   // code-length bytes + payload at code length 16 (longer codes go the general route)
constexpr int kRoundStages = 3;
constexpr int kEncodeCtas = 8;
constexpr int kDecodeCtas = 5;
constexpr int kHopCtas = 4;
constexpr uint32_t kHopBlobs = 2;
template <int STAGES>
struct alignas(1024) RoundWarpSharedT {
    float stage[STAGES][kRound];              // each on a 1024-byte boundary; a round is encoded in place and leaves from here
    alignas(16) float front[STAGES][4];       // the four elements in front of each stage's round
    alignas(8) unsigned long long bar[STAGES];
};
using RoundWarpShared = RoundWarpSharedT<3>;

// General route for one round: any code length, straight from global memory into the round's slot.
__device__ __noinline__ uint32_t encode_round_general(const float* __restrict__ xt, uint32_t len, uint32_t rd, float r, uint32_t* __restrict__ slot,
                                                      uint32_t* round_words, int32_t* outlier, unsigned long long* group_words, int lane)
{
    uint32_t status = 0;
    const uint32_t nb = (len + kBlock - 1) / kBlock;
    const uint32_t bi = 32u * rd + (uint32_t)lane;
    uint32_t planes[33];
    float tmax = 0.0f;
    uint32_t L = 0;
    if (bi < nb) L = general_block(xt, bi, len, r, planes, &tmax);
    if (!(tmax < 1073741824.0f)) status |= kStRange;
    else if (tmax > 32768.5f) status |= kStPrecision;
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    reinterpret_cast<unsigned char*>(slot)[lane] = (unsigned char)L;
    if (L) {
        uint32_t* d = slot + 8 + (incl - nw);
        for (uint32_t k = 0; k <= L; ++k) d[k] = planes[k];
    }
    if (lane == 31) { *round_words = incl; atomicAdd(group_words, (unsigned long long)incl); }
    if (rd == 0 && lane == 0) *outlier = __float2int_rn(__fmul_rn(__ldg(xt), r));
    return status;
}

// The same for a round whose values sit in a stage (the hop's sums): block `lane` of the round from the lane's row.
__device__ __noinline__ uint32_t encode_round_general_staged(const float* stage, float xprev, bool active, uint32_t rd, float r,
                                                             uint32_t* __restrict__ slot, uint32_t* round_words, int32_t* outlier,
                                                             unsigned long long* group_words, int lane)
{
    uint32_t status = 0;
    const char* row = reinterpret_cast<const char*>(stage) + 128 * lane;
    const uint32_t sw = ((uint32_t)lane & 7u) << 4;
    uint32_t m[32];
    uint32_t sg = 0, ob = 0;
    const float tp = __fmul_rn(xprev, r);
    float tm = fabsf(tp);
    uint32_t qp = (uint32_t)__float2int_rn(tp);
    const int32_t q0 = __float2int_rn(__fmul_rn(*reinterpret_cast<const float*>(row + sw), r));
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const float x = *reinterpret_cast<const float*>(row + ((16u * (uint32_t)(j >> 2)) ^ sw) + 4 * (j & 3));
        const float tt = __fmul_rn(x, r);
        tm = fmaxf(tm, fabsf(tt));
        const uint32_t q = (uint32_t)__float2int_rn(tt);
        const int32_t dd = (int32_t)(q - qp);
        qp = q;
        const uint32_t sm = (uint32_t)(dd >> 31);
        m[j] = (((uint32_t)dd ^ sm) - sm) & 0x7FFFFFFFu;
        ob |= m[j];
        sg = __funnelshift_l((uint32_t)dd, sg, 1);
    }
    uint32_t L = active ? code_length(ob) : 0u;
    if (active) {
        if (!(tm < 1073741824.0f)) status |= kStRange;
        else if (tm > 32768.5f) status |= kStPrecision;
    }
    bit_transpose<32>(m);
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    reinterpret_cast<unsigned char*>(slot)[lane] = (unsigned char)L;
    if (L) {
        uint32_t* d = slot + 8 + (incl - nw);
        d[0] = __brev(sg);
#pragma unroll
        for (int k = 0; k < 31; ++k)
            if ((uint32_t)k < L) d[1 + k] = m[k];
    }
    if (lane == 31) { *round_words = incl; atomicAdd(group_words, (unsigned long long)incl); }
    if (rd == 0 && lane == 0) *outlier = q0;
    return status;
}

// Step 2: one CTA per group of 32 tiles of a job turns the group's round slots into its piece of the stream.  The
// tiles' sizes follow from the rounds' sizes; the group's position is the sum of the groups of the job in front of
// it, whose sizes step 1 added up.
struct GroupTable {
    uint32_t begin[kMaxJobs + 1];   // first group (= CTA) of each job; begin[count] = number of groups
};
constexpr uint32_t kPlaceTiles = 32;    // a group of tiles per CTA, a tile per warp
constexpr int kPlaceThreads = 32 * (int)kPlaceTiles;
// Payload words of a tile that the copy engine brings (code lengths up to 11 on average; what is beyond is loaded by the
// lanes).  What bounds the placement: its traffic, slots in and stream out.  288 words per round, asked for together with
// the sizes, save a round trip but bring three times what a compressible array has, from DRAM when the slots are stale:
// compression of 2^26 smooth values 71.6 us, of 2^24 at code lengths around 4 21.2, of 2^28 at 8.5 371; by size 67.2, 20.9 and
// 360.  CTAs of 16 tiles two to an SM 67.4, 21.2, 369, three 74.6, 24.1, 389: more stores in flight get into each other's way.
constexpr uint32_t kPlaceWords = 1536;
constexpr int kPlaceUnroll = 8;      // loads of a round in flight per lane
constexpr size_t kPlaceSmemBytes = (size_t)kPlaceTiles * kPlaceWords * 4;

// Called by one warp of every CTA of the placement once the CTA has read the group sums it needs: the last CTA to
// get there puts the group sums back to zero while the others are still storing.  `used`: group sums the launch may have
// touched.  True (lane 0) there.
__device__ __forceinline__ bool rearm_groups(uint32_t used, const Workspace& ws, int lane)
{
    uint32_t last = 0;
    if (lane == 0) {
        __threadfence();
        last = atomicAdd(ws.done, 1u) == gridDim.x - 1 ? 1u : 0u;
    }
    if (!__shfl_sync(kFull, last, 0)) return false;
    for (uint32_t k = (uint32_t)lane; k < used; k += 32u) ws.group_acc[k] = 0ull;
    if (lane == 0) *ws.done = 0;
    return lane == 0;
}

// f64: a compression of binary64 input (bound in hp64, or from the range pass's keys; the header carries the step as one
// binary64); otherwise a hop (bound and step from the incoming stream's header).
__global__ void __launch_bounds__(kPlaceThreads) place_kernel(const __grid_constant__ JobBatch jb, const __grid_constant__ GroupTable gt, Workspace ws,
                                                              int f64, ParamsF64 hp64, int bound_source)
{
    // What this kernel reads before it waits for step 1 is older than step 1's launch: job table, the incoming
    // streams' headers, the resolved bound.
    __shared__ uint32_t s_words[kPlaceTiles], s_part[kPlaceTiles];
    __shared__ alignas(8) unsigned long long s_bar[kPlaceTiles];
    extern __shared__ __align__(16) unsigned char place_smem[];   // per warp: its tile's payload, round by round
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t* stage = reinterpret_cast<uint32_t*>(place_smem) + (size_t)warp * kPlaceWords;
    if (lane == 0) {
        mbar_init(&s_bar[warp], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    uint32_t status = 0;
    Params prm{0.0f, 1.0f, 1.0f, 1};
    double step64 = 0.0;
    if (f64) {
        hp64 = bound_of_f64(ws, hp64, bound_source);
        step64 = hp64.s; prm.valid = hp64.valid;
    }
    auto put_header = [&](uint32_t* out, int who, unsigned long long n, uint32_t nT) {
        if (!f64) { write_header(out, who, n, prm.eb_abs, prm.s, nT); return; }
        if (who < kHeaderWords) {
            const uint32_t words[kHeaderWords] = {kMagic, kVersionF64, (uint32_t)n, (uint32_t)(n >> 32), (uint32_t)__double2loint(step64),
                                                  (uint32_t)__double2hiint(step64), (uint32_t)kTile, nT};
            uint32_t hv = words[0];
#pragma unroll
            for (int k = 1; k < kHeaderWords; ++k) hv = who == k ? words[k] : hv;
            out[who] = hv;
        }
    };

    int j = 0;
    {
        int lo = 0, hi = jb.count;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (gt.begin[mid] <= blockIdx.x) lo = mid; else hi = mid;
        }
        j = lo;
    }
    const Job& job = jb.job[j];
    if (!f64) {   // a hop: bound and step are the incoming stream's, and the job counts only if its streams agree with it
        const StreamInfo h1 = read_header(job.in_c, job.in_cap);
        bool ok = h1.ok && h1.n == job.n;
        if (job.in_c2) {
            const StreamInfo h2 = read_header(job.in_c2, job.in2_cap);
            ok = ok && h2.ok && h2.n == job.n && __float_as_uint(h2.s) == __float_as_uint(h1.s);
        }
        prm.eb_abs = h1.eb_abs; prm.s = h1.s; prm.valid = ok ? 1 : 0;
    }
    pdl_enter();
    auto rearm = [&] {
        if (rearm_groups((jb.total_tiles >> 5) + (uint32_t)jb.count + 1u, ws, lane) && f64) settle_bound_f64(ws, hp64, bound_source);
    };
    const uint32_t g = blockIdx.x - gt.begin[j];
    const uint32_t tiles = (j + 1 < jb.count ? jb.job[j + 1].tile_begin : jb.total_tiles) - job.tile_begin;
    const unsigned long long n = job.n;
    const uint32_t nT = (uint32_t)((n + kTile - 1) / kTile);
    uint32_t* __restrict__ out = job.out;

    if (n == 0 || !prm.valid) {   // a job without elements, or no valid bound: header and length only
        const bool hdr = prm.valid && job.out_cap >= (unsigned)kHeaderBytes;
        if (tid == 0) *job.out_bytes = hdr ? kHeaderBytes : 0;
        if (hdr) put_header(out, tid, 0, 0);
        if (warp == kPlaceThreads / 32 - 1) rearm();
    } else {
        const uint32_t t0 = kPlaceTiles * g;                       // first tile of the CTA, within the job
        const uint32_t ntl = tiles - t0 < kPlaceTiles ? tiles - t0 : kPlaceTiles;   // tiles of the CTA
        const uint32_t T0 = job.tile_begin + t0;                   // the same, in the launch's numbering
        // Every warp asks for what is as large whatever the rounds' sizes (the sizes themselves, first value, its lane's
        // code-length word) and for its share of the sums of the groups in front; a round trip later for the payloads.
        const uint32_t tl = (uint32_t)warp;
        const bool mine = tl < ntl;
        const uint32_t T = T0 + (mine ? tl : 0u);
        const uint32_t* __restrict__ slot = ws.slots + (size_t)(4u * T) * kRoundSlotWords;
        const uint4 nq4 = *reinterpret_cast<const uint4*>(ws.round_words + 4u * T);
        const uint32_t lword = slot[(size_t)(lane >> 3) * kRoundSlotWords + (lane & 7)];   // code-length word `lane` of the tile
        const uint32_t first = (uint32_t)ws.outliers[T];
        unsigned long long part = 0;
        {
            const uint32_t gslot0 = (job.tile_begin >> 5) + (uint32_t)j;
            for (uint32_t k = (uint32_t)tid; k < g; k += kPlaceThreads) part += ws.group_acc[gslot0 + k];
        }
        const uint32_t nqs[kRoundsPerTile] = {nq4.x, nq4.y, nq4.z, nq4.w};
        uint32_t have[kRoundsPerTile];
        {
            uint32_t room = kPlaceWords;
#pragma unroll
            for (int q = 0; q < kRoundsPerTile; ++q) {
                have[q] = min((nqs[q] + 3u) & ~3u, room);
                room -= have[q];
            }
        }
        if (mine && lane == 0) {   // the copy engine brings the payloads, one behind the other, each rounded up to 16 bytes
            mbar_expect_tx(&s_bar[warp], 4u * (have[0] + have[1] + have[2] + have[3]));
            uint32_t at = 0;
#pragma unroll
            for (int q = 0; q < kRoundsPerTile; ++q) {
                if (have[q]) bulk_load(stage + at, slot + (size_t)q * kRoundSlotWords + 8, 4u * have[q], &s_bar[warp]);
                at += have[q];
            }
        }
        {
            const unsigned long long left = n - (unsigned long long)(t0 + (mine ? tl : 0u)) * kTile;
            const uint32_t len = (uint32_t)(left < (unsigned long long)kTile ? left : (unsigned long long)kTile);
            const uint32_t padw = (((len + kBlock - 1) / kBlock) + 3) >> 2;
#pragma unroll
            for (int d = 16; d >= 1; d >>= 1) part += __shfl_xor_sync(kFull, part, d);
            if (lane == 0) {
                s_words[warp] = mine ? 1u + padw + nq4.x + nq4.y + nq4.z + nq4.w : 0u;
                s_part[warp] = (uint32_t)part;
            }
        }
        __syncthreads();
        if (warp == kPlaceThreads / 32 - 1) rearm();   // every warp's reads of the sums are through
        // the group's place: the groups of the job in front of it are full ones (33 fixed words per tile) with the
        // payload that step 1 added up per group; the tile's place inside the group: the tiles in front of it
        const uint32_t wl = s_words[lane];
        const uint32_t incl = warp_incl_scan(wl, lane);
        const uint32_t my_off = __shfl_sync(kFull, incl - wl, warp);
        const uint32_t base = __reduce_add_sync(kFull, s_part[lane]) + t0 * (1u + (uint32_t)kLWords);
        if (mine) {
            const uint32_t tile = t0 + tl;
            const uint32_t words = s_words[tl];
            const unsigned long long word0 = (unsigned long long)kHeaderWords + nT + base + my_off;
            const bool fits = (word0 + words) * 4ull <= job.out_cap;
            if (!fits) status |= kStCapacity;
            // the copies into this warp's shared memory land before anything else happens (also when the tile does not fit:
            // a CTA must not end with copies into its shared memory still on their way)
            if (!mbar_wait(&s_bar[warp], 0u)) status |= kStTimeout;
            if (fits) {
                uint32_t* __restrict__ dst = out + word0;
                const unsigned long long tleft = n - (unsigned long long)tile * kTile;
                const uint32_t tlen = (uint32_t)(tleft < (unsigned long long)kTile ? tleft : (unsigned long long)kTile);
                const uint32_t tpadw = (((tlen + kBlock - 1) / kBlock) + 3) >> 2;
                if (lane == 0) dst[0] = first;
                if ((uint32_t)lane < tpadw) dst[1 + lane] = lword;
                uint32_t* __restrict__ d = dst + 1 + tpadw;
                const uint32_t* from = stage;
#pragma unroll
                for (int q = 0; q < kRoundsPerTile; ++q) {
                    const uint32_t nq = nqs[q], in_stage = min(nq, have[q]);
#pragma unroll
                    for (int k = 0; k < kPlaceUnroll; ++k) {
                        const uint32_t i = (uint32_t)lane + 32u * k;
                        if (i < in_stage) d[i] = from[i];
                    }
                    const uint32_t* __restrict__ src = slot + (size_t)q * kRoundSlotWords + 8;
                    for (uint32_t i = 32u * kPlaceUnroll + (uint32_t)lane; i < in_stage; i += 32) d[i] = from[i];
                    for (uint32_t i = in_stage + (uint32_t)lane; i < nq; i += 32) d[i] = src[i];
                    from += have[q];
                    d += nq;
                }
                if (lane == 0) out[kHeaderWords + tile] = base + my_off + words;
            }
            if (lane == 0 && tile == nT - 1) *job.out_bytes = (size_t)((word0 + words) * 4ull);
            if (tile == 0) put_header(out, lane, n, nT);
        }
    }
    if (status) atomicOr(ws.status, status);
}

// ------------------------------------------------------------------------------------------------ decompress
//
// A warp decodes a tile of its own in four rounds, lane l of a round taking block 32 * round + l: the block's sign
// word and planes come out of the tile's blob (staged in shared memory by a bulk copy, one tile ahead), the block's
// sum of deltas follows from population counts of the planes, a shuffle scan of those sums gives every block the
// code in front of it, and the lane then walks its 32 elements: inverse bit-matrix transpose, magnitude, sign,
// running code, one multiplication; the values go into the lane's row of a swizzled stage, which one tiled tensor
// store (or, for ragged ends and unaligned arrays, a loop of coalesced stores) moves to the output.

// What a tile's code-length bytes say, found by every lane alike: 0 = inconsistent with the blob's size (or a code
// length above 31, or a non-zero padding byte), 1 = consistent and every code of the tile stays below 2^23 in
// magnitude (fp32 arithmetic is exact), 2 = consistent, integer arithmetic needed.  blob: the tile's words.
__device__ __forceinline__ int describe_blob(const uint32_t* blob, uint32_t words, uint32_t nb, int lane)
{
    const uint32_t padw = (nb + 3) >> 2;
    if (words < 1u + padw) return 0;
    const uint32_t lw = (uint32_t)lane < padw ? blob[1 + lane] : 0u;
    const uint32_t L0 = lw & 0xFFu, L1 = (lw >> 8) & 0xFFu, L2 = (lw >> 16) & 0xFFu, L3 = lw >> 24;
    bool bad = (lw & 0xE0E0E0E0u) != 0u;   // a code length above 31
    const uint32_t b0 = 4u * (uint32_t)lane;   // blocks at or beyond nb are padding of the code-length area: must be zero
    if ((b0 + 0 >= nb && L0) || (b0 + 1 >= nb && L1) || (b0 + 2 >= nb && L2) || (b0 + 3 >= nb && L3)) bad = true;
    const uint32_t sizes = (L0 ? L0 + 1 : 0) + (L1 ? L1 + 1 : 0) + (L2 ? L2 + 1 : 0) + (L3 ? L3 + 1 : 0);
    const uint32_t total = __reduce_add_sync(kFull, sizes);
    // every partial sum of deltas is below sum_b 32 * 2^L_b; with the outlier it must stay below 2^24
    const uint32_t Lmax = max(max(L0, L1), max(L2, L3));
    uint32_t spread = 1u << 24;
    if (Lmax <= 18u) spread = (32u << L0) + (32u << L1) + (32u << L2) + (32u << L3);
    spread = __reduce_add_sync(kFull, min(spread, 1u << 24));   // at most 32 * 2^24 = 2^29: no overflow
    if (__any_sync(kFull, bad) || 1u + padw + total != words) return 0;
    const int32_t outlier = (int32_t)blob[0];
    const uint32_t ao = (uint32_t)(outlier < 0 ? -outlier : outlier);
    return (ao < (1u << 23) && spread < (1u << 23)) ? 1 : 2;
}

// A block's sign word and planes (payload words pay[0 .. L]) as N-bit packed words ready for the inverse transpose,
// N = 8, 16 or 32 (code lengths up to N), and the block's sum of deltas.
template <int N>
__device__ __forceinline__ int32_t load_planes(const uint32_t* pay, uint32_t L, uint32_t& sign, uint32_t (&w)[N])
{
    sign = L ? pay[0] : 0u;
    int32_t total = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        w[k] = (uint32_t)k < L ? pay[1 + k] : 0u;
        // elements with the bit set count 2^k each, negative ones with the opposite sign
        total += (__popc(w[k]) - 2 * __popc(w[k] & sign)) << k;
    }
    return total;
}

// The lane's 32 elements from the transposed words (word i, field h = magnitude of element N h + i), written as
// values into the lane's row of a stage.  Codes are exact in fp32 (the caller checked): the magnitude is read as a
// float from its bits, gets its sign, joins the running code, and one multiplication makes the value.  MODE 0:
// plain decoding; MODE 1: every value is added to the operand in the same place of the row `loc`.
template <int N, int MODE>
__device__ __forceinline__ void expand_block(const uint32_t (&w)[N], uint32_t sign, int32_t code_in_front, float s, char* row, uint32_t sw,
                                             const char* loc)
{
    float run = (float)code_in_front;
    uint32_t sel = N == 8 ? 0x7650u : 0x7610u;   // byte (pair) h of a word under the exponent of 2^23
#pragma unroll 1
    for (int h = 0; h < 32 / N; ++h) {
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            float o[4];
            const uint32_t at = (16u * (uint32_t)(h * (N / 4) + q)) ^ sw;
            if (MODE == 1) {
                // the hop: the magnitudes and the products go two elements to an instruction (sm_100's packed fp32, each half
                // rounded as the scalar operation is); the running code stays a chain of scalar additions, and the sums with the
                // operand stay scalar too: the compiler contracts a packed product and a packed addition behind it into a
                // packed fused multiply-add whatever --fmad says, and Eq. 2 adds to the ROUNDED decompressed value.
                // 43.1 -> 42.4 us per 64 MiB.  The plain decoder gains nothing from packing and keeps the scalar form.
                const float2 neg23 = make_float2(-kTwo23, -kTwo23), s2 = make_float2(s, s);
                const float2 m01 = __fadd2_rn(make_float2(__uint_as_float(prmt(w[4 * q + 0], 0x4B000000u, sel)),
                                                          __uint_as_float(prmt(w[4 * q + 1], 0x4B000000u, sel))), neg23);
                const float2 m23 = __fadd2_rn(make_float2(__uint_as_float(prmt(w[4 * q + 2], 0x4B000000u, sel)),
                                                          __uint_as_float(prmt(w[4 * q + 3], 0x4B000000u, sel))), neg23);
                const float ms[4] = {m01.x, m01.y, m23.x, m23.y};
                float rs[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int i = 4 * q + e;
                    const uint32_t sbit = (sign << (31 - i)) & 0x80000000u;
                    run = __fadd_rn(run, __uint_as_float(__float_as_uint(ms[e]) | sbit));
                    rs[e] = run;
                }
                const float4 l = *reinterpret_cast<const float4*>(loc + at);
                const float2 p01 = __fmul2_rn(make_float2(rs[0], rs[1]), s2), p23 = __fmul2_rn(make_float2(rs[2], rs[3]), s2);
                o[0] = __fadd_rn(p01.x, l.x); o[1] = __fadd_rn(p01.y, l.y); o[2] = __fadd_rn(p23.x, l.z); o[3] = __fadd_rn(p23.y, l.w);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int i = 4 * q + e;
                    const float m = __fsub_rn(__uint_as_float(prmt(w[i], 0x4B000000u, sel)), kTwo23);
                    const uint32_t sbit = (sign << (31 - i)) & 0x80000000u;
                    run = __fadd_rn(run, __uint_as_float(__float_as_uint(m) | sbit));
                    o[e] = __fmul_rn(run, s);
                }
            }
            *reinterpret_cast<float4*>(row + at) = make_float4(o[0], o[1], o[2], o[3]);
        }
        sign >>= N;
        sel += N == 8 ? 0x0001u : 0x0022u;
    }
}

// Reduce operation of the hop: 0 = sum, 1 = max, 2 = min, 3 = average (a sum on every hop); of two operands that
// compare equal Max and Min keep the decoded one.
__device__ __forceinline__ float combine(uint32_t op, float a, float b)
{
    return op == 1u ? ((a < b) ? b : a) : op == 2u ? ((b < a) ? b : a) : __fadd_rn(a, b);
}

// Where a tile's blob is, as known from the index alone.
struct BlobRef {
    const uint32_t* ptr;    // nullptr: no blob (tile beyond the stream, or a stream that does not parse)
    uint32_t words;
    bool staged;            // a bulk copy of its 16-byte-aligned cover is on its way
};

// One round of a tile (blocks 32 rd + lane) by the general route: any code length, integer arithmetic, any reduce
// operation.  blob: the tile's words (shared or global memory); pay_off: payload words of the rounds before; code:
// the code in front of the round; loc_stage: the stage with the operand's round, or nullptr.  Leaves the values in
// `stage`.  Compact rather than fast: the rounds that come here are rare.
__device__ __noinline__ void decode_round_general(const uint32_t* blob, uint32_t padw, uint32_t L, uint32_t* pay_off_io, int32_t* code_io,
                                                  float s, float* stage, int lane, const float* loc_stage, uint32_t op)
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
    char* row = reinterpret_cast<char*>(stage) + 128 * lane;
    const char* loc = reinterpret_cast<const char*>(loc_stage) + 128 * lane;
    const uint32_t sw = ((uint32_t)lane & 7u) << 4;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        run += ((sign >> j) & 1u) ? -(int32_t)w[j] : (int32_t)w[j];
        float v = __fmul_rn(__int2float_rn(run), s);
        const uint32_t at = ((16u * (uint32_t)(j >> 2)) ^ sw) + 4u * (j & 3);
        if (loc_stage) v = combine(op, v, *reinterpret_cast<const float*>(loc + at));
        *reinterpret_cast<float*>(row + at) = v;
    }
}

constexpr int kDecBlobWords = 1024 + 8;   // blob buffers: a window of 4 KiB plus the slack of the 16-byte-aligned cover

// The code lengths of a lane's four blocks of a tile (blocks lane, 32 + lane, 64 + lane, 96 + lane), one per byte, from
// the head of the tile's blob: kept in a register, because the window over a large blob moves away from its head.
__device__ __forceinline__ uint32_t lane_code_lengths(const uint32_t* blob, uint32_t nb, int lane)
{
    const unsigned char* lb = reinterpret_cast<const unsigned char*>(blob + 1);
    uint32_t lp = 0;
#pragma unroll
    for (uint32_t e = 0; e < (uint32_t)kRoundsPerTile; ++e) {
        const uint32_t bi = 32u * e + (uint32_t)lane;
        if (bi < nb) lp |= (uint32_t)lb[bi] << (8u * e);
    }
    return lp;
}

// The window a warp has over its current tile's blob: words [0, end) of the blob can be read at base[word].  A blob
// that a bulk copy can bring (BlobRef::staged) is staged a window at a time: first its front, and when a round reaches
// past the window's end, the window moves to that round's first word.  Other blobs are read where they are.
struct BlobWindow {
    const uint32_t* base;
    uint32_t end;
};
// How much of a blob the copy that brings words [first, ...) covers: bytes to copy from the 16-byte boundary at or
// below that word (at most a buffer's worth, at most to the 16-byte boundary at or above the blob's end).
__device__ __forceinline__ uint32_t window_bytes(const BlobRef& br, uint32_t first)
{
    const uintptr_t g = (uintptr_t)(br.ptr + first), e = (uintptr_t)(br.ptr + br.words);
    const uintptr_t a_beg = g & ~(uintptr_t)15, a_end = (e + 15) & ~(uintptr_t)15;
    const uintptr_t bytes = a_end - a_beg;
    return (uint32_t)(bytes < (uintptr_t)(kDecBlobWords * 4) ? bytes : (uintptr_t)(kDecBlobWords * 4));
}
// The window after that copy has landed in `buf`.
__device__ __forceinline__ BlobWindow window_at(const BlobRef& br, uint32_t first, const uint32_t* buf)
{
    const uint32_t lead = (uint32_t)(((uintptr_t)(br.ptr + first)) & 15u) >> 2;   // words between the boundary and the first word
    BlobWindow w;
    w.base = buf + lead - first;
    const uint32_t got = first + (window_bytes(br, first) >> 2) - lead;
    w.end = got < br.words ? got : br.words;
    return w;
}
// Issues the copy (one lane).
__device__ __forceinline__ void window_request(const BlobRef& br, uint32_t first, uint32_t* buf, unsigned long long* bar)
{
    const uint32_t bytes = window_bytes(br, first);
    mbar_expect_tx(bar, bytes);
    bulk_load(buf, (const void*)(((uintptr_t)(br.ptr + first)) & ~(uintptr_t)15), bytes, bar);
}

// Tiled tensor store of a stage to rows [row0, row0 + 32) of the array behind `map` (one thread).
__device__ __forceinline__ void tensor_store_round(const CUtensorMap* map, uint32_t row0, const float* stage)
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(map), "r"(0), "r"((int)row0), "r"(smem_u32(stage)) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// The same for ragged ends and unaligned arrays: `count` elements of the stage, coalesced.
__device__ __noinline__ void store_round_ragged(float* __restrict__ y, const float* stage, uint32_t count, int lane)
{
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
        const uint32_t e = 32u * k + (uint32_t)lane;
        if (e < count) y[e] = *reinterpret_cast<const float*>(reinterpret_cast<const char*>(stage) + stage_chunk_byte(k, (uint32_t)lane >> 2) + 4 * (lane & 3));
    }
}

// A round's share of a copy that goes along with a compression, where there is no valid bound and nothing is encoded.  Rare.
__device__ __noinline__ void copy_round_plain(float* y, const float* x, unsigned long long left, int lane)
{
    const uint32_t count = left < (unsigned long long)kRound ? (uint32_t)left : (uint32_t)kRound;
#pragma unroll 4
    for (uint32_t e = (uint32_t)lane; e < count; e += 32u) y[e] = x[e];
}

// One round of a tile whose codes are exact in fp32: blocks 32 rd + lane.  Arguments as for decode_round_general;
// MODE as for expand_block.  The lanes of a warp mostly share one width class; a round with a code length above 16
// takes the general route.
template <int N, int MODE>
__device__ __forceinline__ void decode_round_n(const uint32_t* blob, uint32_t padw, uint32_t L, uint32_t& pay_off, int32_t& code, float s,
                                               float* stage, int lane, const float* loc_stage)
{
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    const uint32_t* pay = blob + 1 + padw + pay_off + (incl - nw);
    pay_off += __shfl_sync(kFull, incl, 31);
    char* row = reinterpret_cast<char*>(stage) + 128 * lane;
    const char* loc = reinterpret_cast<const char*>(loc_stage) + 128 * lane;
    const uint32_t sw = ((uint32_t)lane & 7u) << 4;
    // The block's sum of deltas first, so that the scan over the lanes gives the code in front of every block before
    // any element is expanded.
    uint32_t sign;
    uint32_t w[N];
    const int32_t total = load_planes<N>(pay, L, sign, w);
    int32_t inc = total;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t v = __shfl_up_sync(kFull, inc, d);
        if (lane >= d) inc += v;
    }
    bit_transpose<N>(w);
    expand_block<N, MODE>(w, sign, code + inc - total, s, row, sw, loc);
    code += __shfl_sync(kFull, inc, 31);
}
// The width class of round rd of a tile, the same for all lanes: 8, 16, or 0 when a code length above 16 sends the
// round down the general route.
__device__ __forceinline__ int round_class(uint32_t L)
{
    if (__any_sync(kFull, L > 16u)) return 0;
    return __any_sync(kFull, L > 8u) ? 16 : 8;
}
// The decoder's own form: one function with both classes (measured faster there than the two instantiations above
// behind a dispatch, which the hop uses out of line to keep its register count down).
// `ready` is called once by all lanes, after the planes are read and transposed and before the first value is stored:
// the place to make sure the stage is free.
template <int MODE, class Ready>
__device__ __forceinline__ void decode_round(const uint32_t* blob, uint32_t padw, uint32_t L, uint32_t& pay_off, int32_t& code, float s,
                                             float* stage, int lane, const float* loc_stage, Ready&& ready)
{
    if (__any_sync(kFull, L > 16u)) {
        ready();
        decode_round_general(blob, padw, L, &pay_off, &code, s, stage, lane, loc_stage, 0u);
        return;
    }
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    const uint32_t* pay = blob + 1 + padw + pay_off + (incl - nw);
    pay_off += __shfl_sync(kFull, incl, 31);
    char* row = reinterpret_cast<char*>(stage) + 128 * lane;
    const char* loc = reinterpret_cast<const char*>(loc_stage) + 128 * lane;
    const uint32_t sw = ((uint32_t)lane & 7u) << 4;
    uint32_t sign;
    int32_t total;
    if (!__any_sync(kFull, L > 8u)) {
        uint32_t w[8];
        total = load_planes<8>(pay, L, sign, w);
        int32_t inc = total;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t v = __shfl_up_sync(kFull, inc, d);
            if (lane >= d) inc += v;
        }
        bit_transpose<8>(w);
        ready();
        expand_block<8, MODE>(w, sign, code + inc - total, s, row, sw, loc);
        code += __shfl_sync(kFull, inc, 31);
    } else {
        uint32_t w[16];
        total = load_planes<16>(pay, L, sign, w);
        int32_t inc = total;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t v = __shfl_up_sync(kFull, inc, d);
            if (lane >= d) inc += v;
        }
        bit_transpose<16>(w);
        ready();
        expand_block<16, MODE>(w, sign, code + inc - total, s, row, sw, loc);
        code += __shfl_sync(kFull, inc, 31);
    }
}
template <int MODE>
__device__ __forceinline__ void decode_round(const uint32_t* blob, uint32_t padw, uint32_t L, uint32_t& pay_off, int32_t& code, float s,
                                             float* stage, int lane, const float* loc_stage = nullptr)
{
    decode_round<MODE>(blob, padw, L, pay_off, code, s, stage, lane, loc_stage, [] {});
}

struct alignas(1024) DecWarpShared {
    float out[kRound];                     // one output stage
    alignas(16) uint32_t blob[2][kDecBlobWords];   // this tile's blob (or a window over it) and the next tile's
    alignas(8) unsigned long long bar[2];
};
static_assert(sizeof(DecWarpShared) == 13 * 1024, "a warp's share of the shared memory");
// ------------------------------------------------------------------------------------------------ fused hop
//
// The form with two compressed operands (hops with an uncompressed one are in zccl_hop.cuh): out = compress(
// decompress(in_c) (+) decompress(in_c2)), tile by tile, with no uncompressed intermediate in global memory.  A warp
// decodes a round of the second stream onto a stage, the incoming tile's round onto that, and encodes the stage like
// a round of the compressor: into a buffer, off to the round's slot by a bulk store.  The place kernel finishes the
// stream.  An uncompressed copy of the result, when asked for, leaves the stage by a tensor store.

// Out-of-line copies for the hop, whose kernel holds a decoder and an encoder: inlined, the compiler multiplied their
// code along the kernel's branches until instruction fetch bounded it (four times the size, 15 % slower).
template <int N, int MODE>
__device__ __noinline__ void decode_round_call(const uint32_t* blob, uint32_t padw, uint32_t L, uint32_t* pay_off, int32_t* code, float s,
                                               float* stage, int lane, const float* loc_stage)
{
    decode_round_n<N, MODE>(blob, padw, L, *pay_off, *code, s, stage, lane, loc_stage);
}
// the round by its width class (MODE as for expand_block); op: the reduce operation, for the general route
template <int MODE>
__device__ __forceinline__ void decode_round_classes(const uint32_t* blob, uint32_t padw, uint32_t L, uint32_t* pay_off, int32_t* code,
                                                     float s, float* stage, int lane, const float* loc_stage, uint32_t op)
{
    const int cls = round_class(L);
    if (cls == 8) decode_round_call<8, MODE>(blob, padw, L, pay_off, code, s, stage, lane, loc_stage);
    else if (cls == 16) decode_round_call<16, MODE>(blob, padw, L, pay_off, code, s, stage, lane, loc_stage);
    else decode_round_general(blob, padw, L, pay_off, code, s, stage, lane, loc_stage, op);
}
template <int N>
__device__ __noinline__ int encode_round_call(const char* row, uint32_t sw, float xprev, float r, bool active, uint32_t* buf, EncodeCarry* cy, int lane,
                                              uint32_t* status)
{
    // laid out like a tile's blob whose word 0 sits in front of the buffer: code-length bytes at words 1.., payload at word 9
    return encode_round_n<N>(row, sw, xprev, r, active, (uint32_t)lane, 32u, buf - 1, 0u, 1, 9u, (uint32_t)kRoundBufWords - 8u, *cy, lane, *status, [] {});
}

// Advances (pay_off, code) over round e of a tile without expanding it: the blocks' sizes from their code lengths,
// their sums of deltas from population counts of their planes.  Lets a warp start in the middle of a tile.
__device__ __noinline__ void skip_round(const uint32_t* blob, uint32_t padw, uint32_t L, uint32_t* pay_off, int32_t* code, int lane)
{
    const uint32_t nw = L ? L + 1u : 0u;
    const uint32_t incl = warp_incl_scan(nw, lane);
    const uint32_t* pay = blob + 1 + padw + *pay_off + (incl - nw);
    const uint32_t sign = L ? pay[0] : 0u;
    int32_t total = 0;
    for (uint32_t k = 0; k < L; ++k) {
        const uint32_t w = pay[1 + k];
        total += (__popc(w) - 2 * __popc(w & sign)) << k;
    }
    *pay_off += __shfl_sync(kFull, incl, 31);
    *code += (int32_t)__reduce_add_sync(kFull, total);
}

__device__ __forceinline__ uint32_t cj_begin_of(const JobBatch& jb, int j) { return jb.job[j].tile_begin; }

struct alignas(1024) HopWarpShared {
    float loc[2][kRound];                  // the second operand's rounds, replaced in place by the combined values and then
                                           // by the encoded round; 1024-byte boundaries
    alignas(16) uint32_t blob[kDecBlobWords];
    alignas(8) unsigned long long bar_blob;
};
static_assert(sizeof(HopWarpShared) == 13 * 1024, "a warp's share of the shared memory");

// The owner's copy as the dequantised value float(q(y)) * s: `count` elements of the stage, coalesced.
__device__ __noinline__ void store_round_dequantised(float* __restrict__ y, const float* stage, uint32_t count, float r, float s, int lane)
{
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
        const uint32_t e = 32u * k + (uint32_t)lane;
        const float v = *reinterpret_cast<const float*>(reinterpret_cast<const char*>(stage) + stage_chunk_byte(k, (uint32_t)lane >> 2) + 4 * (lane & 3));
        if (e < count) y[e] = __fmul_rn(__int2float_rn(__float2int_rn(__fmul_rn(v, r))), s);
    }
}

template <bool Y, bool SPLIT>
__global__ void __launch_bounds__(kCodecThreads, 4) hop_tiles_c2_kernel(const __grid_constant__ JobBatch jb, const __grid_constant__ TileMaps maps,
                                                                     Workspace ws, uint32_t split_shift_arg)
{
    const uint32_t split_shift = SPLIT ? split_shift_arg : 0u;   // SPLIT false: whole tiles only, known when the kernel is compiled
    // split_shift 0: a warp's unit of work is a tile; 1: two rounds; 2: a round (small launches: more warps at work, and
    // none of them walks four rounds in a row)
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    HopWarpShared& sh = reinterpret_cast<HopWarpShared*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u))[warp];
    uint32_t status = 0;
    if (lane == 0) {
        mbar_init(&sh.bar_blob, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    uint32_t bfill = 0;   // completed copies into the blob buffer (phase parity)

    // the job of the tile looked up last, with its streams' headers
    int cj = -1;
    uint32_t cj_begin = 0, cj_count = 0;
    StreamInfo h1, h2;
    h1.ok = h2.ok = false; h1.n = h2.n = 0; h1.nT = h2.nT = 0; h1.s = h2.s = 1.0f; h1.eb_abs = h2.eb_abs = 0.0f;
    bool job_ok = false;
    auto enter_job = [&](uint32_t t) {
        if (t - cj_begin >= cj_count) {
            cj = find_job(jb, t);
            const Job& q = jb.job[cj];
            cj_begin = q.tile_begin;
            cj_count = (cj + 1 < jb.count ? jb.job[cj + 1].tile_begin : jb.total_tiles) - cj_begin;
            h1 = read_header(q.in_c, q.in_cap);
            h2 = read_header(q.in_c2, q.in2_cap);
            job_ok = h1.ok && h1.n == q.n && h2.ok && h2.n == q.n && __float_as_uint(h2.s) == __float_as_uint(h1.s);
        }
    };
    // a tile's blob out of one of the job's streams, from the index alone (ptr = nullptr, words = ~0: damaged index)
    auto blob_of = [&](const uint32_t* in, unsigned long long cap, uint32_t nT, uint32_t tile) {
        BlobRef br;
        br.ptr = nullptr; br.words = 0xFFFFFFFFu; br.staged = false;
        const uint32_t* idx = in + kHeaderWords;
        const uint32_t w_end = ldg_u32(idx + tile), w_beg = tile ? ldg_u32(idx + tile - 1) : 0u;
        const unsigned long long blob0 = (unsigned long long)kHeaderWords + nT;
        if (w_end <= w_beg || (blob0 + w_end) * 4ull > cap) return br;
        br.ptr = in + blob0 + w_beg;
        br.words = w_end - w_beg;
        return br;
    };
    // the incoming blob of tile t of the launch; its cover is requested into the blob buffer when it fits
    auto request_blob = [&](uint32_t t) {
        BlobRef br;
        br.ptr = nullptr; br.words = 0; br.staged = false;
        if (t >= jb.total_tiles) return br;
        enter_job(t);
        const Job& q = jb.job[cj];
        const uint32_t tile = t - cj_begin;
        if (!job_ok || q.n == 0 || tile >= h1.nT) return br;
        br = blob_of(q.in_c, q.in_cap, h1.nT, tile);
        if (!br.ptr) return br;
        const uintptr_t a_end = ((uintptr_t)(br.ptr + br.words) + 15) & ~(uintptr_t)15;
        if (a_end - (uintptr_t)q.in_c <= (uintptr_t)q.in_cap) {   // the copies may read up to the boundary behind the blob
            if (lane == 0) window_request(br, 0, sh.blob, &sh.bar_blob);
            br.staged = true;
        }
        return br;
    };

    const uint32_t stride = gridDim.x * (uint32_t)kCodecWarps;
    const uint32_t total_units = jb.total_tiles << split_shift, rd_mask = (1u << split_shift) - 1u;
    uint32_t un = blockIdx.x * (uint32_t)kCodecWarps + (uint32_t)warp;   // unit: tile un >> split_shift, from round un & rd_mask on
    uint32_t pl = 0;   // stage in turn
    BlobRef cur = request_blob(un < total_units ? un >> split_shift : 0xFFFFFFFFu);
    EncodeCarry cy;
    cy.pay_used = 0; cy.wide = false;

    while (un < total_units) {
        const uint32_t t = un >> split_shift, rd_first = (un & rd_mask) * (4u >> split_shift);
        // the current tile's facts, before the look-up of the next tile moves on to another job
        enter_job(t);
        const int jcur = cj;
        const Job& job = jb.job[jcur];
        const uint32_t tile = t - cj_begin;
        const StreamInfo hc1 = h1, hc2 = h2;
        const bool ok = job_ok;
        const unsigned long long n = job.n;
        const float s = hc1.s, r = __fdiv_rn(1.0f, hc1.s);
        const unsigned long long start = (unsigned long long)tile * kTile;
        const uint32_t len = (ok && n) ? (uint32_t)((n - start < (unsigned long long)kTile) ? (n - start) : kTile) : 0u;
        const uint32_t nb = (len + kBlock - 1) / kBlock, padw = (nb + 3) >> 2, rounds = (nb + 31) >> 5;
        const uint32_t op = (job.flags >> 1) & 3u;
        const bool summing = op == 0u || op == 3u, deq = (job.flags & 1u) != 0;
        if (!ok) status |= kStBadStream;

        const uint32_t unn = (un + stride < un || un + stride >= total_units) ? 0xFFFFFFFFu : un + stride;
        const uint32_t tn = unn == 0xFFFFFFFFu ? 0xFFFFFFFFu : unn >> split_shift;
        const uint32_t rd_end = rd_first + (4u >> split_shift);
        const uint32_t rd_stop = rd_first >= rounds ? rd_first : (rd_end < rounds ? rd_end : rounds);   // rounds [rd_first, rd_stop)
        if (cur.staged) {
            if (!mbar_wait(&sh.bar_blob, bfill & 1u)) status |= kStTimeout;
            ++bfill;
        }

        // what the two blobs say
        const uint32_t* blob1 = nullptr;
        const uint32_t* blob2 = nullptr;
        BlobWindow win;   // over the incoming blob
        win.base = nullptr; win.end = 0;
        int mode1 = 0, mode2 = 0;
        if (len) {
            if (cur.ptr) {
                win.base = cur.ptr; win.end = cur.words;
                if (cur.staged) win = window_at(cur, 0, sh.blob);
                blob1 = win.base;
                mode1 = describe_blob(blob1, cur.words, nb, lane);   // the head (at most 33 words) is in every first window
            }
            const BlobRef b2 = blob_of(job.in_c2, job.in2_cap, hc2.nT, tile);
            blob2 = b2.ptr;
            mode2 = b2.ptr ? describe_blob(b2.ptr, b2.words, nb, lane) : 0;
            if (mode1 == 0 || mode2 == 0) status |= kStBadStream;
        }
        const bool good = len != 0 && mode1 != 0 && mode2 != 0;

        uint32_t pay1 = 0, pay2 = 0;
        int32_t code1 = good ? (int32_t)blob1[0] : 0, code2 = good ? (int32_t)blob2[0] : 0;
        const uint32_t lp1 = good ? lane_code_lengths(blob1, nb, lane) : 0u, lp2 = good ? lane_code_lengths(blob2, nb, lane) : 0u;
        // moves the window over the incoming blob to round e's first word when the round reaches past its end
        auto reach = [&](uint32_t e) {
            const uint32_t L = (lp1 >> (8u * e)) & 0xFFu;
            const uint32_t first = 1u + padw + pay1;
            if (win.end < cur.words && first + __reduce_add_sync(kFull, L ? L + 1u : 0u) > win.end) {
                __syncwarp();   // every lane is done with the window as it is
                if (lane == 0) window_request(cur, first, sh.blob, &sh.bar_blob);
                if (!mbar_wait(&sh.bar_blob, bfill & 1u)) status |= kStTimeout;
                ++bfill;
                win = window_at(cur, first, sh.blob);
                blob1 = win.base;
            }
            return L;
        };
        float carry_y = 0.0f;
        // The next tile's blob goes into the one blob buffer as soon as this tile's last round is decoded (that look-up moves
        // the job on).
        BlobRef nxt;
        nxt.ptr = nullptr; nxt.words = 0; nxt.staged = false;
        auto look_ahead = [&]() {
            __syncwarp();   // every lane is done with the blob buffer
            nxt = request_blob(tn);
        };
        if (rd_first >= rd_stop || !good) look_ahead();
        if (good && rd_first != 0 && rd_first < rd_stop) {
            // a unit that starts inside its tile: sizes and codes of the rounds in front, and the value in front of it
            for (uint32_t e = 0; e < rd_first; ++e) {
                const uint32_t Le = reach(e);
                skip_round(blob1, padw, Le, &pay1, &code1, lane);
                skip_round(blob2, padw, (lp2 >> (8u * e)) & 0xFFu, &pay2, &code2, lane);
            }
            const float xa = __fmul_rn(__int2float_rn(code1), s);
            const float xb = __fmul_rn(__int2float_rn(code2), s);
            carry_y = combine(op, xa, xb);
        }
        for (uint32_t rd = rd_first; rd < rd_stop; ++rd) {
            float* loc = sh.loc[pl];
            const uint32_t u = 4u * t + rd;
            // The other stage holds the round before, encoded in place and handed to the copy engine, which by the end of this
            // round's decoding is mostly through with it: the next round goes there.
            auto release_other = [&]() {
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
            };
            if (!good) {
                release_other();
                if (lane == 0) ws.round_words[u] = 0;
            } else {
                {   // the second operand's round goes onto the stage, the incoming one's onto it
                    const uint32_t L2 = (lp2 >> (8u * rd)) & 0xFFu;
                    if (mode2 == 1) decode_round_classes<0>(blob2, padw, L2, &pay2, &code2, s, loc, lane, nullptr, 0u);
                    else decode_round_general(blob2, padw, L2, &pay2, &code2, s, loc, lane, nullptr, 0u);
                    __syncwarp();
                }
                const uint32_t L1 = reach(rd);
                if (mode1 == 1 && summing) decode_round_classes<1>(blob1, padw, L1, &pay1, &code1, s, loc, lane, loc, op);
                else decode_round_general(blob1, padw, L1, &pay1, &code1, s, loc, lane, loc, op);
                release_other();
                if (rd + 1 == rd_stop) look_ahead();   // the blob is decoded: the next unit's may come
                __syncwarp();   // the stage's rows, written by all lanes, are visible
                const float* ys = loc;
                const char* row = reinterpret_cast<const char*>(ys) + 128 * lane;
                const uint32_t sw = ((uint32_t)lane & 7u) << 4;
                const float y0 = ys[0];
                const float xprev = lane ? read_last_of_row(ys, (uint32_t)lane - 1u) : (rd ? carry_y : y0);   // carry_y: the value in front of the round
                carry_y = read_last_of_row(ys, 31);
                const uint32_t e0 = rd * (uint32_t)kRound;
                uint32_t* slot = ws.slots + (size_t)u * kRoundSlotWords;
                if (Y && job.y) {   // an uncompressed copy of the result leaves the stage before the encoder writes over it
                    const uint32_t count = len - e0 < (uint32_t)kRound ? len - e0 : (uint32_t)kRound;
                    if (deq) store_round_dequantised(job.y + start + e0, ys, count, r, s, lane);
                    else if (jb.count <= kMaxJobs / 2 && (((uintptr_t)job.y) & 15u) == 0 && count == (uint32_t)kRound) {
                        if (lane == 0) {
                            tensor_store_round(&maps.m[kMaxJobs / 2 + jcur], tile * (uint32_t)kBlocksPerTile + (e0 >> 5), ys);
                            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        }
                    } else store_round_ragged(job.y + start + e0, ys, count, lane);
                    __syncwarp();
                }
                uint32_t* buf = reinterpret_cast<uint32_t*>(loc);   // in place: a round's code never outgrows its 4 KiB
                cy.pay_used = 0;
                const uint32_t bi = 32u * rd + (uint32_t)lane;
                int rc = 3;
                if (!cy.wide) rc = encode_round_call<8>(row, sw, xprev, r, bi < nb, buf, &cy, lane, &status);
                if (rc == 3) rc = encode_round_call<16>(row, sw, xprev, r, bi < nb, buf, &cy, lane, &status);
                const uint32_t gslot = (cj_begin_of(jb, jcur) >> 5) + (uint32_t)jcur + (tile >> 5);
                if (rc == 0) {
                    __syncwarp();   // the buffer's words, written by all lanes, are visible to lane 0's store
                    if (lane == 0) {
                        const uint32_t bytes = (32u + 4u * cy.pay_used + 15u) & ~15u;
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(slot), "r"(smem_u32(buf)), "r"(bytes) : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        ws.round_words[u] = cy.pay_used;
                        atomicAdd(ws.group_acc + gslot, (unsigned long long)cy.pay_used);
                        // exact while |y r| < 2^22; larger codes take the general route
                        if (rd == 0) ws.outliers[t] = (int32_t)(__float_as_uint(__fadd_rn(__fmul_rn(y0, r), kRoundMagic)) - kRoundMagicBits);
                    }
                } else {
                    status |= encode_round_general_staged(ys, xprev, bi < nb, rd, r, slot, ws.round_words + u, ws.outliers + t, ws.group_acc + gslot, lane);
                }
            }
            pl ^= 1u;
        }
        // rounds the tile does not have
        if ((uint32_t)lane >= rd_first && (uint32_t)lane < rd_end && (uint32_t)lane >= rounds) ws.round_words[4u * t + (uint32_t)lane] = 0;
        cur = nxt;
        un = unn;
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (status) atomicOr(ws.status, status);
}

#include "zccl_tiles.cuh"
#include "zccl_decode.cuh"
#include "zccl_stream.cuh"
#include "zccl_hop.cuh"
#include "zccl_ring.cuh"
#include "zccl_codec_f64.cuh"
#include "zccl_codec_tiled.cuh"

// Per-device launch set-up (shared-memory attribute, resident CTAs per SM), done once per device under a lock.
constexpr int kMaxDevices = 64;
constexpr size_t kEncodeTilesSmemBytes = sizeof(EncodeShared) + 1024;
constexpr size_t kStreamSmemBytes = sizeof(StreamShared) + 1024;
constexpr size_t kRoundSmemBytes = sizeof(RoundWarpShared) * kCodecWarps + 1024;
constexpr size_t kDecSmemBytes = sizeof(DecWarpShared) * kCodecWarps + 1024;
constexpr size_t kHopSmemBytes = sizeof(HopWarpShared) * kCodecWarps + 1024;
constexpr size_t kRingSmemBytes = sizeof(RingShared) + 1024;
constexpr size_t kHopTilesSmemBytes = sizeof(HopShared) + 1024;
constexpr size_t kDecodeSmemBytes = sizeof(DecodeShared) + 1024;
constexpr size_t kDec64SmemBytes = sizeof(Decode64Shared) + 1024;
struct DeviceSetup {
    bool ready = false;
    int stream_ctas = 1, dec_ctas = 1, hop_ctas = 1, hop_tiles_ctas = 1, ring_ctas = 1, dec64_ctas = 1, round_tiled_ctas = 1, dec_tiled_ctas = 1;
};
DeviceSetup g_dev[kMaxDevices];
std::mutex g_dev_mu;
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                   const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode_tiled = nullptr;   // the driver's cuTensorMapEncodeTiled, looked up through the runtime

// The forms of the hop kernels.
template <int CAP, int OP, bool Y, bool ONCE>
cudaError_t hop_launch(dim3 grid, cudaStream_t st, const JobBatchT<CAP>& jb, const TileMapsT<CAP == 1 ? 2 : CAP>& maps, const Workspace& ws)
{
    return launch_k(hop_tiles_kernel<CAP, OP, Y, ONCE>, grid, dim3(kDecodeThreads), kHopTilesSmemBytes, st, jb, maps, ws);
}
template <int CAP, bool ONCE>
cudaError_t hop_launch_form(bool choosing, bool y, dim3 grid, cudaStream_t st, const JobBatchT<CAP>& jb, const TileMapsT<CAP == 1 ? 2 : CAP>& maps, const Workspace& ws)
{
    if (choosing) return y ? hop_launch<CAP, 1, true, ONCE>(grid, st, jb, maps, ws) : hop_launch<CAP, 1, false, ONCE>(grid, st, jb, maps, ws);
    return y ? hop_launch<CAP, 0, true, ONCE>(grid, st, jb, maps, ws) : hop_launch<CAP, 0, false, ONCE>(grid, st, jb, maps, ws);
}
template <int CAP, int OP, bool Y, bool ONCE>
cudaError_t hop_smem_attr() { return cudaFuncSetAttribute(hop_tiles_kernel<CAP, OP, Y, ONCE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHopTilesSmemBytes); }
template <int CAP, bool ONCE>
cudaError_t hop_smem_attrs()
{
    cudaError_t e = hop_smem_attr<CAP, 0, false, ONCE>();
    if (e == cudaSuccess) e = hop_smem_attr<CAP, 0, true, ONCE>();
    if (e == cudaSuccess) e = hop_smem_attr<CAP, 1, false, ONCE>();
    if (e == cudaSuccess) e = hop_smem_attr<CAP, 1, true, ONCE>();
    return e;
}
template <bool Y, bool SPLIT>
cudaError_t hop_c2_smem_attr() { return cudaFuncSetAttribute(hop_tiles_c2_kernel<Y, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHopSmemBytes); }

cudaError_t device_setup(const DeviceSetup** out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_dev_mu);
    if (!g_encode_tiled) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q);
        if (e != cudaSuccess) return e;
        if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        g_encode_tiled = reinterpret_cast<EncodeTiledFn>(fn);
    }
    DeviceSetup& d = g_dev[dev];
    if (!d.ready) {
        int a = 0;
        e = cudaFuncSetAttribute(encode_tiles_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEncodeTilesSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(encode_tiles_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEncodeTilesSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(encode_tiles_kernel<kMaxJobs, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEncodeTilesSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(encode_stream_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStreamSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(encode_stream_kernel<kMaxJobs>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStreamSmemBytes);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, encode_stream_kernel<kMaxJobs>, kStreamThreads, kStreamSmemBytes);
        if (e != cudaSuccess) return e;
        d.stream_ctas = a > 0 ? a : 1;
        e = cudaFuncSetAttribute(decode_tiles_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecodeSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_tiles_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecodeSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(decode_tiles_kernel<kMaxDecodeJobs, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecodeSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_tiles_kernel<kMaxDecodeJobs, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecodeSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, decode_tiles_kernel<kMaxDecodeJobs, true>, kDecodeThreads, kDecodeSmemBytes);
        if (e != cudaSuccess) return e;
        d.dec_ctas = a > 0 ? a : 1;
        e = cudaFuncSetAttribute(place_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPlaceSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(ring_tiles_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRingSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(ring_tiles_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRingSmemBytes);
        if (e == cudaSuccess) e = hop_smem_attrs<1, false>();
        if (e == cudaSuccess) e = hop_smem_attrs<1, true>();
        if (e == cudaSuccess) e = hop_smem_attrs<kMaxJobs, false>();
        if (e == cudaSuccess) e = hop_smem_attrs<kMaxJobs, true>();
        if (e == cudaSuccess) e = hop_c2_smem_attr<false, false>();
        if (e == cudaSuccess) e = hop_c2_smem_attr<false, true>();
        if (e == cudaSuccess) e = hop_c2_smem_attr<true, false>();
        if (e == cudaSuccess) e = hop_c2_smem_attr<true, true>();
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, hop_tiles_kernel<kMaxJobs, 1, true, true>, kDecodeThreads, kHopTilesSmemBytes);
        if (e != cudaSuccess) return e;
        d.hop_tiles_ctas = a > 0 ? a : 1;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, ring_tiles_kernel<1>, kDecodeThreads, kRingSmemBytes);
        if (e != cudaSuccess) return e;
        d.ring_ctas = a > 0 ? a : 1;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, hop_tiles_c2_kernel<true, true>, kCodecThreads, kHopSmemBytes);
        if (e != cudaSuccess) return e;
        d.hop_ctas = a > 0 ? a : 1;
        e = cudaFuncSetAttribute(decode_tiles_f64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDec64SmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, decode_tiles_f64_kernel, kDecodeThreads, kDec64SmemBytes);
        if (e != cudaSuccess) return e;
        d.dec64_ctas = a > 0 ? a : 1;
        e = cudaFuncSetAttribute(encode_rounds_tiled_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRoundSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, encode_rounds_tiled_kernel, kCodecThreads, kRoundSmemBytes);
        if (e != cudaSuccess) return e;
        d.round_tiled_ctas = a > 0 ? a : 1;
        e = cudaFuncSetAttribute(decode_tiles_tiled_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDecSmemBytes);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, decode_tiles_tiled_kernel, kCodecThreads, kDecSmemBytes);
        if (e != cudaSuccess) return e;
        d.dec_tiled_ctas = a > 0 ? a : 1;
        d.ready = true;
    }
    *out = &d;
    return cudaSuccess;
}

// The array x of n floats as rows of 32 floats, copied in tiles of 32 rows with the 128-byte swizzle.  Arrays that
// do not start on a 16-byte boundary or have no full row get no map (the kernels load them element by element).
cudaError_t make_row_map(CUtensorMap* map, const float* x, unsigned long long n, uint32_t rows = 32u)
{
    if ((((uintptr_t)x) & 15u) != 0 || n < (unsigned long long)kBlock) return cudaSuccess;
    const cuuint64_t dims[2] = {(cuuint64_t)kBlock, (cuuint64_t)(n / kBlock)};
    const cuuint64_t strides[1] = {(cuuint64_t)kBlock * sizeof(float)};
    const cuuint32_t box[2] = {(cuuint32_t)kBlock, (cuuint32_t)rows};
    const cuuint32_t estr[2] = {1u, 1u};
    const CUresult r = g_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(x), dims, strides, box, estr,
                                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// The array x of n doubles as rows of 16 doubles, copied in tiles of 64 rows with the 128-byte swizzle.
cudaError_t make_row_map_f64(CUtensorMap* map, const double* x, unsigned long long n)
{
    if ((((uintptr_t)x) & 15u) != 0 || n < 16ull) return cudaSuccess;
    const cuuint64_t dims[2] = {16u, (cuuint64_t)(n / 16ull)};
    const cuuint64_t strides[1] = {16u * sizeof(double)};
    const cuuint32_t box[2] = {16u, (cuuint32_t)kRowsPerRound64};
    const cuuint32_t estr[2] = {1u, 1u};
    const CUresult r = g_encode_tiled(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<double*>(x), dims, strides, box, estr,
                                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

// one CTA of the place kernel per group of 32 tiles of every job
uint32_t group_table(const JobBatch& jb, GroupTable& gt)
{
    uint32_t groups = 0;
    for (int j = 0; j < jb.count; ++j) {
        gt.begin[j] = groups;
        const uint32_t tiles = (j + 1 < jb.count ? jb.job[j + 1].tile_begin : jb.total_tiles) - jb.job[j].tile_begin;
        groups += (tiles + kPlaceTiles - 1u) / kPlaceTiles;
    }
    for (int j = jb.count; j <= kMaxJobs; ++j) gt.begin[j] = groups;
    return groups;
}

// Hops with an uncompressed operand.
template <int CAP>
static cudaError_t launch_hop_tiles(const JobBatchT<CAP>& jb, const Workspace& ws, int sm_count, bool& once, cudaStream_t st)
{
    constexpr int kMaps = CAP == 1 ? 2 : CAP, kResult = CAP == 1 ? 1 : CAP / 2;
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    thread_local TileMapsT<kMaps> maps;   // kept off the stack, one per calling thread
    bool y = false, choosing = false;
    for (int j = 0; j < jb.count; ++j) {
        const Job& q = jb.job[j];
        if ((e = make_row_map(&maps.m[j], q.x, q.n, (uint32_t)kBlocksPerTile)) != cudaSuccess) return e;
        if (q.y && jb.count <= kResult && (e = make_row_map(&maps.m[kResult + j], q.y, q.n)) != cudaSuccess) return e;
        y = y || q.y != nullptr;
        const uint32_t op = (q.flags >> 1) & 3u;
        choosing = choosing || op == 1u || op == 2u;
    }
    const unsigned cap = (unsigned)(sm_count * d->hop_tiles_ctas);
    // a launch whose tiles are all resident together finds its places itself; with more the CTAs go on to their next tiles
    // and the placement is a launch of its own
    once = jb.total_tiles <= cap;
    const dim3 grid(once ? jb.total_tiles : cap);
    return once ? hop_launch_form<CAP, true>(choosing, y, grid, st, jb, maps, ws) : hop_launch_form<CAP, false>(choosing, y, grid, st, jb, maps, ws);
}
// Hops with two compressed operands.
static cudaError_t launch_hop_c2(const JobBatch& jb, const Workspace& ws, int sm_count, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    thread_local TileMaps maps;   // 8 KiB: kept off the stack, one per calling thread
    bool y = false;
    for (int j = 0; j < jb.count; ++j) {
        if (!jb.job[j].in_c2) return cudaErrorInvalidValue;   // all of a launch's jobs are of this form
        if (jb.count <= kMaxJobs / 2 && jb.job[j].y && (e = make_row_map(&maps.m[kMaxJobs / 2 + j], jb.job[j].y, jb.job[j].n)) != cudaSuccess)
            return e;
        y = y || jb.job[j].y != nullptr;
    }
    const unsigned long long cap = (unsigned long long)sm_count * d->hop_ctas;
    // launches that would leave warps idle with a tile per warp hand out rounds instead
    const unsigned long long warps = cap * kCodecWarps;
    const uint32_t split_shift = 4ull * jb.total_tiles <= warps ? 2u : 2ull * jb.total_tiles <= warps ? 1u : 0u;
    const unsigned long long want = ((((unsigned long long)jb.total_tiles) << split_shift) + kCodecWarps - 1) / kCodecWarps;
    const dim3 grid((unsigned)(want < cap ? want : cap)), block(kCodecThreads);
    if (split_shift) return y ? launch_k(hop_tiles_c2_kernel<true, true>, grid, block, kHopSmemBytes, st, jb, maps, ws, split_shift)
                              : launch_k(hop_tiles_c2_kernel<false, true>, grid, block, kHopSmemBytes, st, jb, maps, ws, split_shift);
    return y ? launch_k(hop_tiles_c2_kernel<true, false>, grid, block, kHopSmemBytes, st, jb, maps, ws, split_shift)
             : launch_k(hop_tiles_c2_kernel<false, false>, grid, block, kHopSmemBytes, st, jb, maps, ws, split_shift);
}
cudaError_t launch_hop_lanes(const JobBatch& jb, const Workspace& ws, int sm_count, cudaStream_t st)
{
    if (!ws.slots) return cudaErrorInvalidValue;
    bool c2 = false;
    for (int j = 0; j < jb.count; ++j) c2 = c2 || jb.job[j].in_c2 != nullptr;
    cudaError_t e;
    bool once = false;
    if (c2) e = launch_hop_c2(jb, ws, sm_count, st);
    else if (jb.count > 1) e = launch_hop_tiles(jb, ws, sm_count, once, st);
    else {
        JobBatchT<1> one;
        one.job[0] = jb.job[0]; one.count = jb.count; one.total_tiles = jb.total_tiles;
        e = launch_hop_tiles(one, ws, sm_count, once, st);
    }
    if (e != cudaSuccess) return e;
    count_launches(once ? 1 : 2);
    if (once) return cudaSuccess;
    GroupTable gt;
    const uint32_t groups = group_table(jb, gt);
    return launch_k(place_kernel, dim3(groups), dim3(kPlaceThreads), kPlaceSmemBytes, st, jb, gt, ws, 0, ParamsF64{0.0, 1.0, 1.0, 1}, (int)kBoundHost);
}

template <int CAP>
static cudaError_t launch_decode_tiles(const JobBatchT<CAP>& jb, const Workspace& ws, int sm_count, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    thread_local TileMapsT<CAP> maps;   // kept off the stack, one per calling thread
    for (int j = 0; j < jb.count; ++j)
        if ((e = make_row_map(&maps.m[j], jb.job[j].y, jb.job[j].n)) != cudaSuccess) return e;
    const unsigned cap = (unsigned)(sm_count * d->dec_ctas);
    const dim3 grid(jb.total_tiles < cap ? jb.total_tiles : cap);
    return launch_k(jb.total_tiles >= kDealtTiles * grid.x ? decode_tiles_kernel<CAP, true> : decode_tiles_kernel<CAP, false>, grid, dim3(kDecodeThreads),
                    kDecodeSmemBytes, st, jb, maps, ws);
}
cudaError_t launch_decode_lanes(const DecodeBatch& jb, const Workspace& ws, int sm_count, cudaStream_t st)
{
    if (jb.count > 1 || jb.job[0].out) return launch_decode_tiles(jb, ws, sm_count, st);
    JobBatchT<1> one;
    one.job[0] = jb.job[0]; one.count = jb.count; one.total_tiles = jb.total_tiles;
    return launch_decode_tiles(one, ws, sm_count, st);
}

template <int CAP>
static cudaError_t launch_encode_tiles(const JobBatchT<CAP>& jb, const Workspace& ws, int bound_source, Params host_params, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    TileMapsT<CAP> maps;
    for (int j = 0; j < jb.count; ++j)
        if ((e = make_row_map(&maps.m[j], jb.job[j].x, jb.job[j].n)) != cudaSuccess) return e;
    return launch_k(encode_tiles_kernel<CAP, false>, dim3(jb.total_tiles), dim3(kTileThreads), kEncodeTilesSmemBytes, st, jb, maps, ws, host_params, bound_source);
}
template <int CAP>
static cudaError_t launch_encode_stream(const JobBatchT<CAP>& jb, const Workspace& ws, int bound_source, Params host_params, int sm_count, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    thread_local TileMapsT<CAP> maps;   // kept off the stack, one per calling thread
    for (int j = 0; j < jb.count; ++j)
        if ((e = make_row_map(&maps.m[j], jb.job[j].x, jb.job[j].n, (uint32_t)kBlocksPerTile)) != cudaSuccess) return e;
    const unsigned cap = (unsigned)(sm_count * d->stream_ctas);
    const dim3 grid(jb.total_tiles < cap ? jb.total_tiles : cap);
    return launch_any(bound_source == kBoundKeys ? kLaunchStream : kLaunchStreamEarly, 1, encode_stream_kernel<CAP>, grid, dim3(kStreamThreads), kStreamSmemBytes, st, jb, maps, ws, host_params, bound_source);
}
static unsigned ring_tiles(unsigned long long n, int N, unsigned* begin)
{
    const unsigned long long m = (n + N - 1) / N;
    unsigned t = 0;
    for (int c = 0; c < N; ++c) {
        const unsigned long long off = (unsigned long long)c * m, len = off < n ? (n - off < m ? n - off : m) : 0;
        if (begin) begin[c] = t;
        t += (unsigned)((len + kTile - 1) / kTile);
    }
    if (begin) begin[N] = t;
    return t;
}
// Every chunk has elements, and the tiles of all chunks are resident together.
bool ring_fits(unsigned long long n, int N, const Workspace& ws, int sm_count)
{
    const DeviceSetup* d = nullptr;
    if (N < 2 || N > kRingRanks || device_setup(&d) != cudaSuccess) return false;
    const unsigned long long resident = (unsigned long long)sm_count * (unsigned)d->ring_ctas;
    if (n > resident * kTile || (unsigned long long)(N - 1) * ((n + N - 1) / N) >= n) return false;
    const unsigned long long tiles = ring_tiles(n, N, nullptr);
    return tiles <= resident && N * tiles <= ws.state_tiles && N * (tiles / 32 + N + 1) <= group_slots(ws.state_tiles) &&
           ws.skip_publish == 0xFFFFFFFFu;
}
cudaError_t launch_ring(const RingCall& rc, const Workspace& ws, int bound_source, Params host_params, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    RingArgs ra;
    memset(&ra, 0, sizeof(ra));
    thread_local RingMaps maps;
    ra.n = rc.n; ra.m = (rc.n + rc.N - 1) / rc.N; ra.N = rc.N; ra.shift = rc.shift;
    ra.mid = rc.mid; ra.last = rc.last; ra.slot_bytes = rc.slot_bytes; ra.sizes = rc.sizes; ra.flags = rc.flags; ra.whole = rc.whole ? 1 : 0;
    const unsigned tiles = ring_tiles(rc.n, rc.N, ra.tile_begin);
    for (int r = 0; r < rc.N; ++r) {
        ra.send[r] = rc.send[r]; ra.recv[r] = rc.recv[r];
        // rank r ends with chunk r + 1 - shift of the ring
        const unsigned long long off = (unsigned long long)((r + 1 - rc.shift + rc.N) % rc.N) * ra.m;
        const unsigned long long got = rc.whole ? rc.n : (rc.n - off < ra.m ? rc.n - off : ra.m);
        if ((e = make_row_map(&maps.in[r], rc.send[r], rc.n, (uint32_t)kBlocksPerTile)) != cudaSuccess) return e;
        if ((e = make_row_map(&maps.out[r], rc.recv[r], got)) != cudaSuccess) return e;
    }
    const uint32_t op = (rc.flags >> 1) & 3u;
    count_launches(1);
    if (op == 1u || op == 2u)
        return launch_k(ring_tiles_kernel<1>, dim3(tiles), dim3(kDecodeThreads), kRingSmemBytes, st, ra, maps, ws, host_params, bound_source);
    return launch_k(ring_tiles_kernel<0>, dim3(tiles), dim3(kDecodeThreads), kRingSmemBytes, st, ra, maps, ws, host_params, bound_source);
}

// One array of at most kRangeTiles tiles with a relative bound.
cudaError_t launch_encode_relative(const Job& job, float eb, const Workspace& ws, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    JobBatchT<1> jb;
    jb.job[0] = job; jb.job[0].tile_begin = 0;
    jb.count = 1; jb.total_tiles = (uint32_t)((job.n + kTile - 1) / kTile);
    TileMapsT<1> maps;
    if ((e = make_row_map(&maps.m[0], job.x, job.n)) != cudaSuccess) return e;
    count_launches(1);
    return launch_cluster(jb.total_tiles, encode_tiles_kernel<1, true>, dim3(jb.total_tiles), dim3(kTileThreads), kEncodeTilesSmemBytes, st, jb, maps, ws,
                          Params{eb, 1.f, 1.f, 1}, 0);
}
bool encode_relative_fits(unsigned long long n) { return n > 0 && n <= (unsigned long long)kRangeTiles * kTile; }

// Up to seven tiles per SM a CTA per tile (zccl_tiles.cuh), beyond that CTAs that take tile after tile (zccl_stream.cuh).  us, the
// one / the other, arrays in turn, field at 1e-3: 444 tiles 7.0 / 7.4, 888 8.4 / 8.8, 1036 8.9 / 9.1, 1100 9.1 / 9.3, 1180 9.6 / 9.5,
// 1330 14.0 / 10.0; with a relative bound 888 14.9 / 16.0, 1100 15.7 / 16.6, 1330 20.2 / 17.8; gradients (code lengths around 10) 888
// 10.2 / 10.3, 1036 10.8 / 10.7, 1180 11.8 / 11.2; compressed and another one decompressed, field, 888 15.9 / 16.3, 1036 17.5 / 16.9.
constexpr int kTileCtas = 7;
cudaError_t launch_encode_lanes(const JobBatch& jb, const Workspace& ws, int bound_source, Params host_params, int sm_count,
                                cudaStream_t st)
{
    JobBatchT<1> one;   // 7 KB of kernel parameters less
    one.job[0] = jb.job[0]; one.count = jb.count; one.total_tiles = jb.total_tiles;
    const bool single = jb.count == 1;
    count_launches(1);
    if (jb.total_tiles <= (uint32_t)(kTileCtas * sm_count))
        return single ? launch_encode_tiles(one, ws, bound_source, host_params, st) : launch_encode_tiles(jb, ws, bound_source, host_params, st);
    return single ? launch_encode_stream(one, ws, bound_source, host_params, sm_count, st) : launch_encode_stream(jb, ws, bound_source, host_params, sm_count, st);
}

// Binary64 input: rounds into their slots, then the placement (two launches).
cudaError_t launch_encode_f64_lanes(const double* x, unsigned long long n, ParamsF64 hp, int bound_source, uint32_t* out,
                                    unsigned long long out_cap, size_t* out_bytes, const Workspace& ws, int sm_count, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    if (!ws.slots) return cudaErrorInvalidValue;
    const unsigned long long nT = (n + kTile - 1) / kTile;
    thread_local JobBatch jb;
    memset(&jb, 0, sizeof(jb));
    jb.count = 1;
    jb.total_tiles = (uint32_t)(nT ? nT : 1);
    jb.job[0].x = reinterpret_cast<const float*>(x);
    jb.job[0].out = out; jb.job[0].out_bytes = out_bytes; jb.job[0].n = n; jb.job[0].out_cap = out_cap;
    if (jb.total_tiles > ws.max_tiles) return cudaErrorInvalidValue;
    GroupTable gt;
    const uint32_t groups = group_table(jb, gt);
    e = launch_k(encode_rounds_f64_kernel, dim3(jb.total_tiles), dim3(kCodecThreads), 0, st, x, n, ws,
                 hp, bound_source, (unsigned)(sm_count * kEnc64Ctas));
    if (e != cudaSuccess) return e;
    return launch_k(place_kernel, dim3(groups), dim3(kPlaceThreads), kPlaceSmemBytes, st, jb, gt, ws, 1, hp, bound_source);
}

cudaError_t launch_decode_f64_lanes(const uint32_t* in, unsigned long long cap_bytes, double* y, unsigned long long y_cap, const Workspace& ws,
                                    int sm_count, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    CUtensorMap map;
    memset(&map, 0, sizeof(map));
    if ((e = make_row_map_f64(&map, y, y_cap)) != cudaSuccess) return e;
    const unsigned long long tiles = (y_cap + kTile - 1) / kTile;
    if (tiles >= 0xFFFFFFFFull) return cudaErrorInvalidValue;
    JobBatchT<1> jb;
    memset(&jb, 0, sizeof(jb));
    jb.count = 1;
    jb.total_tiles = (uint32_t)(tiles ? tiles : 1);
    jb.job[0].in_c = in; jb.job[0].in_cap = cap_bytes; jb.job[0].y = reinterpret_cast<float*>(y); jb.job[0].n = y_cap;
    const unsigned long long cap = (unsigned long long)sm_count * d->dec64_ctas;
    return launch_k(decode_tiles_f64_kernel, dim3((unsigned)(jb.total_tiles < cap ? jb.total_tiles : cap)), dim3(kDecodeThreads), kDec64SmemBytes, st, jb, map, ws);
}

// Binary32 at another tile size on the tuned kernels: rounds into their slots, then the placement.  False when the
// context's slots do not cover the launch (the caller then takes the plain kernels).
bool tiled_lanes_fit(unsigned long long n, uint32_t T, const Workspace& ws)
{
    const unsigned long long tiles = (n + T - 1) / T, R = (T + kRound - 1) / kRound;
    return ws.slots && tiles * R <= 4ull * ws.max_tiles;   // one slot per round; first codes and group sums are laid out for tiles of 1024
}

cudaError_t launch_encode_tiled_lanes(const float* x, unsigned long long n, uint32_t T, Params hp, bool device_params, uint32_t* out,
                                      unsigned long long out_cap, size_t* out_bytes, const Workspace& ws, int sm_count, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    if (!tiled_lanes_fit(n, T, ws)) return cudaErrorInvalidValue;
    CUtensorMap map;
    memset(&map, 0, sizeof(map));
    const bool mapped = (((uintptr_t)x) & 15u) == 0 && n >= (unsigned long long)kBlock;
    if (mapped && (e = make_row_map(&map, x, n)) != cudaSuccess) return e;
    TiledShape sp;
    sp.T = T; sp.R = (T + kRound - 1) / kRound; sp.lw_full = (T / kBlock + 3) / 4;
    const unsigned long long nT = (n + T - 1) / T;
    const uint32_t tiles = (uint32_t)(nT ? nT : 1);
    const unsigned long long rounds = (unsigned long long)tiles * sp.R;
    const unsigned long long want = (rounds + kCodecWarps - 1) / kCodecWarps;
    const unsigned long long cap = (unsigned long long)sm_count * d->round_tiled_ctas;
    e = launch_k(encode_rounds_tiled_kernel, dim3((unsigned)(want < cap ? want : cap)), dim3(kCodecThreads), kRoundSmemBytes, st, x, n, sp, tiles, map,
                 mapped ? 1 : 0, ws, hp, device_params ? 1 : 0);
    if (e != cudaSuccess) return e;
    return launch_k(place_tiled_kernel, dim3((tiles + 31u) / 32u), dim3(kPlaceThreads), 0, st, out, out_cap, out_bytes, n, sp, tiles, ws, hp,
                    device_params ? 1 : 0);
}

cudaError_t launch_decode_tiled_lanes(const uint32_t* in, unsigned long long cap_bytes, uint32_t T, float* y, unsigned long long y_cap,
                                      const Workspace& ws, int sm_count, cudaStream_t st)
{
    const DeviceSetup* d = nullptr;
    cudaError_t e = device_setup(&d);
    if (e != cudaSuccess) return e;
    CUtensorMap map;
    memset(&map, 0, sizeof(map));
    const bool mapped = (((uintptr_t)y) & 15u) == 0 && y_cap >= (unsigned long long)kBlock;
    if (mapped && (e = make_row_map(&map, y, y_cap)) != cudaSuccess) return e;
    TiledShape sp;
    sp.T = T; sp.R = (T + kRound - 1) / kRound; sp.lw_full = (T / kBlock + 3) / 4;
    const unsigned long long tiles = (y_cap + T - 1) / T;
    if (tiles >= 0xFFFFFFFFull) return cudaErrorInvalidValue;
    const unsigned long long want = (tiles + kCodecWarps - 1) / kCodecWarps;
    const unsigned long long cap = (unsigned long long)sm_count * d->dec_tiled_ctas;
    return launch_k(decode_tiles_tiled_kernel, dim3((unsigned)(want < cap ? (want ? want : 1) : cap)), dim3(kCodecThreads), kDecSmemBytes, st, in,
                    cap_bytes, sp, y, y_cap, (uint32_t)tiles, map, mapped ? 1 : 0, ws);
}

}  // namespace zccl
