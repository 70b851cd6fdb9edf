// Device-side helpers shared by the kernel translation units: scan-state words, mbarrier and bulk-copy wrappers,
// stream header parsing, job lookup, launch re-arming, and the host-side launch wrapper.  Not installed.
#pragma once
#include "zccl_internal.h"

#include <cstdlib>

namespace zccl {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kSpinLimit = 1 << 20;            // polls of a scan state or an mbarrier before giving up
constexpr float kRoundMagic = 12582912.0f;     // 1.5 * 2^23: t + kRoundMagic has rint(t) in its low mantissa bits
constexpr uint32_t kRoundMagicBits = 0x4B400000u;
constexpr float kTwo23 = 8388608.0f;           // 2^23: |d| + 2^23 has the integer |d| in its mantissa
constexpr float kGuardExact = 8.796093e12f;    // 2^43: sum of squares below it => every |x r| < 2^21.5
constexpr float kGuardSmall = 1.0e9f;          // below 2^30: no |x r| can exceed 2^15

// ------------------------------------------------------------------------------------------------ small helpers

__device__ __forceinline__ uint32_t f2key(float f)
{
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key2f(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

__device__ __forceinline__ unsigned long long pack_state(uint32_t epoch, uint32_t inclusive, uint32_t words)
{
    return ((unsigned long long)epoch << 33) | ((unsigned long long)inclusive << 32) | words;
}
__device__ __forceinline__ unsigned long long ld_state(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_state(unsigned long long* p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t ldg_u32(const uint32_t* p) { return __ldg(p); }

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// 16 bytes of shared memory by its 32-bit address: rows start on 128-byte boundaries, so the swizzled chunk k of a row is at
// (row + swizzle) ^ 16 k, one instruction less per access than row + (16 k ^ swizzle).
__device__ __forceinline__ float4 ld_shared4(uint32_t at)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ void st_shared4(uint32_t at, float4 v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait for a bulk copy to land; false after kSpinLimit polls.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t parity)
{
    for (int it = 0; it < kSpinLimit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
// 1-D bulk copy global -> this CTA's shared memory; addresses and size are multiples of 16 bytes.  The proxy
// fence orders earlier ordinary accesses to the destination before the copy engine's writes.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, unsigned long long* bar)
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// Asks for a 16-byte-aligned range of global memory to be brought into L2 (no destination, nothing to wait for).
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// Asks for a tensor map's descriptor (one thread): the first copy through it would wait for the fetch.
__device__ __forceinline__ void prefetch_map(const void* map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel)
{
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// The job that owns tile number `ticket` of the launch: the last one whose first tile is not beyond it.  Jobs of a launch
// are mostly the same size, so the search starts where the job would be if all were as large as the largest (never too
// far): one entry to look at instead of a bisection's chain of six, whose first visits miss the constant cache.
template <class JB>
__device__ __forceinline__ int find_job(const JB& jb, uint32_t ticket)
{
    if (jb.count <= 1) return 0;
    int j = (int)(ticket / jb.most_tiles);
#pragma unroll 1
    while (j + 1 < jb.count && jb.job[j + 1].tile_begin <= ticket) ++j;
    return j;
}

// Programmatic dependent launch: kernels of the library are launched with stream serialisation relaxed (but see
// overlap_allowed), so that their CTAs are dispatched while the kernel in front on the stream drains, and wait here until
// that kernel has completed and its writes are visible.  What stands in front of the wait does not depend on them: barriers, maps,
// requests that move lines into L2, a tile's number from a counter that is in order before anyone is let in, and hint_blob's look
// at two words that are read again behind it.  Only behind the wait does a kernel let the one behind it start to launch, or by
// leaving, so at most one waiting grid is resident at a time.  Without the launch attribute both instructions do nothing.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }   // one thread of a CTA is enough
__device__ __forceinline__ void pdl_enter()
{
    pdl_wait();
    pdl_release();
}

// eb -> (eb_abs, s, r), the reading used throughout: eb_abs = eb * (max - min); step shrunk by 1 - 2^-6; r by one IEEE
// division.
__device__ __forceinline__ Params params_of(float eb, float range)
{
    Params p;
    p.valid = 1;
    if (!(range > 0.0f) || !isfinite(range)) p.valid = 0;
    const float ea = __fmul_rn(eb, range);
    const float ebq = __fmul_rn(ea, 0.984375f);
    const float s = __fmul_rn(ebq, 2.0f);
    if (!(s > 0.0f) || !isfinite(s)) p.valid = 0;
    const float r = __fdiv_rn(1.0f, s);
    if (!isfinite(r)) p.valid = 0;
    p.eb_abs = ea; p.s = s; p.r = r;
    return p;
}

// Where a compression's bound comes from.
enum BoundSource { kBoundHost = 0,     // the launch's parameters
                   kBoundDevice = 1,   // the workspace's resolved bound
                   kBoundKeys = 2 };   // the keys a range pass has left: every CTA resolves the bound eb_abs (relative) itself, and
                                       // whoever re-arms the workspace puts it down and the keys back (settle_bound)
__device__ __forceinline__ Params bound_of(const Workspace& ws, const Params& hp, int source)
{
    if (source == kBoundHost) return hp;
    if (source == kBoundDevice) return *ws.params;
    const uint32_t kmin = *reinterpret_cast<volatile uint32_t*>(ws.minmax + 0), kmax = *reinterpret_cast<volatile uint32_t*>(ws.minmax + 1);
    return params_of(hp.eb_abs, kmin <= kmax ? __fsub_rn(key2f(kmax), key2f(kmin)) : 0.0f);
}
// One thread, when every CTA has the bound (one that reads the re-armed keys finds no range, so without a valid bound any
// time will do).
__device__ __forceinline__ void settle_bound(const Workspace& ws, const Params& prm, int source)
{
    if (source != kBoundKeys) return;
    *ws.params = prm;
    if (!prm.valid) atomicOr(ws.status, kStDegenerate);
    ws.minmax[0] = 0xFFFFFFFFu;
    ws.minmax[1] = 0u;
}

// The same for binary64 (the shrink 1 - 2^-20 keeps |x - x'| <= eb_abs over the whole code range).
__device__ __forceinline__ unsigned long long d2key(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double key2d(unsigned long long k)
{
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k));
}
// (out of line: its division weighed on compressions with an absolute bound, 2^24 gradients 70.8 -> 71.4 us there and back)
__device__ __noinline__ ParamsF64 params_of_f64(double eb, double range)
{
    ParamsF64 p;
    p.valid = range > 0.0 && isfinite(range) ? 1 : 0;
    const double ea = __dmul_rn(eb, range);
    const double ebq = __dmul_rn(ea, 1.0 - 9.5367431640625e-07);   // 1 - 2^-20
    const double s = __dmul_rn(ebq, 2.0);
    if (!(s > 0.0) || !isfinite(s)) p.valid = 0;
    const double r = __ddiv_rn(1.0, s);
    if (!isfinite(r)) p.valid = 0;
    p.eb_abs = ea; p.s = s; p.r = r;
    return p;
}
__device__ __forceinline__ ParamsF64 bound_of_f64(const Workspace& ws, const ParamsF64& hp, int source)
{
    if (source == kBoundHost) return hp;
    const unsigned long long kmin = *reinterpret_cast<volatile unsigned long long*>(ws.minmax64 + 0), kmax = *reinterpret_cast<volatile unsigned long long*>(ws.minmax64 + 1);
    return params_of_f64(hp.eb_abs, kmin <= kmax ? __dsub_rn(key2d(kmax), key2d(kmin)) : 0.0);
}
__device__ __forceinline__ void settle_bound_f64(const Workspace& ws, const ParamsF64& prm, int source)
{
    if (source != kBoundKeys) return;
    *ws.params64 = prm;
    if (!prm.valid) atomicOr(ws.status, kStDegenerate);
    ws.minmax64[0] = 0xFFFFFFFFFFFFFFFFull;
    ws.minmax64[1] = 0ull;
}

// ------------------------------------------------------------------------------------------------ stream header

struct StreamInfo {
    unsigned long long n;
    uint32_t nT;
    float eb_abs, s;
    bool ok;
};

__device__ __forceinline__ StreamInfo read_header(const uint32_t* in, unsigned long long cap_bytes)
{
    StreamInfo h;
    h.ok = false; h.n = 0; h.nT = 0; h.s = 1.0f; h.eb_abs = 0.0f;
    if (cap_bytes < (unsigned)kHeaderBytes) return h;
    const uint32_t magic = ldg_u32(in + 0), ver = ldg_u32(in + 1);
    const unsigned long long n = (unsigned long long)ldg_u32(in + 2) | ((unsigned long long)ldg_u32(in + 3) << 32);
    const float eb_abs = __uint_as_float(ldg_u32(in + 4)), s = __uint_as_float(ldg_u32(in + 5));
    const uint32_t T = ldg_u32(in + 6), nT = ldg_u32(in + 7);
    if (magic != kMagic || ver != kVersion || T != (uint32_t)kTile) return h;
    if ((n + kTile - 1) / kTile != nT) return h;
    if (cap_bytes < (unsigned long long)kHeaderBytes + 4ull * nT) return h;
    if (!(s > 0.0f) || !isfinite(s)) return h;
    h.n = n; h.nT = nT; h.eb_abs = eb_abs; h.s = s; h.ok = true;
    return h;
}

__device__ __forceinline__ void write_header(uint32_t* out, int tid, unsigned long long n, float eb_abs, float s, uint32_t nT)
{
    if (tid < kHeaderWords) {
        uint32_t hv;
        switch (tid) {
            case 0: hv = kMagic; break;
            case 1: hv = kVersion; break;
            case 2: hv = (uint32_t)n; break;
            case 3: hv = (uint32_t)(n >> 32); break;
            case 4: hv = __float_as_uint(eb_abs); break;
            case 5: hv = __float_as_uint(s); break;
            case 6: hv = kTile; break;
            default: hv = nT; break;
        }
        out[tid] = hv;
    }
}

__device__ __forceinline__ void mbar_arrive(unsigned long long* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

inline bool pdl_enabled()
{
    static const bool on = [] { const char* e = getenv("ZCCL_PDL"); return !(e && e[0] == '0'); }();
    return on;
}

// cluster: CTAs per thread-block cluster; kind: see overlap_allowed
template <class... KArgs, class... Args>
cudaError_t launch_any(LaunchKind kind, unsigned cluster, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = overlap_allowed(st, kind) && pdl_enabled() ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <class... KArgs, class... Args>
cudaError_t launch_cluster(unsigned cluster, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args)
{
    return launch_any(kLaunchOther, cluster, kernel, grid, block, smem, st, static_cast<Args&&>(args)...);
}
template <class... KArgs, class... Args>
cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args)
{
    return launch_any(kLaunchOther, 1, kernel, grid, block, smem, st, static_cast<Args&&>(args)...);
}


}  // namespace
}  // namespace zccl
