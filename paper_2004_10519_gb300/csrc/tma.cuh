// TMA plane-ring machinery shared by the TMA-fed stencil passes: tile
// geometry (32 z x FY y columns, two z points per consumer thread, one
// producer warp), mbarrier and cp.async.bulk.tensor helpers in inline PTX,
// the bounded producer/consumer ring, and the host side that encodes
// (and caches per handle) the 3D tensor maps.
//
// The tile height FY is a compile-time constant of the translation unit
// (WP_TILE_Y: 8, 16 or 32 rows; 16 unless the unit defines it).  The
// stencil passes are compiled once per height and the autotuner picks one
// per grid; the arithmetic of a point does not depend on the tile, so every
// height gives the same bits.
#pragma once
#include "tile.cuh"

#include <cuda.h>
#include <algorithm>
#include <cstdlib>
#include <mutex>

#ifndef WP_TILE_Y
#define WP_TILE_Y 16
#endif
static_assert(WP_TILE_Y == 8 || WP_TILE_Y == 16 || WP_TILE_Y == 32, "tile height must be 8, 16 or 32");

namespace {

constexpr int FY = WP_TILE_Y;
using tile::FZ;

constexpr int TZ2 = FZ / 2;        // threads along z, two points each
constexpr int NT2 = TZ2 * FY;      // consumer threads per CTA (FY / 2 warps)
constexpr int NTP = NT2 + 32;      // + one producer warp
// resident CTAs per SM for the launch bounds: `base` at 16 rows, scaled
// with the CTA size (a 32-row CTA has the threads of two 16-row ones)
constexpr int occ(int base) { return FY == 8 ? 2 * base : (FY == 32 ? 1 : base); }
// Elastic passes above space order 8 need more than 96 registers per thread
// and more shared memory than two CTAs per SM allow: they run one CTA per SM.
constexpr int NSTAGE = 3;

// ---------------------------------------------------------------------------
// device: mbarrier / TMA helpers (inline PTX)
// ---------------------------------------------------------------------------
WP_DEV uint32_t saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

WP_DEV void mbar_init(uint64_t *bar, int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count) : "memory");
}
WP_DEV void fence_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
WP_DEV void mbar_expect(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)), "r"(bytes)
                 : "memory");
}
#ifdef WP_CHECK
WP_DEV bool ck_tma(const float *dst, int c0);
#endif
WP_DEV void tma3(float *dst, const CUtensorMap *map, int c0, int c1, int c2, uint64_t *bar)
{
#ifdef WP_CHECK
    if (!ck_tma(dst, c0)) return;
#endif
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            saddr(dst)),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(saddr(bar))
        : "memory");
}
WP_DEV bool mbar_try(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(saddr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
WP_DEV uint64_t gtimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// wait for phase `parity` of bar; false after ~2 s
WP_DEV bool mbar_wait(uint64_t *bar, uint32_t parity)
{
    if (mbar_try(bar, parity)) return true;
    const uint64_t t0 = gtimer();
    while (!mbar_try(bar, parity))
        if (gtimer() - t0 > 2000000000ull) return false;
    return true;
}
WP_DEV void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}
// producer after an abort: wait (bounded) for the stages of iterations
// [a, b] that may still be in flight, so no copy lands after the CTA exits
WP_DEV void drain(uint64_t *full, int ns, int a, int b)
{
    for (int j = a < 0 ? 0 : a; j <= b; j++) mbar_wait(&full[j % ns], (uint32_t)((j / ns) & 1));
}

// 8-byte accesses (z even, row pitch even: always aligned)
// Bounds-checking build (WP_CHECK, selected at run time by WAVEPROP_CHECK=1):
// every shared-memory read must lie in the CTA's dynamic shared memory, every
// global float2 access of a field below the grid size and every TMA copy
// start on a 16-byte boundary in x and in shared memory.  A failing access is
// skipped (loads return zeros) and bit 8 of the handle's error word is set,
// which the host reports as PROP_ECUDA; nothing traps, and a skipped copy
// ends in the bounded wait of its stage (bit 2).  In the normal build the
// checks compile to nothing.
#ifdef WP_CHECK
static __shared__ unsigned long long wp_ck_n;   // elements of a field
static __shared__ int *wp_ck_err;
extern __shared__ __align__(128) float wp_dsm[];
WP_DEV void ck_begin(unsigned long long n, int *err)
{
    wp_ck_n = n;
    wp_ck_err = err;
}
WP_DEV bool ck_fail()
{
    atomicOr(wp_ck_err, 8);
    return false;
}
WP_DEV bool ck_smem(const void *p, unsigned bytes)
{
    unsigned dyn;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    const uint32_t a = saddr(p), b = saddr(wp_dsm);
    return (a >= b && a + bytes <= b + dyn && (a & (bytes - 1)) == 0) || ck_fail();
}
WP_DEV bool ck_field(unsigned o) { return (unsigned long long)o + 2 <= wp_ck_n || ck_fail(); }
// x (innermost, z) coordinate of a copy: 16-byte multiple; destination
// 16-byte aligned inside the dynamic shared memory
WP_DEV bool ck_tma(const float *dst, int c0) { return ((c0 & 3) == 0 || ck_fail()) && ck_smem(dst, 16); }
#else
WP_DEV void ck_begin(unsigned long long, int *) {}
#endif

WP_DEV float2 lds2(const float *p)
{
#ifdef WP_CHECK
    if (!ck_smem(p, 8)) return make_float2(0.f, 0.f);
#endif
    return *reinterpret_cast<const float2 *>(p);
}
// a pair of a field that the kernel before may still be writing when this one
// starts (launch_pass): an ordinary load, after pass_waits.  Never __ldg, nor
// through a restrict pointer: read-only loads may move above the wait, and read
// lines fetched before it
WP_DEV float2 ldf2(const float *p, unsigned o)
{
#ifdef WP_CHECK
    if (!ck_field(o)) return make_float2(0.f, 0.f);
#endif
    return *reinterpret_cast<const float2 *>(p + o);
}
WP_DEV void st2(float *p, unsigned o, float a, float b)
{
#ifdef WP_CHECK
    if (!ck_field(o)) return;
#endif
    *reinterpret_cast<float2 *>(p + o) = make_float2(a, b);
}
WP_DEV float2 dif2(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// paired FP32 arithmetic (one instruction for both lanes; per component the
// result of the scalar operation)
WP_DEV float2 f2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
WP_DEV float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
WP_DEV float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
WP_DEV float2 f2s(float a) { return make_float2(a, a); }
// a - b as fma(-1, b, a): the same rounding as the subtraction
WP_DEV float2 f2sub(float2 a, float2 b) { return __ffma2_rn(make_float2(-1.f, -1.f), b, a); }

// x / a, correctly rounded, from y = RN(1/a) shared by several quotients of the
// same divisor: q = RN(x y), corrected by its exact remainder (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor",
// IBM J. Res. Dev. 34, 1990).  Holds while the remainder, 2^-24 of x, is a normal
// number or zero; an infinite x gives NaN.
WP_DEV float2 div_by(float2 x, float2 a, float2 y)
{
    const float2 q = f2mul(x, y);
    const float2 r = f2fma(make_float2(-a.x, -a.y), q, x);
    return f2fma(r, y, q);
}

// out of line: inlined into the unrolled acoustic pass it cost 2 to 4 % of its time
static __device__ __noinline__ float2 div_ieee(float2 x, float2 a)
{
    return make_float2(__fdiv_rn(x.x, a.x), __fdiv_rn(x.y, a.y));
}
// x / a of a pair for a from 2^-35 to 2^35 (m (1 + sd), m in s^2/m^2): the rounded
// quotient, also where it is infinite or NaN or its operands too large to be scaled;
// below 2^-112 possibly the next number to it
WP_DEV float2 div_model(float2 x, float2 a)
{
    // both times 2^32: the remainder stays a normal number down to quotients of 2^-112
    const float2 sc = make_float2(4294967296.f, 4294967296.f), as = f2mul(a, sc);
    const float2 q = div_by(f2mul(x, sc), as, make_float2(__frcp_rn(as.x), __frcp_rn(as.y)));
    return isfinite(q.x + q.y) ? q : div_ieee(x, a);
}

constexpr int al32(int n) { return (n + 31) & ~31; }   // 128-byte aligned float offsets
constexpr int IS = FZ * FY;                             // interior box (tile of one plane)

// box geometries (floats): rows x cols
template <int M>
struct BX {
    static constexpr int MZ = (M + 3) & ~3;                     // z halo rounded to 16 bytes
    static constexpr int YR = FY + 2 * M, YC = FZ;              // y-halo box
    static constexpr int ZR = FY, ZC = FZ + 2 * MZ;             // z-halo box
    static constexpr int RR = FY + 2 * M, RC = FZ + 2 * MZ;     // rectangle (y and z halo)
    static constexpr int PR = FY + 1, PC = FZ + 4;              // +1 box (interior + row/col)
    static constexpr int YS = al32(YR * YC), ZS = al32(ZR * ZC), RS = al32(RR * RC), PS = al32(PR * PC);
};

// z window of 2M+2 values starting M before the thread's first point:
// w[M + d] = f(z + d), d = -M .. M+1
template <int M>
WP_DEV void zwin(const float *row, int cz, float (&w)[2 * M + 2])
{
#pragma unroll
    for (int j = 0; j <= M; j++) {
        const float2 a = lds2(row + cz - M + 2 * j);
        w[2 * j] = a.x;
        w[2 * j + 1] = a.y;
    }
}

// Programmatic dependent launch of the passes (launch_pass): a pass's CTAs may
// start when every CTA of the kernel before it has, set up their barriers, and
// wait here, before they touch anything in memory, until that kernel has
// completed and its writes are visible.  Hides the launch latency and the
// prologue behind the last CTAs of the pass before.  No effect in a kernel
// that was launched without the attribute.  The fields of such a pass (what any
// pass writes) come by TMA or ordinary loads, and its field pointers carry no
// restrict, for only those are ordered by the wait; __ldg is for the model, the
// layer tables, the sparse-point tables and the wavelets, which no pass writes.
WP_DEV void pass_begins() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
WP_DEV void pass_waits() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The CTAs of a pass beyond its x chunks (blockIdx.z >= nz) sample the receivers
// of the step, one per thread; true for such a CTA.  Saves a launch per step
// that only reads what the pass reads.
WP_DEV bool sample_receivers(const RecDev &r, int nz)
{
    if ((int)blockIdx.z < nz) return false;
    pass_waits();
    const int nth = blockDim.x * blockDim.y, tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int i = (((int)blockIdx.z - nz) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    const long long k = (long long)i * nth + tid;
    if (k < r.n) r.out[k] = record_point(r.idx, r.w, (int)k, r.f0, r.f1, r.f2);
    return true;
}
// the z layers of CTAs that this takes
inline unsigned receiver_layers(const RecDev &r, dim3 grd, dim3 blk)
{
    const long long ctas = ((long long)r.n + blk.x * blk.y - 1) / (blk.x * blk.y), layer = (long long)grd.x * grd.y;
    return (unsigned)((ctas + layer - 1) / layer);
}
// Source terms of the step at the points of a column pair (in-plane offset q0,
// planes [xa, xb)) that this thread has written: f(cell offset, plane, j) for
// each of the cells among them.  A handful of compares per thread and chunk.
template <class F>
WP_DEV void own_sources(const InjDev &I, unsigned q0, int xa, int xb, F f)
{
    for (int j = 0; j < I.n; j++)
        if (I.o[j] - q0 < 2u && I.x[j] >= xa && I.x[j] < xb) f(I.o[j], I.x[j], j);
}

// Producer/consumer plane ring.  full[s] completes when the copies of a
// stage have landed (one arrive with the byte count + the TMA bytes);
// empty[s] when every consumer warp has finished reading it (one arrive per
// warp).  A dedicated producer warp (its lane 0) keeps ns planes in
// flight: it refills a stage as soon as it is released, so consumers never
// wait for each other.  All waits are bounded; a warp that gives up reports
// bit 2 and leaves, and the producer drains its copies in flight first.
constexpr int NWARP = NT2 / 32;

// Stages of the ring: as many as the launch's dynamic shared memory holds behind
// the barriers (8 full, 8 empty) and the number of stages, which the consumers
// read there once a plane rather than hold in a register.
constexpr int MAX_STAGES = 8, BAR_BYTES = 16 * MAX_STAGES + 128;
// dynamic shared memory per CTA (1 KB below the opt-in limit, for static variables) and per SM
constexpr size_t SMEM_MAX = 226 * 1024, SMEM_SM = 228 * 1024;
constexpr size_t ring_bytes(int ns, int stage) { return (size_t)ns * stage * sizeof(float) + BAR_BYTES; }
WP_DEV int ring_stages(int stage)
{
    unsigned dyn;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    return (int)((dyn - BAR_BYTES) / (unsigned)(stage * sizeof(float)));
}
// Dynamic shared memory of a pass of `ctas` CTAs of which `occ` fit an SM: at least
// `least` stages, and where the grid leaves an SM fewer CTAs than fit it, the
// memory of the missing ones as further stages (up to the planes of a chunk).  A
// plane's copies take about three times as long as its arithmetic, so three planes
// in flight keep up when two CTAs or more share an SM, but not when one is alone.
// TTI so 8, 84^3 (99 CTAs), 3 and 4 stages -> 7 and 8: 19.1 -> 17.5 us per step.
inline size_t ring_smem(const prop_s *P, dim3 grd, int occ, int stage, int least)
{
    const long long ctas = (long long)grd.x * grd.y * grd.z;
    const int res = (int)std::min<long long>(occ, std::max<long long>(1, (ctas + P->sms - 1) / P->sms));
    int ns = least;
    if (res < occ) {
        const size_t room = std::min(SMEM_MAX, SMEM_SM / res - 1024);      // 1 KB per CTA is the system's
        ns = (int)std::min<size_t>({(size_t)MAX_STAGES, (size_t)P->xchunk, (room - BAR_BYTES) / (stage * sizeof(float))});
    }
    return ring_bytes(std::max(ns, least), stage);
}

// NS > 0: that many stages, a constant (for a pass without a register to spare).
template <int NS = 0>
struct RingN {
    uint64_t *full;
    int st = 0;
    uint32_t ph = 0;
    WP_DEV explicit RingN(uint64_t *bars) : full(bars) {}
    WP_DEV uint64_t *empty(int s) { return full + MAX_STAGES + s; }
    WP_DEV int stages() { return NS ? NS : *reinterpret_cast<const volatile int *>(full + 2 * MAX_STAGES); }
    WP_DEV void init(int ns)
    {
        *reinterpret_cast<volatile int *>(full + 2 * MAX_STAGES) = ns;
        for (int i = 0; i < ns; i++) {
            mbar_init(&full[i], 1);
            mbar_init(empty(i), NWARP);
        }
        fence_init();
    }
    // producer (lane 0 of the producer warp): plane xa + it into stage it % ns
    template <class F>
    WP_DEV void produce(int xa, int nit, F issue, int *err)
    {
        const int ns = stages();
        int s = 0;
        uint32_t lap = 1;                    // parity of the release of the lap before
        for (int it = 0; it < nit; it++) {
            if (it >= ns && !mbar_wait(empty(s), lap)) {
                atomicOr(err, 2);
                drain(full, ns, it - ns, it - 1);
                return;
            }
            issue(xa + it, s);
            if (++s == ns) {
                s = 0;
                lap ^= 1u;
            }
        }
        // stay until the last copies have landed (bounded), so none can
        // arrive after the CTA has exited even if the consumers gave up
        drain(full, ns, nit - ns, nit - 1);
    }
    WP_DEV bool wait_full() { return mbar_wait(&full[st], ph); }
    // end of iteration: this warp is done with the stage
    WP_DEV void release(int lane)
    {
        __syncwarp();
        if (lane == 0) mbar_arrive(empty(st));
        if (++st == stages()) {
            st = 0;
            ph ^= 1u;
        }
    }
};
using Ring = RingN<>;


// ---------------------------------------------------------------------------
// host: tensor maps
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                CUtensorMapFloatOOBfill);

EncodeTiled encode_fn()
{
    static EncodeTiled fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiled)f;
    });
    return fn;
}

// 3D map of a [NX][NY][NZ] float array with rows PZ floats apart, box (bz, by,
// 1); zero fill outside the grid, the row padding included
bool make_map(CUtensorMap *m, const float *base, const GridDev &g, int bz, int by)
{
    EncodeTiled fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)g.NZ, (cuuint64_t)g.NY, (cuuint64_t)g.NX};
    cuuint64_t strides[2] = {(cuuint64_t)g.PZ * 4, (cuuint64_t)g.PZ * g.NY * 4};
    cuuint32_t box[3] = {(cuuint32_t)bz, (cuuint32_t)by, 1};
    cuuint32_t es[3] = {1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, (void *)base, dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// descriptor of (array, box) from the handle's cache; false if encoding failed
bool map_of(prop_s *P, const float *base, int bz, int by, CUtensorMap *out)
{
    const auto key = std::make_tuple((const void *)base, bz, by);
    auto it = P->tmaps.find(key);
    if (it == P->tmaps.end()) {
        CUtensorMap m;
        if (!make_map(&m, base, P->g, bz, by)) return false;
        it = P->tmaps.emplace(key, m).first;
    }
    *out = it->second;
    return true;
}

// launch of a pass whose kernel begins with pass_begins and pass_waits
template <class... A, class... B>
void launch_pass(void (*kernel)(A...), dim3 grd, dim3 blk, size_t smem, cudaStream_t st, B... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grd;
    c.blockDim = blk;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kernel, static_cast<A>(args)...);     // errors: cudaGetLastError by the caller
}

template <class K>
bool set_smem(K kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

}  // namespace
