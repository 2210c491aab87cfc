// 2D elastic propagator (x-z plane): the velocity-stress system of Sec. IV-A
// (Eq. elas1, elastic listing) with every y term dropped, as in the 2D
// example of Sec. IV-B.  Fields on the staggered grid of the 3D system:
// vx at (x+1/2, z), vz at (x, z+1/2), txx and tzz at nodes, txz at
// (x+1/2, z+1/2); b averaged over the two nodes of a velocity point, mu
// over the four nodes around the txz point; Cerjan taper from the layer
// tables.  The step is two passes (velocity, then stress with the new
// velocities) over 32 x 32 tiles staged in shared memory with their halos
// (2D working sets mostly sit in L2): fed by TMA where the rows are whole
// 16-byte units (padded, see row_pitch), by plain loads otherwise.  dt_sign = -1
// runs the transposed step in the (b_avg vbar, g C tbar) variables (the taper, C
// and the averages are pointwise), which adjoint modelling uses.
#include "tma.cuh"

namespace {

// Tile of 32 (z) x 32 (x) points per CTA of 32 x 8 threads (four x points
// per thread).  Each differentiated field is staged once in shared memory
// with its halo (zero outside the grid = the zero extension of the
// operators); the taps then read shared rows (one wavefront per warp
// access) instead of unaligned read-only-cache loads.
constexpr int TZ = 32, TXR = 32, BXR = 8;

template <int M>
struct Tile2 {
    static constexpr int R = TXR + 2 * M, C = TZ + 2 * M;   // rows (x), columns (z) with halo
};

// stage f[x0 - HX .. x0 + TXR + HX) x [z0 - HZ .. z0 + TZ + HZ) into s (row
// pitch TZ + 2 HZ); a fixed trip count lets every load of a thread be in
// flight before its shared stores
template <int HX, int HZ>
WP_DEV void stage(float *s, const float *__restrict__ f, const GridDev &g, int x0, int z0)
{
    constexpr int cols = TZ + 2 * HZ, n = (TXR + 2 * HX) * cols, NTH = TZ * BXR, IT = (n + NTH - 1) / NTH;
    const int tid = threadIdx.y * TZ + threadIdx.x;
    float v[IT];
#pragma unroll
    for (int it = 0; it < IT; it++) {
        const int i = tid + it * NTH, r = i / cols, c = i % cols;
        const int x = x0 - HX + r, z = z0 - HZ + c;
        v[it] = (i < n && x >= 0 && x < g.NX && z >= 0 && z < g.NZ) ? __ldg(f + (long long)x * g.PZ + z) : 0.f;
    }
#pragma unroll
    for (int it = 0; it < IT; it++) {
        const int i = tid + it * NTH;
        if (i < n) s[i] = v[it];
    }
}

// v <- g (v + c b_avg Dtau(tau)),  c = dt / h (signed)
template <int M>
__global__ void __launch_bounds__(TZ * BXR)
el2_vpass(GridDev g, FDW w, float *vx, float *vz, const float *__restrict__ txx, const float *__restrict__ tzz,
          const float *__restrict__ txz, const float *__restrict__ bu, float c)
{
    using T = Tile2<M>;
    __shared__ float sxx[T::R * TZ], sxz[T::R * T::C], szz[TXR * T::C];
    const int z0 = blockIdx.x * TZ, x0 = blockIdx.y * TXR;
    stage<M, 0>(sxx, txx, g, x0, z0);
    stage<M, M>(sxz, txz, g, x0, z0);
    stage<0, M>(szz, tzz, g, x0, z0);
    __syncthreads();
    const int tz = threadIdx.x, z = z0 + tz;
    if (z >= g.NZ) return;
    const float *tzt = g.tab + 2 * (g.NX + g.NY);
    const float gy = __ldg(g.tab + 2 * g.NX), gzn = __ldg(tzt + 2 * z), gzh = __ldg(tzt + 2 * z + 1);
    const int z1 = min(z + 1, g.NZ - 1);
#pragma unroll
    for (int j = 0; j < TXR / BXR; j++) {
        const int r = threadIdx.y * (TXR / BXR) + j, x = x0 + r;
        if (x >= g.NX) break;
        float dx = 0.f, dz = 0.f;
        const float *rxx = sxx + (r + M) * TZ + tz, *rxz = sxz + (r + M) * T::C + tz + M,
                    *rzz = szz + r * T::C + tz + M;
#pragma unroll
        for (int k = 1; k <= M; k++) {
            const float b = w.b[k - 1];
            // vx: D+x txx + D-z txz ;  vz: D-x txz + D+z tzz
            dx += b * ((rxx[k * TZ] - rxx[(1 - k) * TZ]) + (rxz[k - 1] - rxz[-k]));
            dz += b * ((rxz[(k - 1) * T::C] - rxz[-k * T::C]) + (rzz[k] - rzz[1 - k]));
        }
        const long long q = (long long)x * g.PZ + z;
        const float b0 = __ldg(bu + q);
        const float bx = 0.5f * (b0 + __ldg(bu + (long long)min(x + 1, g.NX - 1) * g.PZ + z));
        const float bz = 0.5f * (b0 + __ldg(bu + (long long)x * g.PZ + z1));
        const float gvx = __ldg(g.tab + 2 * x + 1) * gy * gzn;
        const float gvz = __ldg(g.tab + 2 * x) * gy * gzh;
        vx[q] = gvx * (vx[q] + c * bx * dx);
        vz[q] = gvz * (vz[q] + c * bz * dz);
    }
}

// tau <- g (tau + c C S(v)),  c = dt / h (signed)
template <int M>
__global__ void __launch_bounds__(TZ * BXR)
el2_tpass(GridDev g, FDW w, const float *__restrict__ vx, const float *__restrict__ vz, float *txx, float *tzz,
          float *txz, const float *__restrict__ lam, const float *__restrict__ mu, float c, int *flag, int check)
{
    using T = Tile2<M>;
    __shared__ float svx[T::R * T::C], svz[T::R * T::C];
    const int z0 = blockIdx.x * TZ, x0 = blockIdx.y * TXR;
    stage<M, M>(svx, vx, g, x0, z0);
    stage<M, M>(svz, vz, g, x0, z0);
    __syncthreads();
    const int tz = threadIdx.x, z = z0 + tz;
    if (z >= g.NZ) return;
    const float *tzt = g.tab + 2 * (g.NX + g.NY);
    const float gy = __ldg(g.tab + 2 * g.NX), gzn = __ldg(tzt + 2 * z), gzh = __ldg(tzt + 2 * z + 1);
    const int z1 = min(z + 1, g.NZ - 1);
#pragma unroll
    for (int j = 0; j < TXR / BXR; j++) {
        const int r = threadIdx.y * (TXR / BXR) + j, x = x0 + r;
        if (x >= g.NX) break;
        const float *rvx = svx + (r + M) * T::C + tz + M, *rvz = svz + (r + M) * T::C + tz + M;
        float exx = 0.f, ezz = 0.f, gxz = 0.f;
#pragma unroll
        for (int k = 1; k <= M; k++) {
            const float b = w.b[k - 1];
            exx += b * (rvx[(k - 1) * T::C] - rvx[-k * T::C]);
            ezz += b * (rvz[k - 1] - rvz[-k]);
            gxz += b * ((rvx[k] - rvx[1 - k]) + (rvz[k * T::C] - rvz[(1 - k) * T::C]));
        }
        const long long q = (long long)x * g.PZ + z;
        const int x1 = min(x + 1, g.NX - 1);
        const float mxz = 0.25f * ((__ldg(mu + q) + __ldg(mu + (long long)x * g.PZ + z1)) +
                                   (__ldg(mu + (long long)x1 * g.PZ + z) + __ldg(mu + (long long)x1 * g.PZ + z1)));
        const float l = __ldg(lam + q), m = __ldg(mu + q), tr = exx + ezz;
        const float gn = __ldg(g.tab + 2 * x) * gy * gzn;
        const float gxzt = __ldg(g.tab + 2 * x + 1) * gy * gzh;
        const float a = gn * (txx[q] + c * (l * tr + 2.f * m * exx));
        const float d = gn * (tzz[q] + c * (l * tr + 2.f * m * ezz));
        const float e = gxzt * (txz[q] + c * mxz * gxz);
        txx[q] = a;
        tzz[q] = d;
        txz[q] = e;
        if (check && !(isfinite(a) && isfinite(d) && isfinite(e))) atomicOr(flag, 1);
    }
}

// ---------------------------------------------------------------------------
// The same passes fed by TMA.  A CTA of 256 threads owns 64 (z) x TX (x) points;
// one thread has every box of the tile copied to shared memory (out-of-grid
// elements arrive as zeros), then each thread updates 4 z points on TX / 16 rows
// with 16-byte shared and global accesses.  Bound by the latency of one tile
// (copy, then compute): so little of it as the boxes allow, three CTAs of 32 rows
// per SM to overlap them, 16 rows where 32 leave SMs without a tile, and each pass
// launched into the tail of the one before.  Against the plain-load passes at
// 1781 x 781, so 8 (both passes, sampling and injection): 38.9 -> 20.7 us per step.
// ---------------------------------------------------------------------------
constexpr int QZ = 64, QT = 256;       // z points per tile, threads

template <int M, int TX>
struct Box2 {
    static constexpr int MZ = (M + 3) & ~3;                 // z halo rounded to 16 bytes
    static constexpr int R = TX + 2 * M, ZC = QZ + 2 * MZ;  // rows with x halo, columns with z halo
    static constexpr int PR = TX + 1, PC = QZ + 4;          // one row and one column more
    static constexpr int IN = al32(TX * QZ), XH = al32(R * QZ), ZH = al32(TX * ZC), XZ = al32(R * ZC),
                         P1 = al32(PR * PC);
};
// velocity pass: [t_xx (x halo)] [t_xz (x, z halo)] [t_zz (z halo)] [v_x] [v_z] [b (+1)]
template <int M, int TX>
struct LV2 {
    using B = Box2<M, TX>;
    static constexpr int OXX = 0, OXZ = B::XH, OZZ = OXZ + B::XZ, OVX = OZZ + B::ZH, OVZ = OVX + B::IN,
                         OB = OVZ + B::IN, SZ = OB + B::P1;
    static constexpr uint32_t BYTES = 4u * (B::R * QZ + B::R * B::ZC + TX * B::ZC + 2 * TX * QZ + B::PR * B::PC);
};
// stress pass: [v_x (x, z halo)] [v_z (x, z halo)] [t_xx] [t_zz] [t_xz] [lambda] [mu (+1)]
template <int M, int TX>
struct LT2 {
    using B = Box2<M, TX>;
    static constexpr int OVX = 0, OVZ = B::XZ, OT = 2 * B::XZ, OL = OT + 3 * B::IN, OM = OL + B::IN, SZ = OM + B::P1;
    static constexpr uint32_t BYTES = 4u * (2 * B::R * B::ZC + 4 * TX * QZ + B::PR * B::PC);
};
struct Maps2 {
    CUtensorMap m[7];        // in the order of the boxes
};

WP_DEV void tma2(float *dst, const CUtensorMap *map, int z, int x, uint64_t *bar)
{
#ifdef WP_CHECK
    if (!ck_tma(dst, z)) return;
#endif
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            saddr(dst)),
        "l"(map), "r"(z), "r"(x), "r"(saddr(bar))
        : "memory");
}
WP_DEV void lds4(const float *p, float *o)
{
#ifdef WP_CHECK
    if (!ck_smem(p, 16)) {
        o[0] = o[1] = o[2] = o[3] = 0.f;
        return;
    }
#endif
    const float4 v = *reinterpret_cast<const float4 *>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
WP_DEV void st4(float *p, long long q, const float *o)
{
#ifdef WP_CHECK
    if (!ck_field((unsigned)q + 2)) return;
#endif
    *reinterpret_cast<float4 *>(p + q) = make_float4(o[0], o[1], o[2], o[3]);
}
// the z window of 4 points: w[MZ + d] = f(z + d), d = -MZ .. MZ + 3
template <int MZ>
WP_DEV void win4(const float *row, float (&w)[2 * MZ + 4])
{
#pragma unroll
    for (int j = 0; j < 2 * MZ + 4; j += 4) lds4(row + j, w + j);
}
// barrier, copies of the tile by thread 0, bounded wait; false: timed out
template <class F>
WP_DEV bool load_tile(const GridDev &g, uint64_t *bar, uint32_t bytes, int *err, F copies)
{
    pass_begins();
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        fence_init();
        ck_begin(g.N, err);
    }
    __syncthreads();
    pass_waits();
    if (threadIdx.x == 0) {
        mbar_expect(bar, bytes);
        copies();
    }
    if (mbar_wait(bar, 0)) return true;
    atomicOr(err, 2);
    if (threadIdx.x == 0) mbar_wait(bar, 0);       // no copy may land after the CTA has gone
    return false;
}
// tapers at the 4 nodes and half points in z
WP_DEV void tapers4(const GridDev &g, int z, float (&gn)[4], float (&gh)[4])
{
    const float *tzt = g.tab + 2 * (g.NX + g.NY);
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int zc = min(z + i, g.NZ - 1);
        gn[i] = __ldg(tzt + 2 * zc);
        gh[i] = __ldg(tzt + 2 * zc + 1);
    }
}

template <int M, int TX>
__global__ void __launch_bounds__(QT, 3)
el2_vpass_tma(GridDev g, FDW w, float *vx, float *vz, const __grid_constant__ Maps2 mp, float c,
              const __grid_constant__ RecDev rec, int *err)
{
    using L = LV2<M, TX>;
    using B = Box2<M, TX>;
    constexpr int MZ = B::MZ;
    extern __shared__ __align__(128) float sm[];
    if (sample_receivers(rec, 1)) return;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + L::SZ);
    const int z0 = blockIdx.x * QZ, x0 = blockIdx.y * TX;
    if (!load_tile(g, bar, L::BYTES, err, [&] {
            tma2(sm + L::OXX, &mp.m[0], z0, x0 - M, bar);
            tma2(sm + L::OXZ, &mp.m[1], z0 - MZ, x0 - M, bar);
            tma2(sm + L::OZZ, &mp.m[2], z0 - MZ, x0, bar);
            tma2(sm + L::OVX, &mp.m[3], z0, x0, bar);
            tma2(sm + L::OVZ, &mp.m[4], z0, x0, bar);
            tma2(sm + L::OB, &mp.m[5], z0, x0, bar);
        }))
        return;
    const int q4 = 4 * (threadIdx.x & 15), z = z0 + q4;
    if (z >= g.NZ) return;
    const float gy = __ldg(g.tab + 2 * g.NX);
    float gzn[4], gzh[4];
    tapers4(g, z, gzn, gzh);
#pragma unroll 1
    for (int r = threadIdx.x >> 4; r < TX; r += QT / 16) {
        const int x = x0 + r;
        if (x >= g.NX) break;
        float wxz[2 * MZ + 4], wzz[2 * MZ + 4], dx[4] = {}, dz[4] = {};
        win4<MZ>(sm + L::OXZ + (r + M) * B::ZC + q4, wxz);
        win4<MZ>(sm + L::OZZ + r * B::ZC + q4, wzz);
        const float *xx = sm + L::OXX + (r + M) * QZ + q4, *xz = sm + L::OXZ + (r + M) * B::ZC + MZ + q4;
#pragma unroll
        for (int k = 1; k <= M; k++) {
            const float b = w.b[k - 1];
            float xp[4], xm[4], zp[4], zm[4];
            lds4(xx + k * QZ, xp);
            lds4(xx + (1 - k) * QZ, xm);
            lds4(xz + (k - 1) * B::ZC, zp);
            lds4(xz - k * B::ZC, zm);
#pragma unroll
            for (int i = 0; i < 4; i++) {
                // vx: D+x txx + D-z txz ;  vz: D-x txz + D+z tzz
                dx[i] += b * ((xp[i] - xm[i]) + (wxz[MZ + i + k - 1] - wxz[MZ + i - k]));
                dz[i] += b * ((zp[i] - zm[i]) + (wzz[MZ + i + k] - wzz[MZ + i + 1 - k]));
            }
        }
        const float *sb = sm + L::OB + r * B::PC + q4;
        float b0[5], b1[4], ox[4], oz[4];
        lds4(sb, b0);
        b0[4] = sb[4];
        lds4(x + 1 < g.NX ? sb + B::PC : sb, b1);
        lds4(sm + L::OVX + r * QZ + q4, ox);
        lds4(sm + L::OVZ + r * QZ + q4, oz);
        const float gxn = __ldg(g.tab + 2 * x) * gy, gxh = __ldg(g.tab + 2 * x + 1) * gy;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const float bz = 0.5f * (b0[i] + (z + i + 1 < g.NZ ? b0[i + 1] : b0[i]));
            ox[i] = gxh * gzn[i] * (ox[i] + c * (0.5f * (b0[i] + b1[i])) * dx[i]);
            oz[i] = gxn * gzh[i] * (oz[i] + c * bz * dz[i]);
        }
        const long long q = (long long)x * g.PZ + z;       // beyond an odd NZ: b = v = 0, so zeros
        st4(vx, q, ox);
        st4(vz, q, oz);
    }
}

template <int M, int TX>
__global__ void __launch_bounds__(QT, 3)
el2_tpass_tma(GridDev g, FDW w, float *txx, float *tzz, float *txz, const __grid_constant__ Maps2 mp, float c,
              const __grid_constant__ InjDev inj, int check, int *err)
{
    using L = LT2<M, TX>;
    using B = Box2<M, TX>;
    constexpr int MZ = B::MZ;
    extern __shared__ __align__(128) float sm[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + L::SZ);
    const int z0 = blockIdx.x * QZ, x0 = blockIdx.y * TX;
    if (!load_tile(g, bar, L::BYTES, err, [&] {
            tma2(sm + L::OVX, &mp.m[0], z0 - MZ, x0 - M, bar);
            tma2(sm + L::OVZ, &mp.m[1], z0 - MZ, x0 - M, bar);
            for (int i = 0; i < 3; i++) tma2(sm + L::OT + i * B::IN, &mp.m[2 + i], z0, x0, bar);
            tma2(sm + L::OL, &mp.m[5], z0, x0, bar);
            tma2(sm + L::OM, &mp.m[6], z0, x0, bar);
        }))
        return;
    const int q4 = 4 * (threadIdx.x & 15), z = z0 + q4;
    if (z >= g.NZ) return;
    const float gy = __ldg(g.tab + 2 * g.NX);
    float gzn[4], gzh[4];
    tapers4(g, z, gzn, gzh);
#pragma unroll 1
    for (int r = threadIdx.x >> 4; r < TX; r += QT / 16) {
        const int x = x0 + r;
        if (x >= g.NX) break;
        float wx[2 * MZ + 4], wz[2 * MZ + 4], exx[4] = {}, ezz[4] = {}, gxz[4] = {};
        const float *cx = sm + L::OVX + (r + M) * B::ZC + q4, *cz = sm + L::OVZ + (r + M) * B::ZC + q4;
        win4<MZ>(cx, wx);
        win4<MZ>(cz, wz);
#pragma unroll
        for (int k = 1; k <= M; k++) {
            const float b = w.b[k - 1];
            float xp[4], xm[4], zp[4], zm[4];
            lds4(cx + MZ + (k - 1) * B::ZC, xp);
            lds4(cx + MZ - k * B::ZC, xm);
            lds4(cz + MZ + k * B::ZC, zp);
            lds4(cz + MZ + (1 - k) * B::ZC, zm);
#pragma unroll
            for (int i = 0; i < 4; i++) {
                exx[i] += b * (xp[i] - xm[i]);
                ezz[i] += b * (wz[MZ + i + k - 1] - wz[MZ + i - k]);
                gxz[i] += b * ((wx[MZ + i + k] - wx[MZ + i + 1 - k]) + (zp[i] - zm[i]));
            }
        }
        const float *s0 = sm + L::OM + r * B::PC + q4, *s1 = x + 1 < g.NX ? s0 + B::PC : s0;
        float m0[5], m1[5], l[4], a[4], d[4], e[4];
        lds4(s0, m0);
        m0[4] = s0[4];
        lds4(s1, m1);
        m1[4] = s1[4];
        lds4(sm + L::OL + r * QZ + q4, l);
        lds4(sm + L::OT + r * QZ + q4, a);
        lds4(sm + L::OT + B::IN + r * QZ + q4, d);
        lds4(sm + L::OT + 2 * B::IN + r * QZ + q4, e);
        const float gxn = __ldg(g.tab + 2 * x) * gy, gxh = __ldg(g.tab + 2 * x + 1) * gy;
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const bool last = z + i + 1 >= g.NZ;           // the z + 1 node is clamped to the node itself
            const float mxz = 0.25f * ((m0[i] + (last ? m0[i] : m0[i + 1])) + (m1[i] + (last ? m1[i] : m1[i + 1])));
            const float tr = exx[i] + ezz[i], m2 = 2.f * m0[i], gn = gxn * gzn[i];
            a[i] = gn * (a[i] + c * (l[i] * tr + m2 * exx[i]));
            d[i] = gn * (d[i] + c * (l[i] * tr + m2 * ezz[i]));
            e[i] = gxh * gzh[i] * (e[i] + c * mxz * gxz[i]);
            if (check && !(isfinite(a[i]) && isfinite(d[i]) && isfinite(e[i]))) atomicOr(err, 1);
        }
        const long long q = (long long)x * g.PZ + z;       // beyond an odd NZ: lambda = mu = tau = 0, so zeros
        for (int j = 0; j < inj.n; j++)
            if (inj.x[j] == x && inj.o[j] - (unsigned)z < 4u) {
                const float acc = inject_sum(inj.ptr, inj.tr, inj.w, inj.traces, inj.nt, inj.t, j);
#pragma unroll
                for (int i = 0; i < 4; i++)
                    if (inj.o[j] == (unsigned)(z + i)) {
                        inject_add(a[i], inj.scale, acc);
                        inject_add(d[i], inj.scale, acc);
                    }
            }
        st4(txx, q, a);
        st4(tzz, q, d);
        st4(txz, q, e);
    }
}

// 2D map of a [NX][NZ] field, box (bz, bx)
bool map2_of(prop_s *P, const float *base, int bz, int bx, CUtensorMap *out)
{
    const auto key = std::make_tuple((const void *)base, bz, bx);
    auto it = P->tmaps.find(key);
    if (it == P->tmaps.end()) {
        EncodeTiled fn = encode_fn();
        CUtensorMap m;
        const cuuint64_t dims[2] = {(cuuint64_t)P->g.NZ, (cuuint64_t)P->g.NX}, stride[1] = {(cuuint64_t)P->g.PZ * 4};
        const cuuint32_t box[2] = {(cuuint32_t)bz, (cuuint32_t)bx}, es[2] = {1, 1};
        if (!fn || fn(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, (void *)base, dims, stride, box, es,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
        it = P->tmaps.emplace(key, m).first;
    }
    *out = it->second;
    return true;
}

template <int M, int TX>
int launch_tma(prop_s *P, float *const *S, float dt_sign)
{
    using B = Box2<M, TX>;
    const GridDev &g = P->g;
    Maps2 mv, mt;
    const bool ok = map2_of(P, S[2], QZ, B::R, &mv.m[0]) && map2_of(P, S[4], B::ZC, B::R, &mv.m[1]) &&
                    map2_of(P, S[3], B::ZC, TX, &mv.m[2]) && map2_of(P, S[0], QZ, TX, &mv.m[3]) &&
                    map2_of(P, S[1], QZ, TX, &mv.m[4]) && map2_of(P, P->bu, B::PC, B::PR, &mv.m[5]) &&
                    map2_of(P, S[0], B::ZC, B::R, &mt.m[0]) && map2_of(P, S[1], B::ZC, B::R, &mt.m[1]) &&
                    map2_of(P, S[2], QZ, TX, &mt.m[2]) && map2_of(P, S[3], QZ, TX, &mt.m[3]) &&
                    map2_of(P, S[4], QZ, TX, &mt.m[4]) && map2_of(P, P->lam, QZ, TX, &mt.m[5]) &&
                    map2_of(P, P->mu, B::PC, B::PR, &mt.m[6]);
    if (!ok) return wp_fail(P, PROP_ECUDA, "cuTensorMapEncodeTiled failed");
    const size_t sv = LV2<M, TX>::SZ * sizeof(float) + 64, st = LT2<M, TX>::SZ * sizeof(float) + 64;
    static const bool attr = set_smem(el2_vpass_tma<M, TX>, sv) && set_smem(el2_tpass_tma<M, TX>, st);
    (void)attr;
    const dim3 blk(QT), grd((g.NZ + QZ - 1) / QZ, (g.NX + TX - 1) / TX);
    const float c = dt_sign * g.dt * g.ih;
    const RecDev rec = P->rec;
    launch_pass(el2_vpass_tma<M, TX>, dim3(grd.x, grd.y, 1 + receiver_layers(rec, grd, blk)), blk, sv, P->stream, g,
                P->w, S[0], S[1], mv, c, rec, P->flag);
    launch_pass(el2_tpass_tma<M, TX>, grd, blk, st, P->stream, g, P->w, S[2], S[3], S[4], mt, c, P->inj,
                P->d.check_nan, P->flag);
    P->kern_launches += 2;
    WP_CK(P, cudaGetLastError());
    return PROP_OK;
}
// 32 rows per tile where they make a tile for every SM, else 16
template <int M>
int launch_any(prop_s *P, float *const *S, float dt_sign)
{
    const GridDev &g = P->g;
    const long long tiles = (long long)((g.NZ + QZ - 1) / QZ) * ((g.NX + 31) / 32);
    return tiles >= P->sms ? launch_tma<M, 32>(P, S, dt_sign) : launch_tma<M, 16>(P, S, dt_sign);
}

template <int M>
int launch(prop_s *P, float *const *S, float dt_sign)
{
    const GridDev &g = P->g;
    dim3 blk(TZ, BXR), grd((g.NZ + TZ - 1) / TZ, (g.NX + TXR - 1) / TXR);
    const float c = dt_sign * g.dt * g.ih;
    el2_vpass<M><<<grd, blk, 0, P->stream>>>(g, P->w, S[0], S[1], S[2], S[3], S[4], P->bu, c);
    el2_tpass<M><<<grd, blk, 0, P->stream>>>(g, P->w, S[0], S[1], S[2], S[3], S[4], P->lam, P->mu, c, P->flag,
                                             P->d.check_nan);
    P->kern_launches += 2;
    WP_CK(P, cudaGetLastError());
    return PROP_OK;
}

}  // namespace

// one 2D elastic step of S = (vx, vz, txx, tzz, txz) in place; dt_sign = -1:
// the transposed step in the adjoint-modelling variables
int el2_launch(prop_s *P, float *const *S, float dt_sign)
{
    prof_begin(P, dt_sign > 0 ? 2 : 5);
    int rc;
    if (tma_usable(P)) {
        switch (P->M) {
        case 2: rc = launch_any<2>(P, S, dt_sign); break;
        case 4: rc = launch_any<4>(P, S, dt_sign); break;
        case 6: rc = launch_any<6>(P, S, dt_sign); break;
        case 8: rc = launch_any<8>(P, S, dt_sign); break;
        default: return wp_fail(P, PROP_EINVAL, "unsupported space order");
        }
        prof_end(P, dt_sign > 0 ? 2 : 5);
        return rc;
    }
    switch (P->M) {
    case 2: rc = launch<2>(P, S, dt_sign); break;
    case 4: rc = launch<4>(P, S, dt_sign); break;
    case 6: rc = launch<6>(P, S, dt_sign); break;
    case 8: rc = launch<8>(P, S, dt_sign); break;
    default: return wp_fail(P, PROP_EINVAL, "unsupported space order");
    }
    prof_end(P, dt_sign > 0 ? 2 : 5);
    return rc;
}
