// tlb_kernels.cuh -- kernels and launchers of the ternary ELBM step, templated
// on the dimension D (D2Q9 / D3Q27).  Instantiated once per lattice.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "tlb_device.cuh"

namespace tlb {

// ---- g storage: FP32 [Q][N], or mixed: the rest population g_0 in FP32
// (N floats) followed by the moving populations in FP16, scaled by g_scale
// ([Q-1][N] halves).  g_0 carries phi; the moving ones are small. ----
template <typename GT>
struct GIO;
template <>
struct GIO<float> {
    static __device__ __forceinline__ float ld(const void *p, int i, long long n, const DevParams &q)
    {
        return ((const float *)p)[(long long)i * q.N + n];
    }
    static __device__ __forceinline__ void st(void *p, int i, long long n, float v, const DevParams &q)
    {
        ((float *)p)[(long long)i * q.N + n] = v;
    }
};
template <>
struct GIO<__half> {
    static __device__ __forceinline__ float ld(const void *p, int i, long long n, const DevParams &q)
    {
        if (i == 0) return ((const float *)p)[n];
        const __half *h = (const __half *)((const char *)p + 4 * q.N);
        return __half2float(h[(long long)(i - 1) * q.N + n]) * q.g_unscale;
    }
    static __device__ __forceinline__ void st(void *p, int i, long long n, float v, const DevParams &q)
    {
        if (i == 0) {
            ((float *)p)[n] = v;
            return;
        }
        __half *h = (__half *)((char *)p + 4 * q.N);
        h[(long long)(i - 1) * q.N + n] = __float2half_rn(v * q.g_scale);
    }
};

template <int D>
struct Tile;
template <>
struct Tile<2> {
    static constexpr int X = 32, Y = 8, Z = 1;
};
// 16 x 4 x 4 and not 8 x 8 x 4: rows of 64 bytes halve the lines that a warp's
// loads and stores touch, and the half-warps of the tensor stage lie in one row,
// without bank conflicts; that outweighs 8 % more nodes in the halo (192 x 192 x
// 128: 854 -> 775 us a step; 32 x 4 x 2 with 36 % more: 798; 16 x 8 x 2: 788).
template <>
struct Tile<3> {
    static constexpr int X = 16, Y = 4, Z = 4;
};

// periodic wrap of a coordinate at most one period outside [0, n)
__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// (node indices fit in 32 bits: a lattice holds at most 2^31 - 1 nodes)
__device__ __forceinline__ int node_near(const DevParams &p, int x, int y, int z)
{
    return (int)chk_node(wrap1(x, p.nx) + p.nx * (wrap1(y, p.ny) + p.ny * wrap1(z, p.nz)), p);
}

// Programmatic dependent launch: a stepping kernel lets the next one be
// scheduled at once and waits for its predecessor's results before reading.
// What a predecessor writes -- populations, rho, phi -- changes while the waiting
// grid is alive, so it is read with ordinary loads: read-only ones (__ldg, const
// __restrict__) promise data that does not, and neither the compiler nor the cache
// need keep them behind the wait.  They are for the flags and tables, which
// change between launches alone.  The time is the same: D2Q9 2048 x 2048 171.2 us
// a step with read-only loads, 170.5 with ordinary ones, D3Q27 192 x 192 x 128 746
// and 745.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// Asynchronous global -> shared copies (sm_80+ cp.async): the node's own
// populations are requested before the tile stages and consumed after them.
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Tensor-memory-accelerator copies (cp.async.bulk.tensor): one thread moves a
// tile's box of every direction into shared memory; completion is counted in
// bytes on an mbarrier that the consumers wait on.
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    // make the initialised barrier visible to the tensor-copy (async) proxy
    asm volatile("fence.mbarrier_init.release.cluster;\n"
                 "fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void tma_load_3d(void *dst, const void *tmap, int c0, int c1, int c2, unsigned long long *bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4}], [%5];\n"
                 ::"r"(smem_u32(dst)), "l"(tmap), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tma_load_4d(void *dst, const void *tmap, int c0, int c1, int c2, int c3,
                                            unsigned long long *bar)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4, %5}], [%6];\n"
                 ::"r"(smem_u32(dst)), "l"(tmap), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity)
{
    unsigned done;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                 " selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return done != 0;
}
// waits for the barrier's phase `parity` to complete; false after `ns` nanoseconds
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long *bar, unsigned parity, unsigned long long ns)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_ns() - t0 > ns) return false;
    return true;
}

// dynamic shared memory of the stepping kernel: f (and FP32 g) of the tile's own nodes
template <int D, typename GT>
__host__ __device__ constexpr int stage_bytes()
{
    // f: Q floats; g: Q floats, or g_0 as a float plus Q-1 halves; D3Q27: 128
    // bytes more, to start the area on a 128-byte boundary (tensor copies)
    return Tile<D>::X * Tile<D>::Y * Tile<D>::Z *
               (Lat<D>::Q * 4 + (sizeof(GT) == 4 ? Lat<D>::Q * 4 : 4 + (Lat<D>::Q - 1) * 2)) +
           (D == 3 ? 128 : 0);
}

// ---------------------------------------------------------------------------
// moments: rho = 1 + sum_i (f_i - w_i), phi = sum_i g_i at fluid nodes
// ---------------------------------------------------------------------------
// (32-bit offsets took 2.6 % off the D3Q27 192 x 192 x 128 step)
template <int D, typename GT, bool BIG = D == 2>
__device__ __forceinline__ float2 pop_moments(const DevParams &p, const float *f, const void *g, long long n)
{
    constexpr int Q = Lat<D>::Q;
    float r = 0.f, ph = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        r += *elem<BIG>(f + (long long)i * p.N, (int)n);
        if (sizeof(GT) == 4 || i == 0) ph += *elem<BIG>((const float *)g + (long long)i * p.N, (int)n);
        else ph += GIO<GT>::ld(g, i, n, p);
    }
    return make_float2(1.0f + r, ph);
}

template <int D, typename GT>
__device__ __forceinline__ void moments_node(const DevParams &p, const float *f, const void *g,
                                             const uint8_t *__restrict__ type, float *rho, float *phi, long long n)
{
    constexpr int Q = Lat<D>::Q;
    if (type[n] & TLB_SOLID) {
        if (!(type[n] & TLB_GHOST)) { rho[n] = 0.f; phi[n] = 0.f; }
        return;
    }
    const float2 m = pop_moments<D, GT>(p, f, g, n);
    rho[n] = m.x;
    phi[n] = m.y;
}

template <int D, typename GT>
__global__ void __launch_bounds__(256) moments_kernel(DevParams p, const float *__restrict__ f, const void *g,
                                                      const uint8_t *__restrict__ type, float *rho, float *phi)
{
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < p.N; n += (long long)gridDim.x * blockDim.x)
        moments_node<D, GT>(p, f, g, type, rho, phi, n);
}

template <int D, typename GT>
__global__ void __launch_bounds__(256) moments_batch_kernel(const BatchEntry *__restrict__ E, const int4 *__restrict__ tiles)
{
    pdl_trigger();
    pdl_wait();
    int4 t = tiles[blockIdx.x];
    const BatchEntry &e = E[t.x];
    // the moments need no neighbourhood: the k-th tile of a lattice (in the
    // table's x-fastest order) takes its nodes k*NT .. k*NT + NT - 1 in
    // memory order, so that a warp reads whole 128-byte lines; a lattice has
    // at least N / NT tiles, so every node is covered once
    constexpr int TX = Tile<D>::X, TY = Tile<D>::Y, TZ = Tile<D>::Z, NT = TX * TY * TZ;
    const long long ntx = (e.p.nx + TX - 1) / TX, nty = (e.p.ny + TY - 1) / TY;
    const long long k = t.y / TX + ntx * (t.z / TY + nty * (t.w / TZ));
    const long long n = k * NT + threadIdx.x;
    if (n >= e.p.N) return;
    moments_node<D, GT>(e.p, e.f_in, e.g_in, e.type, const_cast<float *>(e.rho), const_cast<float *>(e.phi), n);
}

// the same for one lattice, its entry by value.  Bound by memory: 216 of 225
// bytes a node are read once (1.18 M nodes, cold: 43 us, 6.2 TB/s); four nodes a
// thread in 16-byte loads gained nothing.
template <int D, typename GT>
__global__ void __launch_bounds__(256) moments_step_kernel(const __grid_constant__ BatchEntry e)
{
    pdl_trigger();
    const long long n = blockIdx.x * 256LL + threadIdx.x;
    pdl_wait();
    if (n < e.p.N)
        moments_node<D, GT>(e.p, e.f_in, e.g_in, e.type, const_cast<float *>(e.rho), const_cast<float *>(e.phi), n);
}

// ---------------------------------------------------------------------------
// ghost layer (Sec. IV): average over fluid-facing axis directions; ghosts
// with only diagonal fluid neighbours take the mean of those neighbours.
// ---------------------------------------------------------------------------
template <int D, class A>
__device__ void ghost_value(const DevParams &p, const A &acc, int x, int y, int z, float &gr_out, float &gp_out)
{
    constexpr int Q = Lat<D>::Q;
    float sr = 0.f, sp = 0.f;
    int cnt = 0;
    // one copy of the (large) axis code, not one per direction; scalar
    // coordinates (no array indexed by the run-time axis)
#pragma unroll 1
    for (int d = 0; d < 2 * D; ++d) {
        const int a = d >> 1, s = (d & 1) ? 1 : -1;
        const int qx = x + (a == 0 ? s : 0), qy = y + (a == 1 ? s : 0), qz = z + (a == 2 ? s : 0);
        float2 m1;
        if (!acc.get(qx, qy, qz, m1)) continue;
        float gr, gp;
        ghost_axis<D>(p, acc, qx, qy, qz, a, m1, gr, gp);
        sr += gr;
        sp += gp;
        ++cnt;
    }
    if (cnt == 0) {
#pragma unroll 1
        for (int i = 1; i < Q; ++i) {
            float2 m;
            if (!acc.get(x + cc<D>(i, 0), y + cc<D>(i, 1), z + cc<D>(i, 2), m)) continue;
            sr += m.x;
            sp += m.y;
            ++cnt;
        }
    }
    gr_out = cnt > 0 ? sr / (float)cnt : 0.f;
    gp_out = cnt > 0 ? sp / (float)cnt : 0.f;
}

template <int D>
__device__ void ghost_node(const DevParams &p, const uint8_t *__restrict__ type, float *rho, float *phi, long long n)
{
    float gr, gp;
    const int x = (int)(n % p.nx), y = (int)((n / p.nx) % p.ny), z = (int)(n / ((long long)p.nx * p.ny));
    ghost_value<D>(p, NodesGlobal{p, type, rho, phi}, x, y, z, gr, gp);
    rho[n] = gr;
    phi[n] = gp;
}

template <int D>
__global__ void __launch_bounds__(128) ghost_kernel(DevParams p, const uint8_t *__restrict__ type, float *rho, float *phi,
                                                    const int *__restrict__ ghosts, int nghost)
{
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nghost) return;
    ghost_node<D>(p, type, rho, phi, ghosts[k]);
}

// index into the Q-tensor components stored per node: 2D {xx, yy, xy}, 3D {xx, yy, zz, xy, xz, yz}
template <int D>
__device__ __forceinline__ int qcomp(int a, int b)
{
    if (a == b) return a;
    int lo = a < b ? a : b, hi = a < b ? b : a;
    if (D == 2) return 2;
    return lo == 0 ? (hi == 1 ? 3 : 4) : 5;
}

// Flag test and moments of a node outside the tile region: from the flag
// array and the node's populations.  Out of line, so that the several call
// sites of the ghost-layer code share one copy of the index arithmetic.
template <int D, typename GT>
__device__ __noinline__ bool node_far(const DevParams &p, const uint8_t *__restrict__ type, const float *f, const void *g,
                                      int x, int y, int z, float2 &m)
{
    const long long n = node_of(p, x, y, z);
    if (type[n] & TLB_SOLID) return false;
    m = pop_moments<D, GT>(p, f, g, n);
    return true;
}

}  // namespace tlb
#include "tlb_step.cuh"
namespace tlb {

// ---------------------------------------------------------------------------
// Passes over given or current fields that are not steps (one CTA = one tile
// of TX x TY x TZ nodes, rho and phi from the moment arrays, the step's functions
// for all that a step computes too): MODE_INIT writes the populations of rho, phi
// and u_init; MODE_AUX the auxiliary fields.
// ---------------------------------------------------------------------------
template <int D, typename GT, int MODE>
__global__ void __launch_bounds__(256) field_kernel(const __grid_constant__ BatchEntry e, const float *__restrict__ u_init,
                                                    AuxOut aux)
{
    using S = StepShared<D>;
    constexpr int Q = Lat<D>::Q, NPOS = Lat<D>::NPOS;
    constexpr int TX = S::TX, TY = S::TY, RY = S::RY, SX = S::SX, SY = S::SY, HZ = D == 3 ? 1 : 0;
    __shared__ S sh;
    const DevParams &p = e.p;
    const int tid = threadIdx.x;
    int x0, y0, z0;
    tile_origin<D>(p, blockIdx.x, x0, y0, z0);
    gather_moments<D, true>(e, x0, y0, z0, sh, [] {});
    tensor_stage<D, true>(p, x0, y0, z0, sh);
    __syncthreads();

    // one node per thread
    const int tx = tid % TX, ty = (tid / TX) % TY, tz = tid / (TX * TY);
    const int x = x0 + tx, y = y0 + ty, z = z0 + tz;
    if (x >= p.nx || y >= p.ny || z >= p.nz) return;
    const int sc = (tx + 1) + SX * ((ty + 1) + SY * (tz + HZ));
    const uint8_t tc = sh.type[sc];
    if (tc & TLB_SOLID) return;
    const int n = x + p.nx * (y + p.ny * z);
    const float2 *c = sh.rp + (tx + 2) + S::PX * ((ty + 2) + RY * (tz + 2 * HZ));
    const float r = c->x, ph = c->y;
    float F[D];
    const float mup = node_force<D, true>(p, sh, sc, tc, r, ph, F);
    if constexpr (MODE == MODE_AUX) {
        const Stress<D> s = node_stress<D, S::PX, RY>(p, c);
        if (aux.p0) aux.p0[n] = s.p0;
        if (aux.mur) aux.mur[n] = fmaf(-p.krp, s.lap.y, fmaf(-p.krr, s.lap.x, bulk_mur(p, r, ph)));
        if (aux.mup) aux.mup[n] = s.mup;
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (aux.F[a]) aux.F[a][n] = a < D ? F[a < D ? a : 0] : 0.f;
#pragma unroll
        for (int j = 0; j < 6; ++j)        // xx yy zz xy xz yz
            if (aux.P[j]) aux.P[j][n] = D == 3 ? (j < 3 ? s.iso + s.d[j] : s.o[j - 3])
                                               : j < 2 ? s.iso + s.d[j] : j == 2 ? s.iso : j == 3 ? s.o[0] : 0.f;
    } else {
        // f = f^eq(rho, v - F/(2 rho)), g = g^eq(phi, v, mu_phi) at the node itself
        const float inv_r = 1.0f / r;
        float v[D], f0[D], fp[D], fm[D], rest = r;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            v[a] = u_init ? u_init[(long long)a * p.N + n] : 0.f;
            const float u = fmaf(-0.5f * F[a], inv_r, v[a]);
            const Fac2 t = eq_factors2<D>(f2(u, u));
            f0[a] = t.f0.x;
            fp[a] = t.fp.x;
            fm[a] = t.fm.x;
            rest *= f0[a];
        }
        float2 eq[NPOS];
        equilibria<D>(r, f0, fp, fm, eq);
        const GEq ge = g_eq<D>(p, ph, mup, v);
        float2 gsum = f2(0.f, 0.f);
        e.f_out[n] = rest - wt<D>(0);
#pragma unroll
        for (int k = 0; k < NPOS; ++k) {
            const float w = wt<D>(2 * k + 1);
            const float2 gk = ge.pair(w, along<D>(k, v));
            gsum = add2(gsum, gk);
            e.f_out[(long long)(2 * k + 1) * p.N + n] = eq[k].x - w;
            e.f_out[(long long)(2 * k + 2) * p.N + n] = eq[k].y - w;
            GIO<GT>::st(e.g_out, 2 * k + 1, n, gk.x, p);
            GIO<GT>::st(e.g_out, 2 * k + 2, n, gk.y, p);
        }
        GIO<GT>::st(e.g_out, 0, n, ph - (gsum.x + gsum.y), p);
    }
}

// ---------------------------------------------------------------------------
// fields: bare velocity u = sum f c / rho at fluid nodes
// ---------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(256) fields_kernel(DevParams p, const float *__restrict__ f, const float *__restrict__ rho,
                                                     const uint8_t *__restrict__ type, float *u)
{
    constexpr int Q = Lat<D>::Q;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < p.N; n += (long long)gridDim.x * blockDim.x) {
        float j[3] = {0.f, 0.f, 0.f};
        bool solid = type[n] & TLB_SOLID;
        if (!solid) {
#pragma unroll
            for (int i = 1; i < Q; ++i) {
                float fi = f[(long long)i * p.N + n];
#pragma unroll
                for (int a = 0; a < D; ++a)
                    if (cc<D>(i, a) != 0) j[a] += (float)cc<D>(i, a) * fi;
            }
        }
        float ir = solid ? 0.f : 1.0f / rho[n];
#pragma unroll
        for (int a = 0; a < D; ++a) u[(long long)a * p.N + n] = j[a] * ir;
    }
}

// ---------------------------------------------------------------------------
// FP64 diagnostics: per-block partial sums (fixed order), then one block.
// ---------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(256) diag_kernel(DevParams p, const float *__restrict__ f, const float *__restrict__ rho,
                                                   const float *__restrict__ phi, const uint8_t *__restrict__ type,
                                                   double *partials)
{
    constexpr int Q = Lat<D>::Q;
    double s[6] = {0, 0, 0, 0, 0, 0};
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < p.N; n += (long long)gridDim.x * blockDim.x) {
        if (type[n] & TLB_SOLID) continue;
        double r = rho[n], ph = phi[n];
        double C1 = (r - (double)p.rho_l) / ((double)p.rho_g - (double)p.rho_l);
        s[0] += r;
        s[1] += ph;
        s[2] += C1;
        s[3] += 0.5 * (1.0 + ph / (double)p.chi - C1);
        s[4] += 0.5 * (1.0 - ph / (double)p.chi - C1);
        double j[3] = {0, 0, 0};
        for (int i = 1; i < Q; ++i) {
            double fi = f[(long long)i * p.N + n];
            for (int a = 0; a < D; ++a) j[a] += cc<D>(i, a) * fi;
        }
        double j2 = 0;
        for (int a = 0; a < D; ++a) j2 += j[a] * j[a];
        s[5] += 0.5 * j2 / r;
    }
    __shared__ double red[6][8];
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int k = 0; k < 6; ++k) {
        double v = s[k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red[k][wid] = v;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        double v = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[threadIdx.x][w];
        partials[(long long)blockIdx.x * 6 + threadIdx.x] = v;
    }
}

template <int D>
__global__ void diag_final_kernel(const double *partials, int nblocks, double *out)
{
    if (threadIdx.x < 6) {
        double v = 0;
        for (int b = 0; b < nblocks; ++b) v += partials[(long long)b * 6 + threadIdx.x];
        out[threadIdx.x] = v;
    }
}

// populations <-> FP64 host-order buffers (dir 0: device -> double, 1: double -> device)
template <int D, typename GT>
__global__ void convert_kernel(DevParams p, float *f, void *g, double *fb, double *gb, int dir)
{
    constexpr int Q = Lat<D>::Q;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < p.N; n += (long long)gridDim.x * blockDim.x) {
        for (int i = 0; i < Q; ++i) {
            long long k = (long long)i * p.N + n;
            if (dir == 0) {
                fb[k] = (double)f[k] + (double)wt<D>(i);
                gb[k] = (double)GIO<GT>::ld(g, i, n, p);
            } else {
                f[k] = (float)(fb[k] - (double)wt<D>(i));
                GIO<GT>::st(g, i, n, (float)gb[k], p);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
inline int grid_for(long long N, int threads)
{
    long long b = (N + threads - 1) / threads;
    long long cap = 152LL * 16;
    return (int)(b < cap ? (b < 1 ? 1 : b) : cap);
}

template <int D>
int Launch<D>::Q() { return Lat<D>::Q; }

template <int D>
int Launch<D>::tile_dims(int a) { return a == 0 ? Tile<D>::X : a == 1 ? Tile<D>::Y : Tile<D>::Z; }

template <int D>
void Launch<D>::moments(const DevParams &p, const DevState &s, cudaStream_t st)
{
    if (p.g_fp16)
        moments_kernel<D, __half><<<grid_for(p.N, 256), 256, 0, st>>>(p, s.f[s.cur], s.g[s.cur], s.type, s.rho, s.phi);
    else
        moments_kernel<D, float><<<grid_for(p.N, 256), 256, 0, st>>>(p, s.f[s.cur], s.g[s.cur], s.type, s.rho, s.phi);
}

template <int D>
void Launch<D>::ghosts(const DevParams &p, const DevState &s, cudaStream_t st)
{
    if (s.nghost > 0)
        ghost_kernel<D><<<(s.nghost + 127) / 128, 128, 0, st>>>(p, s.type, s.rho, s.phi, s.ghosts, s.nghost);
}

template <int D>
void Launch<D>::field_pass(const DevParams &p, const DevState &s, int mode, const float *u_init, AuxOut aux,
                           cudaStream_t st)
{
    // one dimension: the others end at 65535, which a lattice of many tile rows passes
    const int grid = tiles(p), block = Tile<D>::X * Tile<D>::Y * Tile<D>::Z;
    BatchEntry e = {};
    e.p = p;
    e.f_out = s.f[s.cur];
    e.g_out = s.g[s.cur];
    e.rho = s.rho;
    e.phi = s.phi;
    e.type = s.type;
    if (mode == MODE_AUX) field_kernel<D, float, MODE_AUX><<<grid, block, 0, st>>>(e, nullptr, aux);
    else if (p.g_fp16) field_kernel<D, __half, MODE_INIT><<<grid, block, 0, st>>>(e, u_init, aux);
    else field_kernel<D, float, MODE_INIT><<<grid, block, 0, st>>>(e, u_init, aux);
}

template <int D>
void Launch<D>::fields(const DevParams &p, const DevState &s, float *u_out, cudaStream_t st)
{
    fields_kernel<D><<<grid_for(p.N, 256), 256, 0, st>>>(p, s.f[s.cur], s.rho, s.type, u_out);
}

template <int D>
int Launch<D>::diag_blocks(const DevParams &p) { return grid_for(p.N, 256) < 1024 ? grid_for(p.N, 256) : 1024; }

template <int D>
void Launch<D>::diagnostics(const DevParams &p, const DevState &s, double *partials, int nblocks, double *out,
                            cudaStream_t st)
{
    diag_kernel<D><<<nblocks, 256, 0, st>>>(p, s.f[s.cur], s.rho, s.phi, s.type, partials);
    diag_final_kernel<D><<<1, 32, 0, st>>>(partials, nblocks, out);
}

template <int D>
void Launch<D>::convert_pop(const DevParams &p, const DevState &s, int dir, double *fbuf, double *gbuf, cudaStream_t st)
{
    if (p.g_fp16)
        convert_kernel<D, __half><<<grid_for(p.N, 256), 256, 0, st>>>(p, s.f[s.cur], s.g[s.cur], fbuf, gbuf, dir);
    else
        convert_kernel<D, float><<<grid_for(p.N, 256), 256, 0, st>>>(p, s.f[s.cur], s.g[s.cur], fbuf, gbuf, dir);
}

// launch with programmatic stream serialization (the kernel's griddepcontrol.wait
// orders it after its predecessor's memory operations)
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t st, bool pdl,
                       const Args &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = pdl;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int D>
unsigned Launch<D>::bounds_errors()
{
#ifdef TLB_BOUNDS_CHECK
    unsigned v = 0, zero = 0;
    cudaMemcpyFromSymbol(&v, g_bounds_error, sizeof(v));
    cudaMemcpyToSymbol(g_bounds_error, &zero, sizeof(zero));
    return v;
#else
    return 0;
#endif
}

template <int D>
void Launch<D>::moments_batch(const BatchEntry *entries, const int4 *tiles, int ntiles, int g_fp16, cudaStream_t st)
{
    if (ntiles <= 0) return;
    const int nt = Tile<D>::X * Tile<D>::Y * Tile<D>::Z;
    if (g_fp16) launch_pdl(moments_batch_kernel<D, __half>, ntiles, nt, 0, st, true, entries, tiles);
    else launch_pdl(moments_batch_kernel<D, float>, ntiles, nt, 0, st, true, entries, tiles);
}

// per kernel, once per device on the first launch there: the dynamic
// shared-memory opt-ins; returns the device's SM count (D2Q9: the one-wave bound),
// 0 if an opt-in failed, whose launch then fails
template <int D, typename GT>
static int step_setup()
{
    static std::atomic<int> known[64];
    int dev = 0;
    cudaGetDevice(&dev);
    return once_per_device(known, dev, [dev] {
        constexpr int b = stage_bytes<D, GT>();
        bool ok = true;
        const auto opt = [&ok](auto *kernel) {
            ok &= cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, b) == cudaSuccess;
        };
        if constexpr (D == 2) {
            opt(step_batch_kernel<D, GT, 3, false>);
            opt(step_batch_kernel<D, GT, 4, false>);
            opt(step_batch_kernel<D, GT, 4, true>);
            opt(step_kernel<D, GT, 3, false>);
            opt(step_kernel<D, GT, 4, false>);
            opt(step_kernel<D, GT, 4, true>);
        } else {
            opt(step_batch_kernel<D, GT, 2, false>);
            opt(step_kernel<D, GT, 2, false>);
        }
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return ok ? n : 0;
    });
}

template <int D, typename GT>
static void launch_step_batch(const BatchEntry *entries, const int4 *tiles, int ntiles, bool big, cudaStream_t st, int variant)
{
    constexpr size_t bytes = stage_bytes<D, GT>();
    constexpr int nt = Tile<D>::X * Tile<D>::Y * Tile<D>::Z;
    const int nsm = step_setup<D, GT>();
    if constexpr (D == 2) {
        const bool four = variant < 0 ? ntiles > 3 * nsm : variant == 1;
        if (big) launch_pdl(step_batch_kernel<D, GT, 4, true>, ntiles, nt, bytes, st, true, entries, tiles);
        else if (four) launch_pdl(step_batch_kernel<D, GT, 4, false>, ntiles, nt, bytes, st, true, entries, tiles);
        else launch_pdl(step_batch_kernel<D, GT, 3, false>, ntiles, nt, bytes, st, true, entries, tiles);
    } else {
        launch_pdl(step_batch_kernel<D, GT, 2, false>, ntiles, nt, bytes, st, true, entries, tiles);
    }
}

template <int D>
void Launch<D>::step_batch(const BatchEntry *entries, const int4 *tiles, int ntiles, int g_fp16, bool big,
                           cudaStream_t st, int variant)
{
    if (ntiles <= 0) return;
    if (g_fp16) launch_step_batch<D, __half>(entries, tiles, ntiles, big, st, variant);
    else launch_step_batch<D, float>(entries, tiles, ntiles, big, st, variant);
}

template <int D>
int Launch<D>::tiles(const DevParams &p)
{
    const long long t = (long long)((p.nx + Tile<D>::X - 1) / Tile<D>::X) * ((p.ny + Tile<D>::Y - 1) / Tile<D>::Y) *
                        ((p.nz + Tile<D>::Z - 1) / Tile<D>::Z);
    return (int)t;
}

template <int D>
void Launch<D>::wall_tiles(const DevParams &p, const uint8_t *type, uint8_t *out, cudaStream_t st)
{
    wall_tiles_kernel<D><<<tiles(p), 128, 0, st>>>(p, type, out);
}

template <int D>
cudaError_t Launch<D>::moments_step(const BatchEntry &e, cudaStream_t st, bool pdl)
{
    const int grid = (int)((e.p.N + 255) / 256);
    if (e.p.g_fp16) return launch_pdl(moments_step_kernel<D, __half>, grid, 256, 0, st, pdl, e);
    return launch_pdl(moments_step_kernel<D, float>, grid, 256, 0, st, pdl, e);
}

template <int D, typename GT>
static cudaError_t launch_step(const BatchEntry &e, cudaStream_t st, bool pdl)
{
    constexpr size_t bytes = stage_bytes<D, GT>();
    constexpr int nt = Tile<D>::X * Tile<D>::Y * Tile<D>::Z;
    const int nsm = step_setup<D, GT>(), ntiles = Launch<D>::tiles(e.p);
    if constexpr (D == 2) {
        if (big_lattice(e.p.N)) return launch_pdl(step_kernel<D, GT, 4, true>, ntiles, nt, bytes, st, pdl, e);
        if (ntiles > 3 * nsm) return launch_pdl(step_kernel<D, GT, 4, false>, ntiles, nt, bytes, st, pdl, e);
        return launch_pdl(step_kernel<D, GT, 3, false>, ntiles, nt, bytes, st, pdl, e);
    } else {
        return launch_pdl(step_kernel<D, GT, 2, false>, ntiles, nt, bytes, st, pdl, e);
    }
}

template <int D>
cudaError_t Launch<D>::step(const BatchEntry &e, cudaStream_t st, bool pdl)
{
    if (e.p.g_fp16) return launch_step<D, __half>(e, st, pdl);
    return launch_step<D, float>(e, st, pdl);
}

}  // namespace tlb
