// tlb_step.cuh -- the stepping kernel of the ternary ELBM (one CTA = one tile
// of TX x TY x TZ nodes), templated on the dimension D.
//
// What bounds it: no one unit on large lattices.  The populations are read and
// written once (16Q bytes a node), and the arithmetic of a node is large next to
// that: stencils of rho, phi and of the pressure tensor, two product equilibria,
// the entropic root, two relaxations.  D2Q9 issues in 0.6 of the cycles at 30
// warps an SM (waits for loads, the shared-memory queue and the packed FP32 pipe),
// D3Q27 in 0.47 (captured with cold caches; 0.55 over the time of a step) at the 14
// that its registers and shared memory admit, where waits for instructions, for
// loads, at barriers and for dependent results share the rest.  On lattices of one
// wave a step is a tile's chain of stages, run once: instruction fetch is its largest
// stall (5 warps an issue of 1024 x 64 with cold caches, loads 2).
// So the arithmetic is written for few instructions:
//   - opposite directions +c, -c form a pair held in a float2 and handled by
//     the packed FP32 instructions (two results per issue);
//   - (rho, phi) form another such pair in the stencils, which are applied one
//     axis after another in registers (weights are products over the axes);
//   - p_0 comes from the pressure of the equation of state directly (no
//     logarithm, and no cancelling rho Psi' - Psi);
//   - tiles with no solid node within two links (`walls` false: most tiles of
//     a lattice) take a copy of the code without flags, ghost layer, wall rules
//     and bounce-back;
//   - a lattice stepped alone passes its entry by value, so that parameters
//     and array bases are constant-bank operands.
// Warp instructions x 32 a node: D2Q9 2048 x 2048 929, D3Q27 2563 (1506 and 3876
// with directions one by one, flags in every tile and the entry in shared memory).
// Kernel time: D2Q9 4096 x 4096 0.622 ms, 58 % of the measured 6.78 TB/s; D3Q27 192 x
// 192 x 128 0.551 ms, 56 %.
#pragma once
#include "tlb_device.cuh"

namespace tlb {

// ---- packed FP32 pairs ----
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b, the same bits either way: as a subtraction in D2Q9, as a - 1*b in
// D3Q27 (2 % off the 192 x 192 x 128 step, 1 % onto the D2Q9 2048 x 2048 one)
template <int D>
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    if (D == 3) return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
    float2 r;
    asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
        " sub.rn.ftz.f32x2 c, a, b;\n mov.b64 {%0, %1}, c;\n}\n"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

// weight class of the pair k: 0 faces, 1 edges, 2 corners
template <int D>
__host__ __device__ constexpr int pair_class(int k)
{
    int n = 0;
    for (int a = 0; a < D; ++a) n += Lat<D>::pos(k, a) != 0;
    return n - 1;
}

// ---------------------------------------------------------------------------
// Thermodynamics of a node for the step: p_0 and the bulk part of mu_phi.
// p_0 = rho murB + phi mupB - f_B (Eq. bulkpressure) with rho Psi' - Psi
// replaced by the pressure p of the equation of state that Psi comes from:
//   p_0 = (lam1/2) (p + Psi0) + sum_{k=2,3} lam_k s_k (-(C_k - 1/2)(rho/drho +- phi/chi) - s_k/2),
// s_k = C_k (1 - C_k), C_k (C_k - 1/2)(C_k - 1) = -s_k (C_k - 1/2).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float eos_pressure(const DevParams &p, float rho)
{
    if (p.eos == 0) {                        // Carnahan-Starling
        const float e = p.b4 * rho;
        const float r = 1.0f / (1.0f - e);
        const float num = fmaf(e, fmaf(e, 1.0f - e, 1.0f), 1.0f);
        return rho * fmaf(p.RT * num, r * r * r, -(p.a * rho));
    }
    const float br = p.b * rho;
    // no state beyond the pole at b rho = 1, where Psi has no logarithm either: not a
    // number, which the collision reports
    const float rep = br < 1.0f ? p.RT / (1.0f - br) : __int_as_float(0x7fffffff);
    if (p.eos == 1) return rho * fmaf(-p.a, rho, rep);                      // van der Waals
    return rho * (rep - p.aA * rho / fmaf(br, 2.0f - br, 1.0f));            // Peng-Robinson
}

__device__ __forceinline__ float bulk_p0(const DevParams &p, float rho, float phi, float &mupB)
{
    const float C1 = (rho - p.rho_l) * p.inv_rgl;
    const float R = rho * p.inv_drho, a = phi * p.inv_chi;
    const float h = fmaf(-0.5f, C1, 0.5f);
    const float C2 = fmaf(0.5f, a, h), C3 = fmaf(-0.5f, a, h);
    const float s2 = fmaf(-C2, C2, C2), s3 = fmaf(-C3, C3, C3);
    const float m2 = C2 - 0.5f, m3 = C3 - 0.5f;
    const float w2 = p.lam2 * s2, w3 = p.lam3 * s3;
    mupB = fmaf(w3, m3, -(w2 * m2)) * p.inv_chi;
    const float v = fmaf(w2, fmaf(m2, R + a, 0.5f * s2), w3 * fmaf(m3, R - a, 0.5f * s3));
    return fmaf(p.hl1, eos_pressure(p, rho) + p.Psi0, -v);
}

// The bulk part of mu_rho (Eq. bulkchempotrho, the lambda_2 term with the sign of
// the derivative of Eq. BulkEnergy), an auxiliary field that no step needs: the one
// place of the logarithm of Psi, through Psi' as printed for Carnahan-Starling
// (Eq. PsiEOS), and with Psi = rho (C - a rho + RT ln(rho/(1 - b rho))) of van der
// Waals, where Peng-Robinson has - a A/(2 sqrt2 b) ln((b rho + sqrt2 - 1)/(sqrt2 +
// 1 - b rho)) in place of - a rho (a A: p.aA).
__device__ __forceinline__ float bulk_mur(const DevParams &p, float rho, float phi)
{
    const float br = p.b * rho;
    float dpsi;
    if (p.eos == 0) {
        const float q = br - 4.0f;
        dpsi = fmaf(p.RT, 1.0f + logf(rho), fmaf(-2.0f * p.a, rho, p.C)) + 16.0f * p.RT * (br - 12.0f) / (q * q * q);
    } else {
        const float om = 1.0f - br, lg = logf(rho / om);
        if (p.eos == 1) {
            dpsi = fmaf(p.RT, lg, fmaf(-2.0f * p.a, rho, p.C)) + p.RT / om;
        } else {
            const float k = p.aA * (0.35355339f / p.b);      // a A / (2 sqrt2 b)
            const float L = logf((br + 0.41421356f) / (2.41421356f - br));
            dpsi = fmaf(p.RT, lg, fmaf(-k, L, p.C)) + p.RT / om - p.aA * rho / fmaf(br, 2.0f - br, 1.0f);
        }
    }
    const float C1 = (rho - p.rho_l) * p.inv_rgl, a = phi * p.inv_chi;
    const float h = fmaf(-0.5f, C1, 0.5f);
    const float C2 = fmaf(0.5f, a, h), C3 = fmaf(-0.5f, a, h);
    const float g2 = C2 * (C2 - 0.5f) * (C2 - 1.0f), g3 = C3 * (C3 - 0.5f) * (C3 - 1.0f);
    return fmaf(p.hl1, dpsi, fmaf(p.lam2, g2, p.lam3 * g3) * p.inv_drho);
}

// Pressure tensor P = iso I + {d on the diagonal, o = xy, xz, yz off it}, p_0,
// mu_phi and the Laplacians of (rho, phi)
template <int D>
struct Stress {
    float iso, d[D], o[D == 3 ? 3 : 1], p0, mup;
    float2 lap;
};

// The pressure tensor and mu_phi at the node whose (rho, phi) is c[0] in a region
// of row length RX and RY rows per plane.  The stencils (grad Q = 3 sum w_i c_i Q(x + c_i), lap Q =
// 6 sum w_i (Q(x + c_i) - Q(x))) as products of (1, 4, 1)/6 and (-1, 0, 1)/6
// along the axes, on differences to the node itself.
template <int D, int RX, int RY>
__device__ __forceinline__ Stress<D> node_stress(const DevParams &p, const float2 *__restrict__ c)
{
    Stress<D> s;
    const float2 m0 = c[0];
    const float2 four = f2(4.0f, 4.0f);
    float2 g[D], lap;
    if constexpr (D == 3) {
        float2 SS[3], DS[3], ST[3];       // per x plane: smooth y smooth z, diff y smooth z, smooth y diff z
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            float2 S[3], T[3];
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                const int o = (x - 1) + RX * (y - 1);
                const float2 up = sub2<D>(c[o + RX * RY], m0), dn = sub2<D>(c[o - RX * RY], m0);
                S[y] = add2(up, dn);
                if (o != 0) S[y] = fma2(four, sub2<D>(c[o], m0), S[y]);
                T[y] = sub2<D>(up, dn);
            }
            SS[x] = fma2(four, S[1], add2(S[0], S[2]));
            DS[x] = sub2<D>(S[2], S[0]);
            ST[x] = fma2(four, T[1], add2(T[0], T[2]));
        }
        const float2 w = f2(1.0f / 72.0f, 1.0f / 72.0f);
        g[0] = mul2(sub2<D>(SS[2], SS[0]), w);
        g[1] = mul2(fma2(four, DS[1], add2(DS[0], DS[2])), w);
        g[2] = mul2(fma2(four, ST[1], add2(ST[0], ST[2])), w);
        lap = mul2(fma2(four, SS[1], add2(SS[0], SS[2])), f2(1.0f / 36.0f, 1.0f / 36.0f));
    } else {
        float2 S[3], T[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            const float2 up = sub2<D>(c[(x - 1) + RX], m0), dn = sub2<D>(c[(x - 1) - RX], m0);
            S[x] = add2(up, dn);
            if (x != 1) S[x] = fma2(four, sub2<D>(c[x - 1], m0), S[x]);
            T[x] = sub2<D>(up, dn);
        }
        const float2 w = f2(1.0f / 12.0f, 1.0f / 12.0f);
        g[0] = mul2(sub2<D>(S[2], S[0]), w);
        g[1] = mul2(fma2(four, T[1], add2(T[0], T[2])), w);
        lap = mul2(fma2(four, S[1], add2(S[0], S[2])), f2(1.0f / 6.0f, 1.0f / 6.0f));
    }
    float mupB;
    s.p0 = bulk_p0(p, m0.x, m0.y, mupB);
    s.lap = lap;
    const float Lr = fmaf(p.krr, lap.x, p.krp * lap.y), Lp = fmaf(p.kpp, lap.y, p.krp * lap.x);
    s.mup = mupB - Lp;
    // P_ab = krr dr_a dr_b + kpp dp_a dp_b + krp (dr_a dp_b + dp_a dr_b) + iso delta_ab,
    // iso = p0 - rho Lr - phi Lp - (trace of the gradient part)/2
    float hr[D], hp[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        hr[a] = fmaf(p.krr, g[a].x, p.krp * g[a].y);
        hp[a] = fmaf(p.kpp, g[a].y, p.krp * g[a].x);
    }
    auto gg = [&](int a, int b) { return fmaf(g[a].x, hr[b], g[a].y * hp[b]); };
    float tr = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) {
        s.d[a] = gg(a, a);
        tr += s.d[a];
    }
    s.iso = fmaf(-0.5f, tr, fmaf(-m0.y, Lp, fmaf(-m0.x, Lr, s.p0)));
    s.o[0] = gg(0, 1);
    if constexpr (D == 3) {
        s.o[1] = gg(0, 2);
        s.o[2] = gg(1, 2);
    }
    return s;
}

// Q = rho c_s^2 I - P ({xx, yy, xy} in 2D, {xx, yy, zz, xy, xz, yz} in 3D) and
// mu_phi there
template <int D, int RX, int RY>
__device__ __forceinline__ void node_q(const DevParams &p, const float2 *__restrict__ c, float *q, float &mup)
{
    const Stress<D> s = node_stress<D, RX, RY>(p, c);
    const float base = fmaf(c[0].x, 1.0f / 3.0f, -s.iso);
#pragma unroll
    for (int a = 0; a < D; ++a) q[a] = base - s.d[a];
#pragma unroll
    for (int k = 0; k < (D == 3 ? 3 : 1); ++k) q[D + k] = -s.o[k];
    mup = s.mup;
}

// ---------------------------------------------------------------------------
// Product-form equilibria (Eqs. eqrho, A, B) at u and u + du: the D1Q3 factors
// w(c) A(u) B(u)^c of one axis for both velocities (the lanes of the pairs),
// A = 2 - s, B = (2u + s)/(1 - u), s = sqrt(1 + 3 u^2).
// ---------------------------------------------------------------------------
struct Fac2 {
    float2 f0, fp, fm;
};

template <int D>
__device__ __forceinline__ Fac2 eq_factors2(float2 u)
{
    const float2 one = f2(1.0f, 1.0f);
    const float2 t = fma2(f2(3.0f, 3.0f), mul2(u, u), one);
    const float2 s = f2(sqrtf(t.x), sqrtf(t.y));
    const float2 A6 = fma2(s, f2(-1.0f / 6.0f, -1.0f / 6.0f), f2(1.0f / 3.0f, 1.0f / 3.0f));
    const float2 um = sub2<D>(one, u);
    const float2 B = mul2(fma2(f2(2.0f, 2.0f), u, s), f2(1.0f / um.x, 1.0f / um.y));
    // the reciprocal of B refined once: what B is off by then enters the two
    // factors with opposite signs (a momentum, which the collision closes) and
    // not alike (a pressure)
    float2 iB = f2(1.0f / B.x, 1.0f / B.y);
    iB = fma2(iB, fma2(f2(-iB.x, -iB.y), B, one), iB);
    Fac2 r;
    r.f0 = mul2(A6, f2(4.0f, 4.0f));
    r.fp = mul2(A6, B);
    r.fm = mul2(A6, iB);
    return r;
}

// rho times the product of the factors for every pair of directions: lane x
// the +c, lane y the -c direction of pair k
template <int D>
__device__ __forceinline__ void equilibria(float r, const float (&f0)[D], const float (&fp)[D], const float (&fm)[D],
                                           float2 (&e)[Lat<D>::NPOS])
{
    const float2 X = mul2(f2(fp[0], fm[0]), f2(r, r)), Y = f2(fp[1], fm[1]), Ys = f2(fm[1], fp[1]);
    const float x0 = f0[0] * r;
    const float2 XY = mul2(X, Y), XYs = mul2(X, Ys);
    if constexpr (D == 2) {
        e[0] = mul2(X, f2(f0[1], f0[1]));
        e[1] = mul2(Y, f2(x0, x0));
        e[2] = XY;
        e[3] = XYs;
    } else {
        const float2 Z = f2(fp[2], fm[2]), Zs = f2(fm[2], fp[2]);
        const float2 z0 = f2(f0[2], f0[2]), y0 = f2(f0[1], f0[1]);
        const float2 Xy = mul2(X, y0), Yx = mul2(Y, f2(x0, x0));
        const float xy = x0 * f0[1];
        e[0] = mul2(Xy, z0);
        e[1] = mul2(Yx, z0);
        e[2] = mul2(Z, f2(xy, xy));
        e[3] = mul2(XY, z0);
        e[4] = mul2(XYs, z0);
        e[5] = mul2(Xy, Z);
        e[6] = mul2(Xy, Zs);
        e[7] = mul2(Yx, Z);
        e[8] = mul2(Yx, Zs);
        e[9] = mul2(XY, Z);
        e[10] = mul2(XY, Zs);
        e[11] = mul2(XYs, Z);
        e[12] = mul2(XYs, Zs);
    }
}

// shared memory of a stepping CTA (beside the dynamic staging area)
template <int D>
struct StepShared {
    static constexpr int TX = Tile<D>::X, TY = Tile<D>::Y, TZ = Tile<D>::Z, NT = TX * TY * TZ;
    static constexpr int RX = TX + 4, RY = TY + 4, RZ = D == 3 ? TZ + 4 : 1;
    static constexpr int SX = TX + 2, SY = TY + 2, SZ = D == 3 ? TZ + 2 : 1;
    static constexpr int NR = RX * RY * RZ, NS = SX * SY * SZ;
    // row length of rp.  D3Q27: 34 = SX mod 16, so that a half-warp of the tensor
    // stage that crosses a row's end meets no bank twice (1.4 % of the 192 x 192 x
    // 128 step).  With the staged populations a CTA stays below the 100 KB beyond
    // which the L1 cache shrinks (staging rows of 16-byte pieces, where tensor
    // copies are not possible, passed it and was 5 to 8 % slower).
    static constexpr int PX = D == 3 ? 34 : RX;
    // D2Q9 tiles with ghost nodes: flags and moments of the tile + halo 2
    // widened by EM nodes, the reach of the ghost layer (for theta in
    // [20, 160] deg a ghost node's samples lie at most 3 nodes along the wall
    // and 1 across from it; farther nodes are read from global memory)
    static constexpr int EM = 3, BX = RX + 2 * EM, BY = RY + 2 * EM, NB = D == 2 ? BX * BY : 1;
    float4 qa[NS];                        // Q of the tile + halo 1: D3Q27 {xx, yy, zz, xy}; D2Q9 {xx, yy, xy, mu_phi}
    float2 rp[PX * RY * RZ];              // rho, phi of the tile + halo 2
    float2 qb[D == 3 ? NS : 1];           // D3Q27 {xz, yz}
    float mu[D == 3 ? NT : 1];            // D3Q27 mu_phi of the tile's nodes
    float2 box[NB];
    short glist[D == 2 ? NR : 1];         // the region's ghost slots, one per thread in the ghost pass
    uint8_t type[NS];                     // node flags of the tile + halo 1
    uint8_t rtype[NR];                    // ... of the tile + halo 2
    uint8_t btype[NB];
    int nghost;
    unsigned long long tma_bar;           // completion barrier of the tensor copies
};

// Node accessor of the ghost pass of a D2Q9 tile: node flags and moments from
// the box in shared memory, else from the flag array and the node's
// populations.  (ox, oy) is the box's first node.
template <int D, typename GT, int BX, int BY>
struct NodesBox {
    const DevParams &p;
    const uint8_t *type;
    const float *f;
    const void *g;
    const uint8_t *bt;
    const float2 *bm;
    int ox, oy;
    __device__ __forceinline__ bool get(int x, int y, int, float2 &m) const
    {
        const int lx = x - ox, ly = y - oy;
        if ((unsigned)lx < (unsigned)BX && (unsigned)ly < (unsigned)BY) {
            const int k = lx + BX * ly;
            if (bt[k] & TLB_SOLID) return false;
            m = bm[k];
            return true;
        }
        return node_far<D, GT>(p, type, f, g, x, y, 0, m);
    }
};

// Stage A of a D2Q9 tile: rho, phi of the tile + halo 2 summed from the
// populations (no moments pass before the step), the tile's own populations
// kept in `stage`, and in tiles at walls the ghost layer of Sec. IV.  Thread
// tid sums its own node (tile slot tid) and, for tid < NR - NT, one node of
// the halo ring: rows 0-1 and RY-2..RY-1, then the two columns on either side
// of rows 2..RY-3.  Region slots are filled for coordinates below n + 2: the
// tile's nodes use no farther neighbours, and node_near wraps one period only.
template <typename GT, bool WALLS, bool BIG>
__device__ __forceinline__ void gather_2d(const BatchEntry &e, int x0, int y0, StepShared<2> &sh, float *stage)
{
    using S = StepShared<2>;
    constexpr int Q = 9, NT = S::NT, RX = S::RX, RY = S::RY, NR = S::NR, NH = NR - NT, TX = S::TX, TY = S::TY;
    static_assert(NH == 4 * RX + 4 * TY && NT == 256, "halo ring of a 32 x 8 tile");
    const DevParams &p = e.p;
    const int tid = threadIdx.x;
    int kx[2], ky[2];
    kx[0] = 2 + tid % TX;
    ky[0] = 2 + tid / TX;
    const bool has_h = tid < NH;
    {
        const int h = has_h ? tid : 0;
        if (h < 2 * RX) { kx[1] = h % RX; ky[1] = h / RX; }
        else if (h < 4 * RX) { kx[1] = (h - 2 * RX) % RX; ky[1] = RY - 2 + (h - 2 * RX) / RX; }
        else {
            const int c = (h - 4 * RX) & 3;
            kx[1] = c < 2 ? c : TX + c;
            ky[1] = 2 + ((h - 4 * RX) >> 2);
        }
    }
    float fa[2][Q], ga[2][Q];
    __half gh[2][Q];                     // FP16 storage: the raw moving populations
    int na[2];
    bool in[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int X = x0 - 2 + kx[s], Y = y0 - 2 + ky[s];
        in[s] = (s == 0 || has_h) && X < p.nx + 2 && Y < p.ny + 2;
        na[s] = in[s] ? node_near(p, X, Y, 0) : 0;
    }
    // issue both nodes' loads before any sum.  No load is predicated: slots off
    // the lattice read node 0 (what they hold is not used), and the ring's loads
    // are skipped by whole warps (2 % of the 2048 x 2048 step, 2.4 % of a batch)
    auto load = [&](int s) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            fa[s][i] = *elem<BIG>(e.f_in + (long long)i * p.N, na[s]);
            if (sizeof(GT) == 4 || i == 0) {
                ga[s][i] = *elem<BIG>((const float *)e.g_in + (long long)i * p.N, na[s]);
            } else {
                // the value GIO<__half>::ld returns, from one load of the raw half
                gh[s][i] = *elem<BIG>((const __half *)((const char *)e.g_in + 4 * p.N) + (long long)(i - 1) * p.N, na[s]);
                ga[s][i] = __half2float(gh[s][i]) * p.g_unscale;
            }
        }
    };
    load(0);
    if (has_h) load(1);
    {
        // the node's own populations for the collision, in the staging layout
        // (rows of nodes off the lattice hold what their wrapped nodes do)
#pragma unroll
        for (int i = 0; i < Q; ++i) stage[i * NT + tid] = fa[0][i];
        if (sizeof(GT) == 4) {
#pragma unroll
            for (int i = 0; i < Q; ++i) stage[(Q + i) * NT + tid] = ga[0][i];
        } else {
            stage[Q * NT + tid] = ga[0][0];
            __half *s16 = reinterpret_cast<__half *>(&stage[(Q + 1) * NT]);
#pragma unroll
            for (int i = 1; i < Q; ++i) s16[(i - 1) * NT + tid] = gh[0][i];
        }
    }
    bool ghost = false;
    if (WALLS && tid == 0) sh.nghost = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        if (s == 1 && !has_h) break;
        const int k = kx[s] + RX * ky[s];
        // the summation order of the moments kernel
        float2 m = f2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < Q; ++i) m = add2(m, f2(fa[s][i], ga[s][i]));
        m.x = 1.0f + m.x;
        if (WALLS) {
            const uint8_t t = in[s] ? __ldg(e.type + na[s]) : (uint8_t)TLB_SOLID;
            ghost |= (t & TLB_GHOST) != 0;
            if (t & TLB_SOLID) m = f2(0.f, 0.f);
            sh.rtype[k] = t;
        }
        sh.rp[k] = m;
    }
    if constexpr (WALLS) {
        constexpr int EM = S::EM, BX = S::BX, BY = S::BY;
        // the ghost layer of Sec. IV from the fluid moments
        if (__syncthreads_or(ghost)) {
            // list the ghost slots (in any order: each ghost value depends on
            // the box alone), so that no thread takes more than one of them
            for (int k = tid; k < NR; k += NT)
                if (sh.rtype[k] & TLB_GHOST) sh.glist[atomicAdd(&sh.nghost, 1)] = (short)k;
            // the box: region slots copied (where filled) ...
            for (int k = tid; k < NR; k += NT) {
                const int lx = k % RX, ly = k / RX, kb = (lx + EM) + BX * (ly + EM);
                const int X = x0 - 2 + lx, Y = y0 - 2 + ly;
                if (X < p.nx + 2 && Y < p.ny + 2) {
                    sh.btype[kb] = sh.rtype[k];
                    sh.box[kb] = sh.rp[k];
                } else {                      // lattices narrower than a tile
                    const long long n = node_of(p, X, Y, 0);
                    const uint8_t t = __ldg(e.type + n);
                    const float2 m = pop_moments<2, GT>(p, e.f_in, e.g_in, n);
                    sh.btype[kb] = t;
                    sh.box[kb] = (t & TLB_SOLID) ? f2(0.f, 0.f) : m;
                }
            }
            // ... and the margin summed from the populations: at most two
            // nodes per thread, all loads issued before the sums.  Margin
            // index h: rows above, rows below, then the columns either side.
            constexpr int NM = BX * BY - RX * RY;
            static_assert(NM <= 2 * NT, "margin of two nodes per thread");
            int kb[2];
            long long nm[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int h = (tid + NT * j < NM) ? tid + NT * j : 0;
                int bx, by;
                if (h < EM * BX) { bx = h % BX; by = h / BX; }
                else if (h < 2 * EM * BX) { bx = (h - EM * BX) % BX; by = BY - EM + (h - EM * BX) / BX; }
                else {
                    const int c = (h - 2 * EM * BX) % (2 * EM);
                    bx = c < EM ? c : RX + c;
                    by = EM + (h - 2 * EM * BX) / (2 * EM);
                }
                kb[j] = bx + BX * by;
                nm[j] = node_of(p, x0 - 2 - EM + bx, y0 - 2 - EM + by, 0);
            }
            const uint8_t t0 = __ldg(e.type + nm[0]), t1 = __ldg(e.type + nm[1]);
            const float2 m0 = pop_moments<2, GT>(p, e.f_in, e.g_in, nm[0]);
            const float2 m1 = pop_moments<2, GT>(p, e.f_in, e.g_in, nm[1]);
            if (tid < NM) {
                sh.btype[kb[0]] = t0;
                sh.box[kb[0]] = (t0 & TLB_SOLID) ? f2(0.f, 0.f) : m0;
            }
            if (tid + NT < NM) {
                sh.btype[kb[1]] = t1;
                sh.box[kb[1]] = (t1 & TLB_SOLID) ? f2(0.f, 0.f) : m1;
            }
            __syncthreads();
            const NodesBox<2, GT, BX, BY> acc{p, e.type, e.f_in, e.g_in, sh.btype, sh.box, x0 - 2 - EM, y0 - 2 - EM};
            for (int j = tid; j < sh.nghost; j += NT) {
                const int k = sh.glist[j];
                float gr, gp;
                ghost_value<2>(p, acc, x0 - 2 + k % RX, y0 - 2 + k / RX, 0, gr, gp);
                sh.rp[k] = make_float2(gr, gp);
            }
            __syncthreads();      // the ghost values, before the tensor stage reads them
        }
    } else {
        __syncthreads();
    }
}

// D3Q27: requests the tile's own populations into `stage`
template <typename GT>
__device__ __forceinline__ void own_copies_3d(const BatchEntry &e, int x0, int y0, int z0, StepShared<3> &sh, float *stage,
                                              bool use_tma)
{
    constexpr int Q = 27, NT = StepShared<3>::NT, TX = StepShared<3>::TX, TY = StepShared<3>::TY;
    const DevParams &p = e.p;
    const int tid = threadIdx.x;
    if (use_tma) {
        // one thread: a box of TX x TY x TZ nodes x all directions per array
        // (x0 is a multiple of 16 nodes: 16-byte aligned inner coordinate)
        if (tid == 0) {
            mbar_init(&sh.tma_bar, 1);
            const unsigned bytes = (unsigned)(Q * NT * 4) +
                                   (sizeof(GT) == 4 ? (unsigned)(Q * NT * 4) : (unsigned)(NT * 4 + (Q - 1) * NT * 2));
#ifdef TLB_TEST_TMA_TIMEOUT
            // test builds only: the barrier expects 16 bytes more than the
            // copies send, so its wait runs out and the timeout path runs
            mbar_expect_tx(&sh.tma_bar, bytes + 16u);
#else
            mbar_expect_tx(&sh.tma_bar, bytes);
#endif
            tma_load_4d(&stage[0], e.tm[0], x0, y0, z0, 0, &sh.tma_bar);
            if (sizeof(GT) == 4) {
                tma_load_4d(&stage[Q * NT], e.tm[1], x0, y0, z0, 0, &sh.tma_bar);
            } else {
                tma_load_3d(&stage[Q * NT], e.tm[1], x0, y0, z0, &sh.tma_bar);
                tma_load_4d(&stage[(Q + 1) * NT], e.tm[2], x0, y0, z0, 0, &sh.tma_bar);
            }
        }
        return;
    }
    const int ax = x0 + tid % TX, ay = y0 + (tid / TX) % TY, az = z0 + tid / (TX * TY);
    if (ax < p.nx && ay < p.ny && az < p.nz) {
        const int an = ax + p.nx * (ay + p.ny * az);
#pragma unroll
        for (int i = 0; i < Q; ++i) cp_async4(&stage[i * NT + tid], e.f_in + (long long)i * p.N + an);
        if (sizeof(GT) == 4) {
#pragma unroll
            for (int i = 0; i < Q; ++i)
                cp_async4(&stage[(Q + i) * NT + tid], (const float *)e.g_in + (long long)i * p.N + an);
        } else {
            cp_async4(&stage[Q * NT + tid], (const float *)e.g_in + an);
            // the FP16 moving populations of two x-neighbours share a 4-byte
            // word (nx even): the even thread of each pair copies it
            if ((p.nx & 1) == 0 && (tid & 1) == 0) {
                const char *h = (const char *)e.g_in + 4 * p.N;
                __half *s16 = reinterpret_cast<__half *>(&stage[(Q + 1) * NT]);
#pragma unroll
                for (int i = 1; i < Q; ++i)
                    cp_async4(&s16[(i - 1) * NT + tid], h + 2 * ((long long)(i - 1) * p.N + an));
            }
        }
    }
    cp_async_commit();
}

// Stage A of a D3Q27 tile: rho, phi (and flags) of the tile + halo 2 from the
// moments pass, own_copies() called behind those loads (copies requested ahead
// of them would keep them waiting), and in tiles at walls the ghost layer (the
// moments pass leaves ghost nodes alone).  Also the D2Q9 tiles of the field pass.
template <int D, bool WALLS, class OWN>
__device__ __forceinline__ void gather_moments(const BatchEntry &e, int x0, int y0, int z0, StepShared<D> &sh,
                                               const OWN &own_copies)
{
    using S = StepShared<D>;
    constexpr int NT = S::NT, RX = S::RX, RY = S::RY, NR = S::NR, HZ = D == 3 ? 2 : 0;
    const DevParams &p = e.p;
    const int tid = threadIdx.x;
    if constexpr (D == 3 && !WALLS) {
        constexpr int RZ = S::RZ, TX = S::TX, TY = S::TY;
        // the region of a tile away from the lattice's edges lies in memory as
        // rows of RX nodes: two nodes a load where the rows are 8-byte aligned
        if (x0 >= 2 && y0 >= 2 && z0 >= 2 && x0 + TX + 2 <= p.nx && y0 + TY + 2 <= p.ny &&
            z0 + S::TZ + 2 <= p.nz && e.paired) {
            constexpr int RH = RX / 2, NP = RH * RY * RZ, PER = (NP + NT - 1) / NT;
            float2 lr[PER], lp[PER];
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const int k = tid + NT * j;
                const int row = k / RH;
                const int n = k >= NP ? 0
                                      : (int)chk_node(x0 - 2 + 2 * (k - RH * row) +
                                                          p.nx * (y0 - 2 + row % RY + p.ny * (z0 - 2 + row / RY)), p);
                if (k < NP) {
                    lr[j] = *reinterpret_cast<const float2 *>(e.rho + n);
                    lp[j] = *reinterpret_cast<const float2 *>(e.phi + n);
                }
            }
            own_copies();
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const int k = tid + NT * j;
                if (k < NP)
                    reinterpret_cast<float4 *>(sh.rp)[(k / RH) * (S::PX / 2) + k % RH] =
                        make_float4(lr[j].x, lp[j].x, lr[j].y, lp[j].y);
            }
            __syncthreads();
            return;
        }
    }
    // all of a thread's slots loaded in one round (loads issued before use)
    constexpr int PER = (NR + NT - 1) / NT;
    float lr[PER], lp[PER];
    uint8_t lt[PER];
    bool ghost = false;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int k = tid + NT * j;
        const int X = x0 - 2 + k % RX, Y = y0 - 2 + (k / RX) % RY, Z = z0 - HZ + k / (RX * RY);
        const bool in = k < NR && X < p.nx + 2 && Y < p.ny + 2 && Z < p.nz + HZ;
        const int n = in ? node_near(p, X, Y, Z) : 0;
        if (WALLS) lt[j] = in ? __ldg(e.type + n) : (uint8_t)TLB_SOLID;
        lr[j] = in ? e.rho[n] : 0.f;
        lp[j] = in ? e.phi[n] : 0.f;
    }
    own_copies();
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int k = tid + NT * j;
        if (k >= NR) break;
        sh.rp[(k / RX) * S::PX + k % RX] = make_float2(lr[j], lp[j]);
        if (WALLS) {
            sh.rtype[k] = lt[j];
            ghost |= (lt[j] & TLB_GHOST) != 0;
        }
    }
    if (WALLS && ghost) {
        const NodesGlobal acc{p, e.type, e.rho, e.phi};
#pragma unroll 1
        for (int k = tid; k < NR; k += NT) {
            if (!(sh.rtype[k] & TLB_GHOST)) continue;      // unfilled slots hold TLB_SOLID alone
            float gr, gp;
            ghost_value<D>(p, acc, x0 - 2 + k % RX, y0 - 2 + (k / RX) % RY, z0 - HZ + k / (RX * RY), gr, gp);
            sh.rp[(k / RX) * S::PX + k % RX] = make_float2(gr, gp);
        }
    }
    __syncthreads();
}

// Force at a first-layer node (Sec. IV): no value is taken from a solid node.
// Along an axis with an adjacent solid node the derivative is one-sided; along
// the others a solid term is replaced by its mirror image across the wall axes.
template <int D, class QC, int NF>
__device__ __forceinline__ void wall_force(const QC &qc, const uint8_t *stype, uint8_t tc, int sc, float (&F)[NF])
{
    constexpr int Q = Lat<D>::Q, SX = StepShared<D>::SX, SY = StepShared<D>::SY;
    auto off = [](int cx, int cy, int cz) { return cx + SX * (cy + SY * cz); };
    const bool wall[3] = {(tc & TLB_WALLX) != 0, (tc & TLB_WALLY) != 0, (tc & TLB_WALLZ) != 0};
#pragma unroll
    for (int gdir = 0; gdir < D; ++gdir) {
        if (wall[gdir]) {
            // fluid-side differences, doubled
#pragma unroll
            for (int i = 1; i < Q; ++i) {
                if (cc<D>(i, gdir) == 0) continue;
                const int m = sc + off(cc<D>(i, 0), cc<D>(i, 1), cc<D>(i, 2));
                if (stype[m] & TLB_SOLID) continue;
                const float wc = 6.0f * wt<D>(i) * (float)cc<D>(i, gdir);
#pragma unroll
                for (int a = 0; a < D; ++a) F[a] = fmaf(wc, qc(qcomp<D>(a, gdir), m) - qc(qcomp<D>(a, gdir), sc), F[a]);
            }
        } else {
#pragma unroll
            for (int i = 1; i < Q; ++i) {
                if (cc<D>(i, gdir) == 0) continue;
                int cx = cc<D>(i, 0), cy = cc<D>(i, 1), cz = cc<D>(i, 2);
                int m = sc + off(cx, cy, cz);
                if (stype[m] & TLB_SOLID) {
                    // mirror image across the wall axes, else the node itself
                    if (wall[0]) cx = -cx;
                    if (wall[1]) cy = -cy;
                    if (D == 3 && wall[2]) cz = -cz;
                    const int mm = sc + off(cx, cy, cz);
                    m = (stype[mm] & TLB_SOLID) ? sc : mm;
                }
                const float wc = 3.0f * wt<D>(i) * (float)cc<D>(i, gdir);
#pragma unroll
                for (int a = 0; a < D; ++a) F[a] = fmaf(wc, qc(qcomp<D>(a, gdir), m), F[a]);
            }
        }
    }
}

// Wetting force of method 1 (Eq. forceBC) on fluid nodes off the first layer
template <int D, int NF>
__device__ __forceinline__ void wetting_force(const DevParams &p, const uint8_t *stype, uint8_t tc, int sc, float r,
                                              float ph, float (&F)[NF])
{
    constexpr int Q = Lat<D>::Q, SX = StepShared<D>::SX, SY = StepShared<D>::SY;
    if (p.wetting != TLB_WET_FORCE || !(tc & TLB_NEAR) || (p.kw_rho == 0.f && p.kw_phi == 0.f)) return;
    const float rrel = (r - p.rho_g) * p.inv_drho;
    const float amp = rrel * fmaf(ph * p.inv_chi, p.kw_phi, p.kw_rho);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const int m = sc + cc<D>(i, 0) + SX * (cc<D>(i, 1) + SY * cc<D>(i, 2));
        if (!(stype[m] & TLB_FIRST)) continue;
#pragma unroll
        for (int a = 0; a < D; ++a) F[a] = fmaf(amp, wt<D>(i) * (float)cc<D>(i, a), F[a]);
    }
}

// Q and mu_phi at every fluid node of the tile + halo 1 (tiles at walls: with
// the node flags, which the force reads)
template <int D, bool WALLS>
__device__ __forceinline__ void tensor_stage(const DevParams &p, int x0, int y0, int z0, StepShared<D> &sh)
{
    using S = StepShared<D>;
    constexpr int RX = S::RX, RY = S::RY, SX = S::SX, SY = S::SY, NS = S::NS, HZ = D == 3 ? 1 : 0;
    // slot stride: the compile-time thread count for D2Q9 (the loop unrolls;
    // measured faster), the run-time one for D3Q27 (unrolled measured 3 % slower)
    const int KSTEP = D == 2 ? S::NT : (int)blockDim.x;
    for (int k = threadIdx.x; k < NS; k += KSTEP) {
        const int lx = k % SX, ly = (k / SX) % SY, lz = k / (SX * SY);
        const int c = (lx + 1) + RX * ((ly + 1) + RY * (lz + HZ));
        float q[D == 2 ? 3 : 6], mup;
        bool off = false;
        if (WALLS) {
            const int X = x0 - 1 + lx, Y = y0 - 1 + ly, Z = z0 - HZ + lz;
            const uint8_t tk = (X >= p.nx + 1 || Y >= p.ny + 1 || Z >= p.nz + 1) ? (uint8_t)TLB_SOLID : sh.rtype[c];
            sh.type[k] = tk;
            off = tk & TLB_SOLID;
        }
        if (off) {
#pragma unroll
            for (int j = 0; j < (D == 2 ? 3 : 6); ++j) q[j] = 0.f;
            mup = 0.f;
        } else {
            node_q<D, S::PX, RY>(p, sh.rp + (lx + 1) + S::PX * ((ly + 1) + RY * (lz + HZ)), q, mup);
        }
        if constexpr (D == 2) {
            sh.qa[k] = make_float4(q[0], q[1], q[2], mup);
        } else {
            sh.qa[k] = make_float4(q[0], q[1], q[2], q[3]);
            sh.qb[k] = make_float2(q[4], q[5]);
            // for the tile's own nodes
            const int tx = lx - 1, ty = ly - 1, tz = lz - 1;
            if ((unsigned)tx < (unsigned)S::TX && (unsigned)ty < (unsigned)S::TY && (unsigned)tz < (unsigned)S::TZ)
                sh.mu[tx + S::TX * (ty + S::TY * tz)] = mup;
        }
    }
}

// Force F = div(rho c_s^2 I - P) of the node at slot sc with the wall rules
// (Sec. IV), and mu_phi, from the tensor stage of the tile
template <int D, bool WALLS>
__device__ __forceinline__ float node_force(const DevParams &p, const StepShared<D> &sh, int sc, uint8_t tc, float r,
                                            float ph, float (&F)[D])
{
    constexpr int Q = Lat<D>::Q, NPOS = Lat<D>::NPOS, SX = StepShared<D>::SX, SY = StepShared<D>::SY;
    // component c (qcomp order) of Q at slot m
    auto qc = [&](int c, int m) -> float {
        if constexpr (D == 2) return c == 0 ? sh.qa[m].x : c == 1 ? sh.qa[m].y : sh.qa[m].z;
        else return c == 0 ? sh.qa[m].x : c == 1 ? sh.qa[m].y : c == 2 ? sh.qa[m].z : c == 3 ? sh.qa[m].w
                    : c == 4 ? sh.qb[m].x : sh.qb[m].y;
    };
#pragma unroll
    for (int a = 0; a < D; ++a) F[a] = 0.f;
    if (!WALLS || !(tc & TLB_FIRST)) {
        // no solid node within one link: the isotropic stencil on the
        // differences of opposite neighbours, summed per weight
        float acc[D][D];
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int b = 0; b < D; ++b) acc[a][b] = 0.f;
#pragma unroll
        for (int k = 0; k < NPOS; ++k) {
            const int o = Lat<D>::pos(k, 0) + SX * (Lat<D>::pos(k, 1) + SY * Lat<D>::pos(k, 2));
            const float4 ap = sh.qa[sc + o], am = sh.qa[sc - o];
            float t[6];
            const float2 t0 = sub2<D>(f2(ap.x, ap.y), f2(am.x, am.y));
            t[0] = t0.x;
            t[1] = t0.y;
            if constexpr (D == 2) {
                t[2] = ap.z - am.z;
            } else {
                const float2 t1 = sub2<D>(f2(ap.z, ap.w), f2(am.z, am.w)), t2 = sub2<D>(sh.qb[sc + o], sh.qb[sc - o]);
                t[2] = t1.x;
                t[3] = t1.y;
                t[4] = t2.x;
                t[5] = t2.y;
            }
#pragma unroll
            for (int a = 0; a < D; ++a)
#pragma unroll
                for (int b = 0; b < D; ++b)
                    if (Lat<D>::pos(k, b) != 0)
                        acc[pair_class<D>(k)][a] += Lat<D>::pos(k, b) > 0 ? t[qcomp<D>(a, b)] : -t[qcomp<D>(a, b)];
        }
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
            for (int k = 0; k < D; ++k)
                F[a] = fmaf(3.0f * (k == 0 ? wt<D>(1) : k == 1 ? wt<D>(2 * D + 1) : wt<D>(Q - 1)), acc[k][a], F[a]);
    } else {
        wall_force<D>(qc, sh.type, tc, sc, F);
    }
    if (WALLS) wetting_force<D>(p, sh.type, tc, sc, r, ph, F);
    return D == 2 ? sh.qa[sc].w : sh.mu[threadIdx.x];
}

// Where a node's populations go: push streaming with halfway bounce-back.
// The node index plus one offset per axis and sign (periodic wrap included;
// node indices fit in 32 bits).
template <int D>
struct Push {
    const DevParams &p;
    int n, xm, xp, ym, yp, zm, zp;
    __device__ __forceinline__ Push(const DevParams &q, int x, int y, int z) : p(q)
    {
        n = x + q.nx * (y + q.ny * z);
        xm = x == 0 ? q.nx - 1 : -1;
        xp = x == q.nx - 1 ? 1 - q.nx : 1;
        ym = (y == 0 ? q.ny - 1 : -1) * q.nx;
        yp = (y == q.ny - 1 ? 1 - q.ny : 1) * q.nx;
        const int pl = D == 3 ? q.nx * q.ny : 0;
        zm = D == 3 ? (z == 0 ? q.nz - 1 : -1) * pl : 0;
        zp = D == 3 ? (z == q.nz - 1 ? 1 - q.nz : 1) * pl : 0;
    }
    __device__ __forceinline__ int to(int cx, int cy, int cz) const
    {
        int m = n;
        if (cx != 0) m += cx > 0 ? xp : xm;
        if (cy != 0) m += cy > 0 ? yp : ym;
        if (D == 3 && cz != 0) m += cz > 0 ? zp : zm;
        return (int)chk_node(m, p);
    }
};

// ELBM collision of f (Eqs. ELBMequation, ELBMForcingExactDiff,
// EntropyEquation).  f0, fp[k] hold f~ = f - w of the rest population and of
// the pairs on entry; v is the fluid velocity on return, and dl0, dl the
// relaxation terms D, fp0, fp the mirror state less the weight, f' - w, with
// f_new - w = (f' - w) + ab D.  own, stride: Q floats of shared memory of the
// thread's own (free for scratch).
template <int D>
__device__ __forceinline__ void collide_f(const BatchEntry &e, float r, float ph, const float (&F)[D], float f0,
                                          float2 (&fp)[Lat<D>::NPOS], float2 (&dl)[Lat<D>::NPOS], float &fp0, float &dl0,
                                          float &ab, float (&v)[D], float *own, int stride)
{
    constexpr int Q = Lat<D>::Q, NPOS = Lat<D>::NPOS;
    const DevParams &p = e.p;
    const float inv_r = 1.0f / r;
    float2 j2[D];
#pragma unroll
    for (int a = 0; a < D; ++a) j2[a] = f2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < NPOS; ++k)
#pragma unroll
        for (int a = 0; a < D; ++a)
            if (Lat<D>::pos(k, a) != 0) j2[a] = Lat<D>::pos(k, a) > 0 ? add2(j2[a], fp[k]) : sub2<D>(j2[a], fp[k]);
    float u0[D], up[D], um[D], d0[D], dp[D], dm[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        const float u = (j2[a].x - j2[a].y) * inv_r;
        const float du = F[a] * inv_r;          // delta u = F dt / rho
        v[a] = fmaf(0.5f, du, u);               // fluid velocity
        const Fac2 t = eq_factors2<D>(f2(u, u + du));
        u0[a] = t.f0.x; up[a] = t.fp.x; um[a] = t.fm.x;
        d0[a] = t.f0.y; dp[a] = t.fp.y; dm[a] = t.fm.y;
    }
    // The relaxation D_i = f^eq_i(u) - f_i carries no mass or momentum and the
    // forcing term F_i = f^eq_i(u+du) - f^eq_i(u) carries mass 0 and momentum F.
    // In FP32 the rest population closes the mass balances and the +-axis
    // pairs the momentum balances, so the update conserves both to rounding.
    // The mirror state f' = f + F_i (Eq. mirror_state) is kept less the weight,
    // like f: formed as f^eq(u + du) - D_i it would drift (mass 8e-6 off after
    // 1000 steps of a 64 x 64 drop instead of 2.5e-7).
    {
        float2 eq[NPOS], ed[NPOS];
        equilibria<D>(r, u0, up, um, eq);
        equilibria<D>(r, d0, dp, dm, ed);
        float2 rdl = f2(0.f, 0.f), rF = f2(0.f, 0.f), mdl[D], mF[D];
#pragma unroll
        for (int a = 0; a < D; ++a) mdl[a] = mF[a] = f2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < NPOS; ++k) {
            const float w = wt<D>(2 * k + 1);
            const float2 di = sub2<D>(sub2<D>(eq[k], f2(w, w)), fp[k]);    // f^eq(u) - f = f^eq(u + du) - f'
            const float2 Fi = sub2<D>(ed[k], eq[k]);
            rdl = add2(rdl, di);
            rF = add2(rF, Fi);
#pragma unroll
            for (int a = 0; a < D; ++a)
                if (Lat<D>::pos(k, a) != 0) {
                    mdl[a] = Lat<D>::pos(k, a) > 0 ? add2(mdl[a], di) : sub2<D>(mdl[a], di);
                    mF[a] = Lat<D>::pos(k, a) > 0 ? add2(mF[a], Fi) : sub2<D>(mF[a], Fi);
                }
            dl[k] = di;
            fp[k] = add2(fp[k], Fi);
        }
        dl0 = -(rdl.x + rdl.y);
        fp0 = f0 - (rF.x + rF.y);
#pragma unroll
        for (int a = 0; a < D; ++a) {             // axis directions: pair a
            const float hd = 0.5f * (mdl[a].x - mdl[a].y), hF = 0.5f * (F[a] - (mF[a].x - mF[a].y));
            dl[a].x -= hd;
            dl[a].y += hd;
            fp[a].x += hF;
            fp[a].y -= hF;
        }
    }
    // Entropic alpha (Eq. EntropyEquation) from x_i = D_i / f'_i.  The moments
    // a_2 .. a_4 of x alone give alpha = 2 + e1 + e2, to a fraction of its
    // rounding up to max|x| = ALPHA_SHORT_MAX.  Above it the moments a_5 .. a_7 complete
    // the fifth-order series, above ALPHA_SERIES_MAX Halley's method follows.
    float al = 2.0f, fmn, xmax, a2, a3, a4;
    {
        const float q0 = fp0 + wt<D>(0);
        const float x = dl0 * (1.0f / q0);
        fmn = q0;
        const float t2 = dl0 * x, t3 = t2 * x;
        a2 = t2;
        a3 = t3;
        a4 = t3 * x;
        xmax = fabsf(x);
        float2 b2 = f2(0.f, 0.f), b3 = b2, b4 = b2;
#pragma unroll
        for (int k = 0; k < NPOS; ++k) {
            const float w = wt<D>(2 * k + 1);
            const float2 q = add2(fp[k], f2(w, w));
            fmn = fminf(fmn, fminf(q.x, q.y));
            const float2 xk = mul2(dl[k], f2(1.0f / q.x, 1.0f / q.y));
            xmax = fmaxf(xmax, fmaxf(fabsf(xk.x), fabsf(xk.y)));
            const float2 c2 = mul2(dl[k], xk), c3 = mul2(c2, xk);
            b2 = add2(b2, c2);
            b3 = add2(b3, c3);
            b4 = fma2(c3, xk, b4);
        }
        a2 += b2.x + b2.y;
        a3 += b3.x + b3.y;
        a4 += b4.x + b4.y;
    }
    // not positive, or not a number (a minimum passes NaN over; the sums behind
    // the rest population carry it)
    if (!(r > 0.f) || !(fmn > 0.f) || !(fp0 + wt<D>(0) > 0.f) || !(fabsf(dl0) <= 3.0e38f)) {
        atomicOr(e.status, STATUS_DIVERGED);
    } else if (xmax >= 1e-5f && a2 > 0.f) {
        if (xmax <= ALPHA_SHORT_MAX) {
            al = alpha_short(a2, a3, a4);
        } else {
            float a5, a6, a7;
            {
                const float x = dl0 * (1.0f / (fp0 + wt<D>(0)));
                const float c5 = ((dl0 * x) * x) * x * x;
                a5 = c5;
                a6 = c5 * x;
                a7 = c5 * x * x;
                float2 b5 = f2(0.f, 0.f), b6 = b5, b7 = b5;
#pragma unroll
                for (int k = 0; k < NPOS; ++k) {
                    const float w = wt<D>(2 * k + 1);
                    const float2 q = add2(fp[k], f2(w, w));
                    const float2 xk = mul2(dl[k], f2(1.0f / q.x, 1.0f / q.y));
                    const float2 c4 = mul2(mul2(mul2(dl[k], xk), xk), xk), x2 = mul2(xk, xk), c6 = mul2(c4, x2);
                    b5 = fma2(c4, xk, b5);
                    b6 = add2(b6, c6);
                    b7 = fma2(c6, xk, b7);
                }
                a5 += b5.x + b5.y;
                a6 += b6.x + b6.y;
                a7 += b7.x + b7.y;
            }
            al = alpha_series(a2, a3, a4, a5, a6, a7);
            if (xmax > ALPHA_SERIES_MAX) {
                // f' over f' - w and x over D, to hold no further arrays; back behind it
                // (a rounding more each, so that the balances closed above hold to a
                // few roundings of f' there and not to those of D)
                float xs[Q], fs[Q], xneg = 0.f;
                fs[0] = fp0 + wt<D>(0);
                xs[0] = dl0 * (1.0f / fs[0]);
#pragma unroll
                for (int k = 0; k < NPOS; ++k) {
                    fs[2 * k + 1] = fp[k].x + wt<D>(2 * k + 1);
                    fs[2 * k + 2] = fp[k].y + wt<D>(2 * k + 1);
                    xs[2 * k + 1] = dl[k].x * (1.0f / fs[2 * k + 1]);
                    xs[2 * k + 2] = dl[k].y * (1.0f / fs[2 * k + 2]);
                }
                // positivity bound alpha_max = 1 / max(-x_i)
#pragma unroll
                for (int i = 0; i < Q; ++i) xneg = fmaxf(xneg, -xs[i]);
                const float amax = xneg > 0.f ? 1.0f / xneg : 3.0e38f;
                al = alpha_newton<Q>(fs, xs, amax, al, own, stride);
                fp0 = fs[0] - wt<D>(0);
                dl0 = xs[0] * fs[0];
#pragma unroll
                for (int k = 0; k < NPOS; ++k) {
                    fp[k] = f2(fs[2 * k + 1] - wt<D>(2 * k + 1), fs[2 * k + 2] - wt<D>(2 * k + 1));
                    dl[k] = f2(xs[2 * k + 1] * fs[2 * k + 1], xs[2 * k + 2] * fs[2 * k + 2]);
                }
            }
        }
    }
    ab = al * local_beta(p, r, ph);
}

// The new f of a node to its neighbours.  BB: with halfway bounce-back, bit i
// of solid_nb set when the neighbour x + c_i is solid.
template <int D, bool BB, bool BIG>
__device__ __forceinline__ void push_f(const BatchEntry &e, const Push<D> &to, unsigned solid_nb, float fp0, float dl0,
                                       const float2 (&fp)[Lat<D>::NPOS], const float2 (&dl)[Lat<D>::NPOS], float ab)
{
    const long long N = e.p.N;
    auto put = [&](int i, float val) {
        float *fo = e.f_out + (long long)i * N;
        if (BB && (solid_nb & (1u << i))) (e.f_out + (long long)opp<D>(i) * N)[to.n] = val;
        else *elem<BIG>(fo, to.to(cc<D>(i, 0), cc<D>(i, 1), cc<D>(i, 2))) = val;
    };
    e.f_out[to.n] = fmaf(ab, dl0, fp0);
    const float2 ab2 = f2(ab, ab);
#pragma unroll
    for (int k = 0; k < Lat<D>::NPOS; ++k) {
        const float2 fn = fma2(ab2, dl[k], fp[k]);
        put(2 * k + 1, fn.x);
        put(2 * k + 2, fn.y);
    }
}

// c.v of the pair k's first direction
template <int D>
__device__ __forceinline__ float along(int k, const float (&v)[D])
{
    float cv = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a)
        if (Lat<D>::pos(k, a) != 0) cv += Lat<D>::pos(k, a) > 0 ? v[a] : -v[a];
    return cv;
}

// g^eq(phi, v, mu_phi): g^eq_i = w_i (A + B c.v + C (c.v)^2), an even and an odd
// part per pair
struct GEq {
    float A, B, C;
    __device__ __forceinline__ float2 pair(float w, float cv) const
    {
        const float ev = fmaf((w * C) * cv, cv, w * A), od = w * B;
        return f2(fmaf(od, cv, ev), fmaf(-od, cv, ev));
    }
};

template <int D>
__device__ __forceinline__ GEq g_eq(const DevParams &p, float ph, float mup, const float (&v)[D])
{
    float v2 = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) v2 = fmaf(v[a], v[a], v2);
    return {fmaf(3.0f * p.Gamma, mup, -(1.5f * ph * v2)), 3.0f * ph, 4.5f * ph};
}

// LBGK of g (Eq. CahnHilliardLBM) with g^eq(phi, v, mu_phi), pushed like f
template <int D, typename GT, bool BB, bool BIG, class LD>
__device__ __forceinline__ void relax_g(const BatchEntry &e, const Push<D> &to, unsigned solid_nb, float ph, float mup,
                                        const float (&v)[D], const LD &ld_g)
{
    const DevParams &p = e.p;
    auto put = [&](int i, float val) {
        const int m = to.to(cc<D>(i, 0), cc<D>(i, 1), cc<D>(i, 2));
        if (BB && (solid_nb & (1u << i))) GIO<GT>::st(e.g_out, opp<D>(i), to.n, val, p);
        else if constexpr (sizeof(GT) == 4) *elem<BIG>((float *)e.g_out + (long long)i * p.N, m) = val;
        else *elem<BIG>((__half *)((char *)e.g_out + 4 * p.N) + (long long)(i - 1) * p.N, m) = __float2half_rn(val * p.g_scale);
    };
    const GEq eq = g_eq<D>(p, ph, mup, v);
    const float2 itau = f2(p.inv_tau_g, p.inv_tau_g);
    float2 gsum = f2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < Lat<D>::NPOS; ++k) {
        const float w = wt<D>(2 * k + 1);
        const float2 gi = f2(ld_g(2 * k + 1), ld_g(2 * k + 2));
        const float2 ge = eq.pair(w, along<D>(k, v));
        gsum = add2(gsum, ge);
        const float2 gn = fma2(sub2<D>(ge, gi), itau, gi);
        put(2 * k + 1, gn.x);
        put(2 * k + 2, gn.y);
    }
    const float g0 = ld_g(0);
    const float ge0 = ph - (gsum.x + gsum.y);
    GIO<GT>::st(e.g_out, 0, to.n, fmaf(ge0 - g0, p.inv_tau_g, g0), p);
}

// One tile: gather, pressure tensor (halo 1), then one node per thread: force,
// ELBM collision of f, LBGK of g, push streaming with halfway bounce-back.
template <int D, typename GT, bool WALLS, bool BIG>
__device__ __forceinline__ void step_tile(const BatchEntry &e, int x0, int y0, int z0, StepShared<D> &sh, float *stage)
{
    using S = StepShared<D>;
    constexpr int Q = Lat<D>::Q, NPOS = Lat<D>::NPOS;
    constexpr int TX = S::TX, TY = S::TY, NT = S::NT, RX = S::RX, RY = S::RY, SX = S::SX, SY = S::SY;
    constexpr int HZ = D == 3 ? 1 : 0;
    const DevParams &p = e.p;
    const int tid = threadIdx.x;
    // tensor copies need the staging area 128-byte aligned (checked, uniform per CTA)
    const bool use_tma = D == 3 && e.tm[0] != nullptr && (smem_u32(stage) & 127u) == 0;
    if constexpr (D == 2) gather_2d<GT, WALLS, BIG>(e, x0, y0, sh, stage);
    else gather_moments<D, WALLS>(e, x0, y0, z0, sh, [&] { own_copies_3d<GT>(e, x0, y0, z0, sh, stage, use_tma); });

    tensor_stage<D, WALLS>(p, x0, y0, z0, sh);
    // every thread's staged copies complete before the barrier, so each thread
    // may read copies made by another (the FP16 pairs) and none is pending
    // when a thread leaves
    if (D == 3 && use_tma) {
        // every thread waits on the copies' barrier (its completion makes the
        // tensor copies visible to the waiting thread), at most one second; a
        // CTA whose copies did not land flags the lattice, waits once more
        // (bounded) so that no copy is left in flight, and skips the tile
        const bool lost = !mbar_wait_bounded(&sh.tma_bar, 0, 1000000000ull);
        if (__syncthreads_or(lost)) {
            if (tid == 0) atomicOr(e.status, STATUS_TIMEOUT);
            if (lost) mbar_wait_bounded(&sh.tma_bar, 0, 1000000000ull);
            return;
        }
    } else {
        if (D == 3) cp_async_wait_all();
        __syncthreads();
    }

    // ---- one node per thread ----
    const int tx = tid % TX, ty = (tid / TX) % TY, tz = tid / (TX * TY);
    const int x = x0 + tx, y = y0 + ty, z = z0 + tz;
    if (x >= p.nx || y >= p.ny || z >= p.nz) return;
    const int sc = (tx + 1) + SX * ((ty + 1) + SY * (tz + HZ));
    const uint8_t tc = WALLS ? sh.type[sc] : (uint8_t)0;
    if (tc & TLB_SOLID) return;
    const float2 rph = sh.rp[(tx + 2) + S::PX * ((ty + 2) + RY * (tz + 2 * HZ))];
    const float r = rph.x, ph = rph.y;
    float F[D];
    const float mup = node_force<D, WALLS>(p, sh, sc, tc, r, ph, F);
    float2 fp[NPOS], dl[NPOS];
    const float f0 = stage[tid];
#pragma unroll
    for (int k = 0; k < NPOS; ++k) fp[k] = f2(stage[(2 * k + 1) * NT + tid], stage[(2 * k + 2) * NT + tid]);
    float fp0, dl0, ab, v[D];
    collide_f<D>(e, r, ph, F, f0, fp, dl, fp0, dl0, ab, v, stage + tid, NT);
    const Push<D> to(p, x, y, z);
    // only first-layer nodes have solid neighbours
    unsigned solid_nb = 0;
    if (WALLS && (tc & TLB_FIRST)) {
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const int m = sc + cc<D>(i, 0) + SX * (cc<D>(i, 1) + SY * cc<D>(i, 2));
            if (sh.type[m] & TLB_SOLID) solid_nb |= 1u << i;
        }
    }
    push_f<D, WALLS, BIG>(e, to, solid_nb, fp0, dl0, fp, dl, ab);
    auto ld_g = [&](int i) -> float {
        if (sizeof(GT) == 4) return stage[(Q + i) * NT + tid];
        if (D == 2 || (p.nx & 1) == 0) {
            const __half *s16 = reinterpret_cast<const __half *>(&stage[(Q + 1) * NT]);
            return i == 0 ? stage[Q * NT + tid] : __half2float(s16[(i - 1) * NT + tid]) * p.g_unscale;
        }
        return GIO<GT>::ld(e.g_in, i, to.n, p);
    };
    relax_g<D, GT, WALLS, BIG>(e, to, solid_nb, ph, mup, v, ld_g);
}

// dynamic shared memory of the stepping kernel: f and g of the tile's own nodes
template <int D>
__device__ __forceinline__ float *step_stage()
{
    // f[Q][NT], then FP32 g[Q][NT] (or the FP32 rest channel [NT] and the FP16
    // moving channels [Q-1][NT]); D3Q27: from the first 128-byte boundary of
    // the dynamic area (tensor-copy destinations)
    extern __shared__ __align__(16) float stage_raw[];
    return D == 3 ? stage_raw + (((128u - (smem_u32(stage_raw) & 127u)) & 127u) >> 2) : stage_raw;
}

// tile k of a lattice (x fastest): its origin
template <int D>
__device__ __forceinline__ void tile_origin(const DevParams &p, unsigned k, int &x0, int &y0, int &z0)
{
    const unsigned ntx = ((unsigned)p.nx + Tile<D>::X - 1) / Tile<D>::X, nty = ((unsigned)p.ny + Tile<D>::Y - 1) / Tile<D>::Y;
    const unsigned row = k / ntx;
    x0 = (int)(k - row * ntx) * Tile<D>::X;
    if (D == 2) {
        y0 = (int)row * Tile<D>::Y;
        z0 = 0;
    } else {
        const unsigned pl = row / nty;
        y0 = (int)(row - pl * nty) * Tile<D>::Y;
        z0 = (int)pl * Tile<D>::Z;
    }
}

// A lattice stepped alone: the entry by value, one CTA per tile.
// MINB: resident CTAs per SM the registers are budgeted for.  D2Q9 comes in
// two builds with the same code (the register allocation alone differs):
// 3 CTAs/SM (80 registers, fewer spills) for launches that fit in one wave,
// 4 CTAs/SM (64 registers, more warps to hide latency) for larger ones.
// A step: D2Q9 64 x 64 8.1 us, 1024 x 64 12.2, 2048 x 2048 171; D3Q27 32 x 32 x 20
// 24, 101 x 100 x 100 218, 192 x 192 x 128 760, both passes.  Over a tile table, with
// 8 x 8 x 4 tiles and without the pairs they took 8.6, 13.1, 238, 28, 306, 1022.
template <int D, typename GT, int MINB, bool BIG>
__global__ void __launch_bounds__(256, MINB) step_kernel(const __grid_constant__ BatchEntry e)
{
    __shared__ StepShared<D> sh;
    pdl_trigger();
    int x0, y0, z0;
    const unsigned tile = D == 3 && e.backwards ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    tile_origin<D>(e.p, tile, x0, y0, z0);
    float *stage = step_stage<D>();
    // a lattice of few tiles brings their wall flags among the parameters: the
    // load is a round trip ahead of everything else (0.4 us a step)
    bool walls;
    if (e.wall_known) {
        walls = (e.wall_bits[tile >> 5] >> (tile & 31)) & 1u;
        pdl_wait();
    } else {
        // ahead of the wait: written by tlb_set_solid, which synchronises, or
        // before a launch that does not start early (tlb_step_noalloc)
        walls = __ldg(e.wall_tiles + tile) != 0;
        pdl_wait();
    }
    if (walls) step_tile<D, GT, true, BIG>(e, x0, y0, z0, sh, stage);
    else step_tile<D, GT, false, BIG>(e, x0, y0, z0, sh, stage);
}

// The same over a tile -> lattice table (lattice index, tile origin): the
// lattices of a batch in one launch, bit-identical to each stepped alone.
template <int D, typename GT, int MINB, bool BIG>
__global__ void __launch_bounds__(256, MINB) step_batch_kernel(const BatchEntry *__restrict__ E, const int4 *__restrict__ tiles)
{
    __shared__ StepShared<D> sh;
    __shared__ BatchEntry se;
    pdl_trigger();
    pdl_wait();
    const int4 t = tiles[blockIdx.x];
    static_assert(sizeof(BatchEntry) % 4 == 0 && sizeof(BatchEntry) / 4 <= 256, "entry copy");
    if (threadIdx.x < sizeof(BatchEntry) / 4)
        reinterpret_cast<int *>(&se)[threadIdx.x] = reinterpret_cast<const int *>(&E[t.x])[threadIdx.x];
    __syncthreads();
    float *stage = step_stage<D>();
    const int ntx = (se.p.nx + Tile<D>::X - 1) / Tile<D>::X, nty = (se.p.ny + Tile<D>::Y - 1) / Tile<D>::Y;
    const int k = t.y / Tile<D>::X + ntx * (t.z / Tile<D>::Y + nty * (t.w / Tile<D>::Z));
    if (se.wall_tiles[k]) step_tile<D, GT, true, BIG>(se, t.y, t.z, t.w, sh, stage);
    else step_tile<D, GT, false, BIG>(se, t.y, t.z, t.w, sh, stage);
}

// wall_tiles[k] = 1 for the tiles with a solid node in the tile + halo 2 (all
// that a tile's nodes depend on: wall rules and bounce-back reach one link,
// the ghost layer and the wetting force two)
template <int D>
__global__ void __launch_bounds__(128) wall_tiles_kernel(DevParams p, const uint8_t *__restrict__ type, uint8_t *wall_tiles)
{
    using S = StepShared<D>;
    int x0, y0, z0;
    tile_origin<D>(p, blockIdx.x, x0, y0, z0);
    bool solid = false;
    for (int k = threadIdx.x; k < S::NR; k += blockDim.x)
        solid |= (type[node_of(p, x0 - 2 + k % S::RX, y0 - 2 + (k / S::RX) % S::RY, (D == 3 ? z0 - 2 : 0) + k / (S::RX * S::RY))] &
                  TLB_SOLID) != 0;
    if (__syncthreads_or(solid)) solid = true;
    if (threadIdx.x == 0) wall_tiles[blockIdx.x] = solid;
}

}  // namespace tlb
