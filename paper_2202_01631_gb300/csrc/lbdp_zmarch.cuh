// lbdp_zmarch.cuh -- the two bulk kernels of the single-box step, marching
// along z through a tile of 32 x 8 lattice columns.
//
//   kz_fused    chemical potentials, pressure tensor, force and
//               collide-stream in one pass: per plane, the block stages psi
//               of the 36 x 12 columns around its tile (two-node halo) and
//               phi, computes mu and P for the 34 x 10 columns of the plane
//               (one-node halo) into a ring of shared-memory planes, and then
//               the force and the collide-stream of its own tile one plane
//               behind.  mu is written for the transport; P and F never leave
//               the chip.  Nodes next to a particle are left to the
//               side-stream kernels (k_pt_part, k_f_part,
//               k_collide_particles).
//   kz_scalars  the psi/phi transport (Eq. diffusion_reaction) from a ring of
//               34 x 10 planes of psi, phi, mu and u.
//
// A tile column is one thread; a block walks ZC planes (its z chunk) with
// one barrier per plane.  Halo planes of a chunk are staged (and, for the
// pressure tensor, computed) by both neighbouring chunks.  The batched kernels
// run the same bodies on the same tiles, so a box gives the same bits in them.
#pragma once

#include "lbdp_kernels.cuh"
#include "lbdp_vec.cuh"

namespace lbdp {

constexpr int kZX = 32, kZY = 8, kZThreads = kZX * kZY;
constexpr int kZ1X = kZX + 2, kZ1Y = kZY + 2, kZ1 = kZ1X * kZ1Y;   // 34 x 10: one-node halo
constexpr int kZ2X = kZX + 4, kZ2Y = kZY + 4, kZ2 = kZ2X * kZ2Y;   // 36 x 12: two-node halo
// ring depths: with these, one barrier per plane separates every write of a
// ring slot from the last read of the plane it held (see kz_fused)
constexpr int kPsiRing = 5, kPhiRing = 4, kPtRing = 4, kScalRing = 5;

// in-plane slot offset of direction i in planes of row width W
template <int W>
__host__ __device__ constexpr int poff(int i)
{
    return cx(i) + W * cy(i);
}

// Nodes a thread of a bulk kernel works on together: the node of its column in each
// half of the block's z chunk.  Two in FP32 arithmetic (packed instructions,
// one set of column offsets, 64-bit shared loads); one in FP64, which has no
// packed form and no registers to spare.
template <class R>
__host__ __device__ constexpr int zm_halves()
{
    return sizeof(R) == 8 ? 1 : 2;
}

// Particles whose nodes may lie in the columns a block stages: the planes lo
// .. lo + len - 1 (before wrapping) hold them.
struct SolidPlanes {
    int n;
    int lo[kMaxParticles], len[kMaxParticles];
};
// What the wetting ghosts of kz_fused need of them; slot[k] is where particle
// k stands in the list.
struct GhostPart {
    Geo g;
    double Hk;
    float Hk_f;
};
struct GhostParts {
    uint8_t slot[kMaxParticles];
    GhostPart geo[kMaxParticles];
};

template <class F, int NP>
struct FusedSmem {
    // the stress of a slot in two 16-byte vectors, (p_iso, grad_x psi) and
    // (grad_y psi, grad_z psi), each with the halves of a field side by side:
    // a neighbour's eight numbers come in two conflict-free 128-bit loads
    F pa[kPtRing][kZ1][2 * NP];
    F pb[kPtRing][kZ1][2 * NP];
    F psi[kPsiRing][kZ2][NP];
    F phi[kPhiRing][kZ1][NP];
    SolidPlanes sol;
    GhostParts ghost;
    // nodes of the plane in hand that take the general body (NP slot + half),
    // and how many, for even and odd iterations
    uint16_t todo[NP * kZ1];
    int ntodo[2];
};

template <class F>
struct ScalSmem {
    F g[kScalRing][kZ1][2];    // psi, phi
    F mu[kScalRing][kZ1][2];   // mu_psi, mu_phi
    F u[kScalRing][3][kZ1];
    SolidPlanes sol;
};

// Column coordinate of halo offset l (may be negative) from tile origin o on
// an axis: wrapped on a periodic axis, -1 beyond a wall.
__device__ __forceinline__ int zm_coord(int o, int l, int L, int per) { return wrap_coord(o + l, L, per); }

// ---------------------------------------------------------------------------
// planes with solid nodes.  A plane of a tile is clear when none of the
// columns the block stages there lies inside a particle or beyond a wall; its
// nodes need no flags.  The test is made from the particles' positions (a few
// integers per plane); masks and boundary flags are loaded only for planes
// next to one that is not clear.
// ---------------------------------------------------------------------------

// Whether [lo, lo + len) and [o, o + flen) share a coordinate on an axis of
// length L.
__device__ __forceinline__ bool spans_meet(int lo, int len, int o, int flen, int L, int per)
{
    if (!per) return lo < o + flen && lo + len > o;
    int a = (lo - o) % L;
    if (a < 0) a += L;
    return a < flen || a + len > L;
}

// The particles near the block's columns (grown by halo on each side), at the
// positions the current mask was made from; extra(k, i, record) takes particle
// k, i-th of the list.  kNew: from the positions after this step's particle
// update (gn), grown by what a step's velocity moves them.
template <bool kNew, class Fn>
__device__ __forceinline__ void find_solids(const DevParams& P, const DevPtrs& D, int x0, int y0, int halo,
                                            SolidPlanes& sp, Fn extra)
{
    if (threadIdx.x == 0) sp.n = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < P.np; k += blockDim.x) {
        const DevPart& q = D.parts[k];
        // |x - X| < R lies strictly between floor(X) - ceil(R) and
        // floor(X) + ceil(R) + 1
        int lo[3], w[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int g = kNew ? 1 + (int)ceilf(fabsf(q.Uf[a])) : 0;
            lo[a] = (kNew ? q.gn.Xi[a] : q.g.Xi[a]) - q.Rc - g;
            w[a] = 2 * (q.Rc + 1 + g);
        }
        if (spans_meet(lo[0], w[0], x0 - halo, kZX + 2 * halo, P.nx, P.per[0]) &&
            spans_meet(lo[1], w[1], y0 - halo, kZY + 2 * halo, P.ny, P.per[1])) {
            const int i = atomicAdd(&sp.n, 1);
            sp.lo[i] = lo[2];
            sp.len[i] = w[2];
            extra(k, i, q);
        }
    }
    __syncthreads();
}

// Whether the tile's columns reach beyond a wall in x or y.
__device__ __forceinline__ bool beyond_xy(const DevParams& P, int x0, int y0, int halo)
{
    return (!P.per[0] && (x0 < halo || x0 + kZX + halo > P.nx)) || (!P.per[1] && (y0 < halo || y0 + kZY + halo > P.ny));
}

// Whether plane p (before wrapping) is not clear.
__device__ __forceinline__ bool plane_solid(const DevParams& P, const SolidPlanes& sp, bool xywall, int p)
{
    bool s = xywall || (!P.per[2] && (p < 0 || p >= P.nz));
    for (int i = 0; i < sp.n; ++i) s = s || spans_meet(sp.lo[i], sp.len[i], p, 1, P.nz, P.per[2]);
    return s;
}

// ---------------------------------------------------------------------------
// accessors over the shared-memory planes (same interface as GAcc)
// ---------------------------------------------------------------------------
// chemical-potential body of a node next to a particle or a wall, in one half
// of the planes of kz_fused: psi and phi from the staged planes, the masks of
// the neighbours (few nodes need them) from memory
template <class F, int NP>
struct ZAccMu {
    int nb[19];
    const uint8_t* mk;
    const F* ps[3];
    int o2;   // NP * slot + half
    F phi_own;
    const GhostParts* gp;
    __device__ __forceinline__ const GhostPart& part(const DevPtrs&, int k) const { return gp->geo[gp->slot[k]]; }
    __device__ __forceinline__ uint8_t mask(int i) const { return nb[i] >= 0 ? mk[nb[i]] : kWallSlot; }
    template <int K>
    __device__ __forceinline__ F get(int i) const
    {
        if (K == 0) return ps[1 + cz(i)][o2 + NP * poff<kZ2X>(i)];
        return phi_own;   // field 1 is read at the node itself only
    }
};

// Bit 2 a + s of beyond: the neighbours on side s (0 below, 1 above) of axis a
// lie beyond a wall.
__device__ __forceinline__ bool beyond_wall(unsigned beyond, int i)
{
    const unsigned c = (cx(i) < 0 ? 1u : cx(i) > 0 ? 2u : 0u) | (cy(i) < 0 ? 4u : cy(i) > 0 ? 8u : 0u) |
                       (cz(i) < 0 ? 16u : cz(i) > 0 ? 32u : 0u);
    return (beyond & c) != 0;
}

// force body of a node next to a wall, in one half of the planes of kz_fused:
// the stress (p_iso, grad psi) of the one-halo planes
template <class F, int NP>
struct ZAccP {
    const F* pa[3];
    const F* pb[3];
    int o1;   // 2 * NP * slot + half
    unsigned beyond;
    __device__ __forceinline__ uint8_t mask(int i) const { return beyond_wall(beyond, i) ? kWallSlot : (uint8_t)0; }
    template <int K>
    __device__ __forceinline__ F get(int i) const
    {
        const F* p = K < 2 ? pa[1 + cz(i)] : pb[1 + cz(i)];
        return p[o1 + 2 * NP * poff<kZ1X>(i) + (K & 1) * NP];
    }
};

// transport body of a node next to a wall: psi, phi, mu_psi, mu_phi, u of the
// one-halo planes of kz_scalars
template <class F>
struct ZAccS {
    const F (*g[3])[2];
    const F (*mu[3])[2];
    const F (*u[3])[kZ1];
    int s1;
    unsigned beyond;
    __device__ __forceinline__ uint8_t mask(int i) const { return beyond_wall(beyond, i) ? kWallSlot : (uint8_t)0; }
    template <int K>
    __device__ __forceinline__ F get(int i) const
    {
        const int p = 1 + cz(i), s = s1 + poff<kZ1X>(i);
        return K < 2 ? g[p][s][K] : K < 4 ? mu[p][s][K - 2] : u[p][K < 4 ? 0 : K - 4][s];
    }
};

// ---------------------------------------------------------------------------
// asynchronous global -> shared copies (cp.async): the copy engine writes the
// shared-memory ring directly, so a staged plane costs no registers and its
// latency is hidden behind the planes computed meanwhile
// ---------------------------------------------------------------------------
template <int B>
__device__ __forceinline__ void cp_async(void* sdst, const void* gsrc, bool valid)
{
    static_assert(B == 4 || B == 8 || B == 16, "4-, 8- or 16-byte copies");
    const unsigned s = (unsigned)__cvta_generic_to_shared(sdst);
    // src-size 0 writes zeros and reads nothing (a slot beyond a wall)
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(s), "l"(gsrc), "n"(B),
                 "r"(valid ? B : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Columns (x + nx y) of this thread's staging slots, fixed for the whole
// march: cps for the two-halo psi slots, cph for the one-halo phi slots;
// -1 for a column beyond a wall or a slot this thread does not have.
struct MuCols {
    int cps[2], cph[2];
};

__device__ __forceinline__ void mu_cols(const DevParams& P, int x0, int y0, MuCols& c)
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int s = threadIdx.x + h * kZThreads;
        c.cps[h] = -1;
        c.cph[h] = -1;
        if (s < kZ2) {
            const int gx = zm_coord(x0, s % kZ2X - 2, P.nx, P.per[0]);
            const int gy = zm_coord(y0, s / kZ2X - 2, P.ny, P.per[1]);
            if (gx >= 0 && gy >= 0) c.cps[h] = gx + P.nx * gy;
        }
        if (s < kZ1) {
            const int gx = zm_coord(x0, s % kZ1X - 1, P.nx, P.per[0]);
            const int gy = zm_coord(y0, s / kZ1X - 1, P.ny, P.per[1]);
            if (gx >= 0 && gy >= 0) c.cph[h] = gx + P.nx * gy;
        }
    }
}

// Issue the copies of psi (two-halo slots) and phi (one-halo slots) of plane
// p (of half h) into ring slots rpsi, rphi.  kQuiet: no column or plane lies
// beyond a wall.
template <class F, int NP, bool kQuiet>
__device__ __forceinline__ void mu_plane_async(const DevParams& P, const DevPtrs& D, const MuCols& c, int p, int h,
                                               FusedSmem<F, NP>& sm, int rpsi, int rphi)
{
    const int gz = wrap_coord(p, P.nz, P.per[2]);
    const int base = !kQuiet && gz < 0 ? 0 : gz * P.nx * P.ny;
    const F* psi = (const F*)D.psi_src;
    const F* phi = (const F*)D.phi_src;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int s = threadIdx.x + k * kZThreads;
        if (k == 0 || s < kZ2) {
            const bool ok = kQuiet || (c.cps[k] >= 0 && gz >= 0);
            cp_async<(int)sizeof(F)>(&sm.psi[rpsi][s][h], psi + (base + (ok ? c.cps[k] : 0)), ok);
        }
        if (k == 0 || s < kZ1) {
            const bool ok = kQuiet || (c.cph[k] >= 0 && gz >= 0);
            cp_async<(int)sizeof(F)>(&sm.phi[rphi][s][h], phi + (base + (ok ? c.cph[k] : 0)), ok);
        }
    }
}

// What the one-halo slots of plane p hold: kind of this thread's slots.
enum : uint8_t { kFree = 0, kNextTo = 1, kSolid = 2 };   // fluid; next to a particle; not fluid
__device__ __forceinline__ uint8_t slot_kind(const DevPtrs& D, int n)
{
    const uint8_t m = D.mask[n], b = D.bflag[n];
    return m ? kSolid : (b ? kNextTo : kFree);
}

template <int NP>
struct MuKind {
    uint8_t k[2][NP];
};

template <int NP>
__device__ __forceinline__ void mu_kind_fetch(const DevParams& P, const DevPtrs& D, const MuCols& c, int p, int h,
                                              MuKind<NP>& M)
{
    const int gz = wrap_coord(p, P.nz, P.per[2]);
    const int base = gz * P.nx * P.ny;
#pragma unroll
    for (int k = 0; k < 2; ++k) M.k[k][h] = (c.cph[k] >= 0 && gz >= 0) ? slot_kind(D, base + c.cph[k]) : (uint8_t)kSolid;
}

// Transport planes: columns (x + nx y) of this thread's one-halo slots,
// fixed for the march (-1: beyond a wall, or no slot).
struct ScalCols {
    int c[2];
};

__device__ __forceinline__ void scal_cols(const DevParams& P, int x0, int y0, ScalCols& c)
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int s = threadIdx.x + h * kZThreads;
        c.c[h] = -1;
        if (s < kZ1) {
            const int gx = zm_coord(x0, s % kZ1X - 1, P.nx, P.per[0]);
            const int gy = zm_coord(y0, s / kZ1X - 1, P.ny, P.per[1]);
            if (gx >= 0 && gy >= 0) c.c[h] = gx + P.nx * gy;
        }
    }
}

// Planes per z chunk of a launch with gridDim.z chunks.
__host__ __device__ __forceinline__ int zm_chunk(int nz, int chunks) { return (nz + chunks - 1) / chunks; }

// ---------------------------------------------------------------------------
// kz_fused
// ---------------------------------------------------------------------------
// What bounds the fused kernel is instruction issue, so its two bodies are
// written for few instructions (256^3, eight spheres, FP32):
//   - a thread works on two nodes, one in each half of the block's z chunk
//     (packed FP32 arithmetic, one set of column offsets for both, 64- and
//     128-bit shared loads of the halves side by side);
//   - the 19-point stencils are summed plane by plane.  A stress plane's
//     contributions to the force of the plane below, its own and the one above
//     are formed from nine neighbours once and carried in registers (ForceSums),
//     instead of 18 neighbours and 18 products P . c per node;
//   - the collision uses the quadratic form cu (a cu + b cF) of a direction as
//     the components of one symmetric tensor per node.
// A node next to a particle or a wall takes the general body for its mu and
// stress (mup_values, from global memory), one next to a wall the general
// force body (fdiv_values); a node next to a particle is collided by
// k_collide_particles.  The form a node takes depends on the node alone, so
// every chunk length gives the same bits.

// This thread's stage-1 slots (mu and the stress of the 34 x 10 columns of a
// plane), fixed for the whole march: the slot in the two-halo plane, and the
// column x + nx y where mu is written (-1: a halo column, another block's).
struct MuSlots {
    int s2[2], wcol[2];
};

__device__ __forceinline__ void mu_slots(const DevParams& P, int x0, int y0, MuSlots& m)
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int q = threadIdx.x + h * kZThreads;
        const int lx = q % kZ1X - 1, ly = q / kZ1X - 1;
        m.s2[h] = (lx + 2) + kZ2X * (ly + 2);
        m.wcol[h] = (q < kZ1 && lx >= 0 && lx < kZX && ly >= 0 && ly < kZY && x0 + lx < P.nx && y0 + ly < P.ny)
                        ? (x0 + lx) + P.nx * (y0 + ly)
                        : -1;
    }
}

// mu and the stress of clear nodes (mu_pressure, every neighbour fluid) from
// three psi planes: the same sums of differences, taken plane by plane.
template <class R, int NP>
__device__ __forceinline__ void mu_clear(const PrmR<R>& Q, const R* pm, const R* p0, const R* pp, int s2,
                                         Vec<R, NP> phi, Vec<R, NP> dps, Vec<R, NP> dph, bool want_p,
                                         Vec<R, NP>& mps, Vec<R, NP>& mph, Vec<R, NP> (&pt)[kPtFields])
{
    using V = Vec<R, NP>;
    auto ld = [&](const R* p, int d) { return *reinterpret_cast<const V*>(p + NP * (s2 + d)); };
    constexpr int Y = kZ2X;
    const V o = ld(p0, 0);
    // the plane itself: axis and diagonal neighbours
    const V xp = ld(p0, 1), xm = ld(p0, -1), yp = ld(p0, Y), ym = ld(p0, -Y);
    const V gxa = xp - xm, gya = yp - ym;
    const V a4 = ((xp - o) + (xm - o)) + ((yp - o) + (ym - o));
    const V q1 = ld(p0, 1 + Y), q2 = ld(p0, -1 - Y), q3 = ld(p0, 1 - Y), q4 = ld(p0, -1 + Y);
    const V e = q1 - q2, f = q3 - q4;
    const V d4 = ((q1 - o) + (q2 - o)) + ((q3 - o) + (q4 - o));
    // the planes above and below: the node's own column and four diagonals
    const V su = ld(pp, 0) - o, sd = ld(pm, 0) - o;
    const V uxp = ld(pp, 1), uxm = ld(pp, -1), uyp = ld(pp, Y), uym = ld(pp, -Y);
    const V lxp = ld(pm, 1), lxm = ld(pm, -1), lyp = ld(pm, Y), lym = ld(pm, -Y);
    const V up4 = ((uxp - o) + (uxm - o)) + ((uyp - o) + (uym - o));
    const V lo4 = ((lxp - o) + (lxm - o)) + ((lyp - o) + (lym - o));
    const V sa = a4 + (su + sd), sdg = d4 + (up4 + lo4);
    const V lap = vfma((R)(1.0 / 3.0), sa, (R)(1.0 / 6.0) * sdg);
    const V gxd = (e + f) + ((uxp - uxm) + (lxp - lxm));
    const V gyd = (e - f) + ((uyp - uym) + (lyp - lym));
    const V gzd = up4 - lo4;
    const V g0 = vfma((R)(1.0 / 6.0), gxa, (R)(1.0 / 12.0) * gxd);
    const V g1 = vfma((R)(1.0 / 6.0), gya, (R)(1.0 / 12.0) * gyd);
    const V g2 = vfma((R)(1.0 / 6.0), su - sd, (R)(1.0 / 12.0) * gzd);
    const V ps = o + dps, ph = phi + dph;
    const V t = vfma(ps, ps, V::of((R)-1));   // psi^2 - 1
    V dphi;
    if (Q.E != (R)0) {
        V th;
#pragma unroll
        for (int h = 0; h < NP; ++h) th.set(h, tanh_r(ps.lane(h)));
        dphi = ph - vfma(Q.E, th, V::of(Q.phib));
        mps = (Q.A * ps) * t - Q.kappa * lap - ((Q.C * Q.E) * dphi) * (V::of((R)1) - th * th);
    } else {
        dphi = ph - V::of(Q.phib);
        mps = (Q.A * ps) * t - Q.kappa * lap;
    }
    mph = Q.C * dphi;
    if (!want_p) return;
    const V fs = vfma(((R)0.25 * Q.A) * t, t, ((R)0.5 * mph) * dphi);   // f + A/4
    const V gg = vfma(g0, g0, vfma(g1, g1, g2 * g2));
    pt[0] = vfma(ps, mps, ph * mph) - vfma((R)0.5 * Q.kappa, gg, fs);   // less A/4
    pt[1] = g0;
    pt[2] = g1;
    pt[3] = g2;
}

// Store the stress of slot q (half h) and mu of its node n (n < 0: another
// block's, or a plane of another chunk).
template <class R, class F, int NP>
__device__ __forceinline__ void mu_put(const DevPtrs& D, FusedSmem<F, NP>& sm, bool thermo, int rt, int q, int h, int n,
                                       R mps, R mph, const R (&pt)[kPtFields])
{
    if (thermo) {
        sm.pa[rt][q][h] = (F)pt[0];
        sm.pa[rt][q][NP + h] = (F)pt[1];
        sm.pb[rt][q][h] = (F)pt[2];
        sm.pb[rt][q][NP + h] = (F)pt[3];
    }
    if (n >= 0) ((Two<F>*)D.mu)[n] = {(F)mps, (F)mph};
}

// Stage 1 of one plane per half (zs): mu and the stress of the 34 x 10
// columns, two slots per thread; mu is written for the tile's own columns
// where own.  Bit h of gen: half h may hold nodes next to particles or walls,
// kind says where.  Those are listed and then shared out over the block, one
// per thread: the general body is a chain of loads and an inverse square root
// per link, and a warp that held a few such nodes in each of its slots and
// halves would run it four times over (24^3, one sphere R = 3: 52 us with the
// general body in place).
template <class C, int NP, bool kQuiet>
__device__ __forceinline__ void fused_stage1(const DevParams& P, const DevPtrs& D,
                                             FusedSmem<typename C::fld_t, NP>& sm, const MuSlots& ms, int x0, int y0,
                                             const int (&zs)[NP], const bool (&own)[NP], const int (&rp)[3], int rf,
                                             int rt, Vec<typename C::real, NP> dps, Vec<typename C::real, NP> dph,
                                             unsigned gen, const MuKind<NP>& kind, int odd)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    using V = Vec<R, NP>;
    const PrmR<R>& Q = prm<R>(P);
    const int sxy = P.nx * P.ny;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        const int q = threadIdx.x + k * kZThreads;
        if (k == 1 && q >= kZ1) break;
        const int s2 = k == 0 ? ms.s2[0] : ms.s2[1];
        const int wcol = k == 0 ? ms.wcol[0] : ms.wcol[1];
        V mps, mph, pt[kPtFields];
        mu_clear<R, NP>(Q, &sm.psi[rp[0]][0][0], &sm.psi[rp[1]][0][0], &sm.psi[rp[2]][0][0], s2,
                        *reinterpret_cast<const V*>(&sm.phi[rf][q][0]), dps, dph, P.thermo != 0, mps, mph, pt);
        unsigned skip = 0;
        if (!kQuiet && gen) {
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                if (!(gen >> h & 1u)) continue;
                const uint8_t kd = k == 0 ? kind.k[0][h] : kind.k[1][h];
                bool todo = kd == kNextTo;
                if (kd == kFree)
                    todo = near_wall(P, zm_coord(x0, q % kZ1X - 1, P.nx, P.per[0]),
                                     zm_coord(y0, q / kZ1X - 1, P.ny, P.per[1]), wrap_coord(zs[h], P.nz, P.per[2]));
                if (todo) sm.todo[atomicAdd(&sm.ntodo[odd], 1)] = (uint16_t)(NP * q + h);
                if (todo || kd == kSolid) skip |= 1u << h;
            }
        }
        if (P.thermo) {
            V* pa = reinterpret_cast<V*>(&sm.pa[rt][q][0]);
            V* pb = reinterpret_cast<V*>(&sm.pb[rt][q][0]);
            pa[0] = pt[0];
            pa[1] = pt[1];
            pb[0] = pt[2];
            pb[1] = pt[3];
        }
        if (wcol >= 0) {
#pragma unroll
            for (int h = 0; h < NP; ++h)
                if (own[h] && (kQuiet || !(skip >> h & 1u))) {
                    const int n = wcol + sxy * zs[h];
                    ((Two<F>*)D.mu)[n] = {(F)mps.lane(h), (F)mph.lane(h)};
                }
        }
    }
    if (kQuiet || !gen) return;
    __syncthreads();
    const int nt = sm.ntodo[odd];
#pragma unroll 1
    for (int i = threadIdx.x; i < nt; i += kZThreads) {
        const int e = sm.todo[i], h = e % NP, q = e / NP;
        const int lx = q % kZ1X - 1, ly = q / kZ1X - 1;
        const int zp = h == 0 ? zs[0] : zs[NP - 1];
        const int x = zm_coord(x0, lx, P.nx, P.per[0]), y = zm_coord(y0, ly, P.ny, P.per[1]);
        const int z = wrap_coord(zp, P.nz, P.per[2]);
        ZAccMu<F, NP> a;
        neighbours(P, x, y, z, a.nb);
        a.mk = D.mask;
#pragma unroll
        for (int j = 0; j < 3; ++j) a.ps[j] = &sm.psi[rp[j]][0][0];
        a.o2 = NP * ((lx + 2) + kZ2X * (ly + 2)) + h;
        a.phi_own = sm.phi[rf][q][h];
        a.gp = &sm.ghost;
        R m1, m2, p4[kPtFields];
        mup_values<C>(P, D, x, y, z, a, dps.lane(0), dph.lane(0), m1, m2, p4);
        const bool put = (h == 0 ? own[0] : own[NP - 1]) && lx >= 0 && lx < kZX && ly >= 0 && ly < kZY &&
                         x0 + lx < P.nx && y0 + ly < P.ny;
        mu_put<R, F, NP>(D, sm, P.thermo != 0, rt, q, h, put ? (x0 + lx) + P.nx * (y0 + ly) + sxy * zp : -1, m1, m2,
                         p4);
    }
}

// The force of a clear node in the link form, -3 sum_i w_i P(x + c_i) . c_i,
// summed plane by plane (weights 2 on axis links and 1 on diagonal ones, 1/36
// in the end).  With the sums over a plane, of P at the node's neighbours there,
//   U = sum over the axis neighbours of P . c,   Q = the same of P . e_z,
//   V = sum over the diagonal neighbours of P . c,   Z = P . e_z at the node's
// column, plane q adds 2 Z + U + Q to the node below, 2 U + V to its own node
// and -2 Z + U - Q to the node above.  prev: what the plane below last seen
// still lacks one plane of; next: what the node above the last plane has.
template <class R, int NP>
struct ForceSums {
    Vec<R, NP> prev[3], next[3];
};

// Take in the stress plane (pa, pb); returns the finished sums of the plane
// below in out.
template <class R, int NP>
__device__ __forceinline__ void force_plane(const R* pa, const R* pb, int s1, R kappa, ForceSums<R, NP>& c,
                                            Vec<R, NP> (&out)[3])
{
    using V = Vec<R, NP>;
    struct alignas(2 * NP * sizeof(R)) V2 {
        V a, b;
    };
    constexpr int Y = kZ1X;
    auto la = [&](int d) { return *reinterpret_cast<const V2*>(pa + 2 * NP * (s1 + d)); };   // p, gx
    auto lb = [&](int d) { return *reinterpret_cast<const V2*>(pb + 2 * NP * (s1 + d)); };   // gy, gz
    V U[3], Q[3], W[3];
    {   // +x, -x
        const V2 a = la(1), b = lb(1), d = la(-1), e = lb(-1);
        const V kp = kappa * a.b, km = kappa * d.b, zp = kappa * b.b, zm = kappa * e.b;
        const V xzp = kp * b.b, xzm = km * e.b;
        U[0] = (a.a - d.a) + (kp * a.b - km * d.b);
        U[1] = kp * b.a - km * e.a;
        U[2] = xzp - xzm;
        Q[0] = xzp + xzm;
        Q[1] = vfma(zp, b.a, zm * e.a);
        Q[2] = (a.a + d.a) + vfma(zp, b.b, zm * e.b);
    }
    {   // +y, -y
        const V2 a = la(Y), b = lb(Y), d = la(-Y), e = lb(-Y);
        const V kp = kappa * b.a, km = kappa * e.a, zp = kappa * b.b, zm = kappa * e.b;
        const V yzp = kp * b.b, yzm = km * e.b;
        U[0] = U[0] + (kp * a.b - km * d.b);
        U[1] = U[1] + ((a.a - d.a) + (kp * b.a - km * e.a));
        U[2] = U[2] + (yzp - yzm);
        Q[0] = Q[0] + vfma(zp, a.b, zm * d.b);
        Q[1] = Q[1] + (yzp + yzm);
        Q[2] = Q[2] + ((a.a + d.a) + vfma(zp, b.b, zm * e.b));
    }
    {   // (1, 1), (-1, -1)
        const V2 a = la(1 + Y), b = lb(1 + Y), d = la(-1 - Y), e = lb(-1 - Y);
        const V sp = kappa * (a.b + b.a), sm = kappa * (d.b + e.a), dp = a.a - d.a;
        W[0] = dp + (sp * a.b - sm * d.b);
        W[1] = dp + (sp * b.a - sm * e.a);
        W[2] = sp * b.b - sm * e.b;
    }
    {   // (1, -1), (-1, 1)
        const V2 a = la(1 - Y), b = lb(1 - Y), d = la(-1 + Y), e = lb(-1 + Y);
        const V sp = kappa * (a.b - b.a), sm = kappa * (d.b - e.a), dp = a.a - d.a;
        W[0] = W[0] + (dp + (sp * a.b - sm * d.b));
        W[1] = W[1] + ((sp * b.a - sm * e.a) - dp);
        W[2] = W[2] + (sp * b.b - sm * e.b);
    }
    const V2 a = la(0), b = lb(0);
    const V kz = kappa * b.b;
    const V Z[3] = {kz * a.b, kz * b.a, vfma(kz, b.b, a.a)};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        out[k] = c.prev[k] + vfma((R)2, Z[k], U[k] + Q[k]);
        c.prev[k] = vfma((R)2, U[k], c.next[k] + W[k]);
        c.next[k] = vfma((R)-2, Z[k], U[k] - Q[k]);
    }
}

// BGK collision with Guo forcing of NP nodes, with the
// populations of a weight class scaled by its weight: for c of diagonal
// weight w, g* = (1 - 1/tau) g + (T_c + e) +- h.c with
//   T_c = cu (c.v), v = w (4.5 rho u / tau + 9 (1 - 1/(2 tau)) F),
//   h   = w (3 rho u / tau + 3 (1 - 1/(2 tau)) F),
//   e   = w [(rho - rho0 - 1.5 rho u^2) / tau - 3 (1 - 1/(2 tau)) u.F],
// twice that for axis directions and 12 e for the rest one.  T_c of the six
// axes and planes comes from the products u_a v_b.  g becomes g*.
template <class R, int NP>
__device__ __forceinline__ void collide_values(const PrmR<R>& Q, Vec<R, NP> (&g)[19], const Vec<R, NP> (&F)[3],
                                               Vec<R, NP> (&u)[3])
{
    using V = Vec<R, NP>;
    // moments from the sums and differences of opposite pairs
    V m[9], dr = g[0];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        m[k] = g[2 * k + 1] - g[2 * k + 2];
        dr = dr + (g[2 * k + 1] + g[2 * k + 2]);
    }
    const V jx = (m[0] + (m[3] + m[4])) + (m[5] + m[6]);
    const V jy = (m[1] + (m[3] - m[4])) + (m[7] + m[8]);
    const V jz = (m[2] + (m[5] - m[6])) + (m[7] - m[8]);
    const V rho = V::of(Q.rho0) + dr;
    const V ir = recip(rho);
    u[0] = vfma((R)0.5, F[0], jx) * ir;
    u[1] = vfma((R)0.5, F[1], jy) * ir;
    u[2] = vfma((R)0.5, F[2], jz) * ir;
    const R itau = Q.itau, omf = Q.omf, keep = (R)1 - itau, w = wgt_r<R>(7);
    const V uu = vfma(u[0], u[0], vfma(u[1], u[1], u[2] * u[2]));
    const V uF = vfma(u[0], F[0], vfma(u[1], F[1], u[2] * F[2]));
    const V ri = (w * itau) * rho;
    const V e = vfma((R)-3 * w * omf, uF, vfma((R)-1.5 * ri, uu, (w * itau) * dr));
    const V av = (R)4.5 * ri, ah = (R)3 * ri;
    V v[3], h[3], T[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        v[a] = vfma((R)9 * w * omf, F[a], av * u[a]);
        h[a] = vfma((R)3 * w * omf, F[a], ah * u[a]);
        T[a] = u[a] * v[a];
    }
    g[0] = vfma(keep, g[0], (R)12 * e);
#pragma unroll
    for (int a = 0; a < 3; ++a) {   // +-x, +-y, +-z
        const int j = 2 * a + 1;
        const V pe = T[a] + e, pp = pe + h[a], pm = pe - h[a];
        g[j] = vfma(keep, g[j], pp + pp);
        g[j + 1] = vfma(keep, g[j + 1], pm + pm);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {   // the planes xy, xz, yz: (a, b), -(a, b), (a, -b), -(a, -b)
        const int a = k == 2 ? 1 : 0, b = k == 0 ? 1 : 2, j = 7 + 4 * k;
        const V base = (T[a] + T[b]) + e, S = vfma(u[a], v[b], u[b] * v[a]);
        const V pp = base + S, pm = base - S, hp = h[a] + h[b], hm = h[a] - h[b];
        g[j] = vfma(keep, g[j], pp + hp);
        g[j + 1] = vfma(keep, g[j + 1], pp - hp);
        g[j + 2] = vfma(keep, g[j + 2], pm + hm);
        g[j + 3] = vfma(keep, g[j + 3], pm - hm);
    }
}

// What a thread of kz_fused keeps about its column.
struct FusedCol {
    int x, y, nxy;         // coordinates, x + nx y
    int xo[3], yo[3];      // x - 1, x, x + 1 and nx (y - 1, y, y + 1), wrapped or clamped
    bool in;               // inside the box
    unsigned beyond;       // walls next to it in x and y (as ZAccP::beyond)
};

__device__ __forceinline__ void fused_col(const DevParams& P, int x0, int y0, FusedCol& c)
{
    const int nx = P.nx, ny = P.ny;
    const int x = x0 + (int)(threadIdx.x & (kZX - 1)), y = y0 + (int)threadIdx.x / kZX;
    c.x = x;
    c.y = y;
    c.in = x < nx && y < ny;
    c.nxy = x + nx * y;
    c.beyond = (!P.per[0] ? (x == 0 ? 1u : 0u) | (x == nx - 1 ? 2u : 0u) : 0u) |
               (!P.per[1] ? (y == 0 ? 4u : 0u) | (y == ny - 1 ? 8u : 0u) : 0u);
    c.xo[0] = x > 0 ? x - 1 : (P.per[0] ? nx - 1 : 0);
    c.xo[1] = x;
    c.xo[2] = x < nx - 1 ? x + 1 : (P.per[0] ? 0 : x);
    c.yo[0] = (y > 0 ? y - 1 : (P.per[1] ? ny - 1 : 0)) * nx;
    c.yo[1] = y * nx;
    c.yo[2] = (y < ny - 1 ? y + 1 : (P.per[1] ? 0 : y)) * nx;
}

// Stage 2 of one plane per half (zs, valid where val): every pull load of the
// nodes first, then the force from the stress plane above (rt[2], just
// computed) while they are in flight, then the collide-stream.  Bit h of gen:
// half h may hold solid nodes, nodes next to particles (left to
// k_collide_particles) or nodes next to walls.
template <class C, int NP, bool kQuiet>
__device__ __forceinline__ void fused_stage2(const DevParams& P, const DevPtrs& D,
                                             const FusedSmem<typename C::fld_t, NP>& sm, const FusedCol& col,
                                             const int (&zs)[NP], const bool (&val)[NP], bool emit,
                                             const int (&rt)[3], unsigned gen,
                                             ForceSums<typename C::real, NP>& fs)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    using S = typename C::pop_t;
    using V = Vec<R, NP>;
    const PrmR<R>& Q = prm<R>(P);
    const int tx = threadIdx.x & (kZX - 1), ty = threadIdx.x / kZX;
    const int s1 = (tx + 1) + kZ1X * (ty + 1);
    if (!col.in) return;
    V fl[19];
    const int sxy = P.nx * P.ny;
    const int NN = (int)P.N;   // 19 N < 2^31: one index addition per access
    const S* fs_ = (const S*)D.f_src;
    S* fd = (S*)D.f_dst;
    if (emit) {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            const int z = min(zs[h], P.nz - 1);   // a half past its last plane loads something valid
            const int zo[3] = {(z > 0 ? z - 1 : (P.per[2] ? P.nz - 1 : 0)) * sxy, z * sxy,
                               (z < P.nz - 1 ? z + 1 : (P.per[2] ? 0 : z)) * sxy};
#pragma unroll
            for (int j = 0; j < 19; ++j) {
                const int m = col.xo[1 - cx(j)] + col.yo[1 - cy(j)] + zo[1 - cz(j)];
                fl[j].set(h, (R)PopStore<S>::load_dev(fs_, j * NN + m, j, Q.rho0));
            }
        }
    }
    bool put[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        put[h] = val[h];
        if (!kQuiet && emit && val[h] && (gen >> h & 1u)) put[h] = slot_kind(D, col.nxy + sxy * zs[h]) == kFree;
    }
    V f3[3];
    if (P.thermo) {
        V sum[3];
        force_plane<R, NP>(&sm.pa[rt[2]][0][0], &sm.pb[rt[2]][0][0], s1, Q.kappa, fs, sum);
#pragma unroll
        for (int k = 0; k < 3; ++k) f3[k] = vfma((R)(-1.0 / 12.0), sum[k], V::of(Q.g[k]));
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) f3[k] = V::of(Q.g[k]);
    }
    if (!emit) return;
    if (!kQuiet && gen) {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            const unsigned zw = !P.per[2] ? (zs[h] == 0 ? 16u : 0u) | (zs[h] == P.nz - 1 ? 32u : 0u) : 0u;
            if (!put[h] || !(col.beyond | zw)) continue;
            ZAccP<F, NP> a;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                a.pa[k] = &sm.pa[rt[k]][0][0];
                a.pb[k] = &sm.pb[rt[k]][0][0];
            }
            a.o1 = 2 * NP * s1 + h;
            a.beyond = col.beyond | zw;
            R Fx, Fy, Fz;
            fdiv_values<C>(P, a, Fx, Fy, Fz);
            f3[0].set(h, Fx);
            f3[1].set(h, Fy);
            f3[2].set(h, Fz);
            R one[19];
#pragma unroll
            for (int j = 0; j < 19; ++j) one[j] = fl[j].lane(h);
            bulk_wall_links<C>(P, D, col.x, col.y, zs[h], one);
#pragma unroll
            for (int j = 0; j < 19; ++j) fl[j].set(h, one[j]);
        }
    }
    V u[3];
    collide_values<R, NP>(Q, fl, f3, u);
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        if (!put[h]) continue;
        const int n = col.nxy + sxy * zs[h];
#pragma unroll
        for (int j = 0; j < 19; ++j) PopStore<S>::store_dev(fd, j * NN + n, j, Q.rho0, fl[j].lane(h));
        F* uo = (F*)D.u;
#pragma unroll
        for (int k = 0; k < 3; ++k) uo[k * NN + n] = (F)u[k].lane(h);
    }
}

// ring position advanced by one
template <int N>
__device__ __forceinline__ int ring_next(int r)
{
    return r + 1 == N ? 0 : r + 1;
}

// Resident blocks per SM the fused kernel is compiled for: two (128
// registers), 512 threads with two nodes each in FP32 and one in FP64.
template <class C>
constexpr int fused_blocks_per_sm()
{
    return 2;
}

// The march of one block: columns x0 .. x0 + 31, y0 .. y0 + 7, planes
// z0 .. z0 + nt - 1 (nt >= 1) in NP halves of na planes (the last one may be
// a plane short, or empty).  kQuiet: every plane the block stages is clear, so
// the loop holds no flag, no general body and no wall.
template <class C, bool kQuiet>
__device__ __forceinline__ void fused_march(const DevParams& P, const DevPtrs& D, int x0, int y0, int z0, int nt,
                                            bool xywall, FusedSmem<typename C::fld_t, zm_halves<typename C::real>()>& sm)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    constexpr int NP = zm_halves<R>();
    using V = Vec<R, NP>;
    const int na = (nt + NP - 1) / NP;
    int zh[NP], nh[NP];   // first plane and number of planes of each half
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        zh[h] = z0 + h * na;
        nh[h] = h == 0 ? na : nt - na;
    }
    MuCols cols;
    mu_cols(P, x0, y0, cols);
    MuSlots ms;
    mu_slots(P, x0, y0, ms);
    FusedCol col;
    fused_col(P, x0, y0, col);
    const V dps = V::of(corr_r<R>(D, 0)), dph = V::of(corr_r<R>(D, 1));
    // Ring slots: psi of plane p at (p - zh + 2) mod 5, phi at (p - zh + 2)
    // mod 4, the stress at (p - zh + 1) mod 4.  Iteration t computes the
    // stress of plane zh + t - 1 (stage 1), issues the copies of psi/phi of
    // zh + t + 2, waits for those of zh + t + 1, and collides plane zh + t - 2
    // (stage 2).  With these ring depths the one barrier per iteration orders
    // every write of a slot after the last read of the plane it held.  Bit k
    // of win[h] in iteration t: plane zh + t + 1 - k is not clear.
    unsigned win[NP];
    MuKind<NP> K;   // the slots of plane zh + t - 1
    if (!kQuiet) {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            win[h] = 0;
            for (int k = -2; k < 1; ++k) win[h] = (win[h] << 1) | (unsigned)plane_solid(P, sm.sol, xywall, zh[h] + k);
            if (win[h]) mu_kind_fetch<NP>(P, D, cols, zh[h] - 1, h, K);
        }
    }
#pragma unroll
    for (int h = 0; h < NP; ++h)
        for (int k = 0; k < 3; ++k) mu_plane_async<F, NP, kQuiet>(P, D, cols, zh[h] - 2 + k, h, sm, k, k);
    cp_async_commit();
#pragma unroll
    for (int h = 0; h < NP; ++h) mu_plane_async<F, NP, kQuiet>(P, D, cols, zh[h] + 1, h, sm, 3, 3);
    cp_async_commit();
    if (threadIdx.x == 0) sm.ntodo[0] = 0;
    cp_async_wait<1>();
    __syncthreads();
    ForceSums<R, NP> fs;
#pragma unroll
    for (int k = 0; k < 3; ++k) fs.prev[k] = fs.next[k] = V::of((R)0);
    // rp0: psi slot of plane zh + t - 2; rf: phi slot of zh + t - 1; rt0:
    // stress slot of zh + t - 1
    int rp0 = 0, rf = 1, rt0 = 0;
#pragma unroll 1
    for (int t = 0; t <= na + 1; ++t) {
        const int rpa = ring_next<kPsiRing>(rp0), rpb = ring_next<kPsiRing>(rpa), rpc = ring_next<kPsiRing>(rpb);
        const int rpd = ring_next<kPsiRing>(rpc);
        unsigned gen1 = 0, gen2 = 0;
        int z1[NP], z2[NP];
        bool own[NP], val[NP];
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            if (!kQuiet) {
                win[h] = (win[h] << 1) | (unsigned)plane_solid(P, sm.sol, xywall, zh[h] + t + 1);
                gen1 |= (win[h] & 0x0Eu) ? 1u << h : 0u;   // planes t - 2 .. t
                gen2 |= (win[h] & 0x1Cu) ? 1u << h : 0u;   // planes t - 3 .. t - 1
            }
            z1[h] = zh[h] + t - 1;
            z2[h] = zh[h] + t - 2;
            own[h] = t >= 1 && t <= nh[h];
            val[h] = t >= 2 && t - 2 < nh[h];
        }
        const int rp1[3] = {rp0, rpa, rpb};   // planes zh + t - 2 .. zh + t
        fused_stage1<C, NP, kQuiet>(P, D, sm, ms, x0, y0, z1, own, rp1, rf, rt0, dps, dph, gen1, K, t & 1);
        if (!kQuiet && threadIdx.x == 0) sm.ntodo[(t & 1) ^ 1] = 0;
        if (t + 2 <= na + 1) {                             // zh + t + 2
            const int rfd = rf < 1 ? rf + 3 : rf - 1;       // its phi slot
#pragma unroll
            for (int h = 0; h < NP; ++h)
                mu_plane_async<F, NP, kQuiet>(P, D, cols, zh[h] + t + 2, h, sm, rpd, rfd);
        }
        if (!kQuiet) {   // planes t - 1 .. t + 1 decide what the slots of zh + t are
#pragma unroll
            for (int h = 0; h < NP; ++h)
                if (win[h] & 0x07u) mu_kind_fetch<NP>(P, D, cols, zh[h] + t, h, K);
        }
        cp_async_commit();
        cp_async_wait<1>();   // this thread's copies of plane zh + t + 1 have landed
        __syncthreads();
        const int rt2[3] = {rt0 < 2 ? rt0 + 2 : rt0 - 2, rt0 == 0 ? kPtRing - 1 : rt0 - 1, rt0};
        fused_stage2<C, NP, kQuiet>(P, D, sm, col, z2, val, t >= 2, rt2, gen2, fs);
        rp0 = rpa;
        rf = ring_next<kPhiRing>(rf);
        rt0 = ring_next<kPtRing>(rt0);
    }
    cp_async_wait<0>();
}

// One block of kz_fused, smem of fused_smem_bytes<C>() bytes.
template <class C>
__device__ __forceinline__ void kz_fused_run(const DevParams& P, const DevPtrs& D, int x0, int y0, int z0, int nt,
                                             unsigned char* smem_raw)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    constexpr int NP = zm_halves<R>();
    static_assert(sizeof(R) == sizeof(F), "the staged planes are read as arithmetic vectors");
    FusedSmem<F, NP>& sm = *reinterpret_cast<FusedSmem<F, NP>*>(smem_raw);
    find_solids<false>(P, D, x0, y0, 2, sm.sol, [&](int k, int i, const DevPart& q) {
        sm.ghost.slot[k] = (uint8_t)i;
        sm.ghost.geo[i].g = q.g;
        sm.ghost.geo[i].Hk = q.Hk;
        sm.ghost.geo[i].Hk_f = q.Hk_f;
    });
    const bool xywall = beyond_xy(P, x0, y0, 2);
    // planes any iteration looks at: z0 - 2 .. z0 + NP na + 1
    bool quiet = !xywall && (P.per[2] || (z0 >= 2 && z0 + nt + NP + 1 <= P.nz));
    for (int i = 0; i < sm.sol.n; ++i)
        quiet = quiet && !spans_meet(sm.sol.lo[i], sm.sol.len[i], z0 - 2, nt + NP + 3, P.nz, P.per[2]);
    if (quiet)
        fused_march<C, true>(P, D, x0, y0, z0, nt, xywall, sm);
    else
        fused_march<C, false>(P, D, x0, y0, z0, nt, xywall, sm);
}

template <class C>
constexpr size_t fused_smem_bytes()
{
    return sizeof(FusedSmem<typename C::fld_t, zm_halves<typename C::real>()>);
}

// Single box: grid (column tiles in x, in y, z chunks).
template <class C>
__global__ void __launch_bounds__(kZThreads, fused_blocks_per_sm<C>()) kz_fused(const __grid_constant__ DevParams P,
                                                                               const __grid_constant__ DevPtrs D)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];   // fused_smem_bytes<C>()
    const int zc = zm_chunk(P.nz, gridDim.z);
    const int z0 = blockIdx.z * zc;
    const int nt = min(z0 + zc, P.nz) - z0;   // planes of this chunk
    if (nt <= 0) return;                      // block-uniform
    kz_fused_run<C>(P, D, blockIdx.x * kZX, blockIdx.y * kZY, z0, nt, smem_raw);
}

// ---------------------------------------------------------------------------
// kz_scalars
// ---------------------------------------------------------------------------
// What bounds the transport is instruction issue and shared-memory bandwidth
// (18 neighbours of seven fields per node), so:
//   - the links are taken plane by plane: when plane q arrives, its eight
//     neighbours of a column are read once and serve the in-plane links of
//     plane q and the links up to it from q - 1 and down to it from q + 1
//     (ScalSums), half the reads of 18 neighbours per node;
//   - the linear parts, M lap mu and the divergence of u, are sums over a plane
//     that the three planes share; the upwind part is left with one minimum
//     and two multiply-adds per link:
//       sum_i w_i [M (mu_i - mu) - (ub g)_upwind],  b_i = c.(u + u_i) = 2 ub_i,
//       = sum_i w_i [M (mu_i - mu) - (min(b_i, 0) (g_i - g) + c.u_i g) / 2]
//     (sum_i w_i c.u = 0);
//   - the sink k_d (phi - phi0) is (k_d / C) mu_phi, which is staged already;
//   - psi and phi, and mu_psi and mu_phi, lie side by side in shared memory and
//     go through packed FP32 instructions.
// Solid nodes and those next to particles are left out, nodes next to walls
// take the general body; which form a node takes depends on the node alone.
// One node per thread and 24 warps per SM: with two nodes per thread, as in
// kz_fused, the kernel issues a fifth fewer instructions but has 16 warps and
// waits more.  Measured on GB300, eight spheres at 256^3, FP32: 344 us with 18
// neighbours per node, 328 with two nodes per thread, 250 so; FP64 96^3 549 ->
// 406 us, there by the FP64 operations saved.

// Issue the copies of the seven transport fields of plane p into ring slot r.
template <class F, bool kQuiet>
__device__ __forceinline__ void scal_plane_async(const DevParams& P, const DevPtrs& D, const ScalCols& c, int p,
                                                 ScalSmem<F>& sm, int r)
{
    const int NN = (int)P.N;
    const F* psi = (const F*)D.psi_src;
    const F* phi = (const F*)D.phi_src;
    const F* mu = (const F*)D.mu;
    const F* u = (const F*)D.u;
    const int gz = wrap_coord(p, P.nz, P.per[2]);
    const int base = !kQuiet && gz < 0 ? 0 : gz * P.nx * P.ny;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int s = threadIdx.x + k * kZThreads;
        if (k == 0 || s < kZ1) {
            const bool ok = kQuiet || (c.c[k] >= 0 && gz >= 0);
            const int g = ok ? base + c.c[k] : 0;
            cp_async<(int)sizeof(F)>(&sm.g[r][s][0], psi + g, ok);
            cp_async<(int)sizeof(F)>(&sm.g[r][s][1], phi + g, ok);
            cp_async<2 * (int)sizeof(F)>(&sm.mu[r][s][0], mu + 2 * g, ok);
#pragma unroll
            for (int a = 0; a < 3; ++a) cp_async<(int)sizeof(F)>(&sm.u[r][a][s], u + (a * NN + g), ok);
        }
    }
}

// The sums of one node over the planes seen so far, in units of the diagonal
// weight 1/36 (axis links count twice): ad = sum min(b, 0) (g_i - g) for psi
// and phi, dv = sum c.u_i, lp = sum (mu_i - mu) for both.
template <class R>
struct ScalSums {
    Two<R> ad, lp;
    R dv;
};

// A column's own psi, phi and u in one plane.
template <class R>
struct ScalOwn {
    Two<R> g;
    R u[3];
};

// One plane of the ring.
template <class R>
struct ScalPlane {
    const R (*g)[2];
    const R (*mu)[2];
    const R (*u)[kZ1];
    __device__ __forceinline__ Two<R> gp(int s) const { return *reinterpret_cast<const Two<R>*>(g[s]); }
    __device__ __forceinline__ Two<R> mp(int s) const { return *reinterpret_cast<const Two<R>*>(mu[s]); }
};
template <class F>
__device__ __forceinline__ ScalPlane<F> scal_ring(const ScalSmem<F>& sm, int r)
{
    return {sm.g[r], sm.mu[r], sm.u[r]};
}

template <class R>
__device__ __forceinline__ ScalOwn<R> scal_own(const ScalPlane<R>& f, int s)
{
    return {f.gp(s), {f.u[0][s], f.u[1][s], f.u[2][s]}};
}

// One link: b = c.(u + u_i) (minus it when kNeg) and the difference d of psi
// and phi along it, into the upwind sums.
template <bool kNeg, class R>
__device__ __forceinline__ void upwind(R b, Two<R> d, Two<R>& a)
{
    const R m = kNeg ? -max0(b) : min0(b);   // min(-b, 0) = -max(b, 0)
    a.a = fma_x(m, d.a, a.a);
    a.b = fma_x(m, d.b, a.b);
}

// Take in plane q (f): completes prev, the sums of the node below, adds the
// in-plane links to cur and starts next, the node above.  a, o, b: the
// column's own values in planes q - 1, q, q + 1; mm, m0: mu_psi, mu_phi of the
// column in planes q - 1 and q.  inner: the node of plane q is of this chunk.
template <class R>
__device__ __forceinline__ void scal_plane(const ScalPlane<R>& f, int s1, bool inner, const ScalOwn<R>& a,
                                           const ScalOwn<R>& o, const ScalOwn<R>& b, Two<R> mm, Two<R> m0,
                                           ScalSums<R>& prev, ScalSums<R>& cur, ScalSums<R>& next)
{
    constexpr int Y = kZ1X;
    // the column itself: links up from q - 1 and down from q + 1
    {
        const R bu = add_x(a.u[2], o.u[2]), bd = add_x(b.u[2], o.u[2]);
        next.ad = {0, 0};
        upwind<false>(add_x(bu, bu), sub2(o.g, a.g), prev.ad);
        upwind<true>(add_x(bd, bd), sub2(o.g, b.g), next.ad);
    }
    R e = 0, z4 = 0;             // in-plane sums over the axis neighbours
    Two<R> l4{0, 0}, ad2{0, 0};
#pragma unroll
    for (int k = 0; k < 4; ++k) {   // +x, -x, +y, -y
        const int ax = k / 2;
        const bool neg = k & 1;
        const int s = s1 + (neg ? -1 : 1) * (ax == 0 ? 1 : Y);
        const Two<R> g = f.gp(s);
        const R nu = f.u[ax][s], nz = f.u[2][s];
        l4 = add2(l4, sub2(f.mp(s), m0));
        z4 = add_x(z4, nz);
        e = neg ? add_x(e, -nu) : add_x(e, nu);
        const R bi = add_x(o.u[ax], nu);   // c.(u + u_i) in the plane, minus it on the negative side
        // c = (+-1, 0, 1) from q - 1: +-(u + u_i) + (uz + uz_i); (+-1, 0, -1) from q + 1
        const R az = add_x(a.u[2], nz), an = add_x(a.u[ax], nu), bz = add_x(b.u[2], nz), bn = add_x(b.u[ax], nu);
        if (neg) {
            upwind<true>(bi, sub2(g, o.g), ad2);
            upwind<false>(add_x(az, -an), sub2(g, a.g), prev.ad);
            upwind<true>(add_x(bz, bn), sub2(g, b.g), next.ad);
        } else {
            upwind<false>(bi, sub2(g, o.g), ad2);
            upwind<false>(add_x(az, an), sub2(g, a.g), prev.ad);
            upwind<true>(add_x(bz, -bn), sub2(g, b.g), next.ad);
        }
    }
    const R Z = fma_x((R)2, o.u[2], z4);
    const Two<R> d6 = sub2(m0, mm);
    prev.dv = add_x(prev.dv, add_x(e, Z));
    prev.lp = add2(prev.lp, fma2(Two<R>{6, 6}, d6, l4));
    next.dv = add_x(e, -Z);
    next.lp = l4;
    if (!inner) return;
    // diagonal neighbours in the plane
    const R us = add_x(o.u[0], o.u[1]), ud = add_x(o.u[0], -o.u[1]);
    R v = 0;
    Two<R> d4{0, 0};
#pragma unroll
    for (int k = 0; k < 4; ++k) {   // (1,1), (-1,-1), (1,-1), (-1,1)
        const bool neg = k & 1, anti = k >= 2;
        const int s = s1 + (neg ? -1 : 1) * (anti ? 1 - Y : 1 + Y);
        const Two<R> g = f.gp(s);
        const R nx = f.u[0][s], ny = f.u[1][s];
        d4 = add2(d4, sub2(f.mp(s), m0));
        const R cu = anti ? add_x(nx, -ny) : add_x(nx, ny);
        v = neg ? add_x(v, -cu) : add_x(v, cu);
        const R bi = add_x(anti ? ud : us, cu);
        if (neg)
            upwind<true>(bi, sub2(g, o.g), cur.ad);
        else
            upwind<false>(bi, sub2(g, o.g), cur.ad);
    }
    cur.ad = fma2(Two<R>{2, 2}, ad2, cur.ad);
    cur.dv = add_x(cur.dv, fma_x((R)2, e, v));
    cur.lp = add2(cur.lp, fma2(Two<R>{-6, -6}, d6, fma2(Two<R>{2, 2}, l4, d4)));
}

// The lattice-Boltzmann transport of a clear node (scalars_compute_lb) from
// the planes below, own and above: the increments of psi and phi less the
// correction and the sink.
template <class R>
__device__ __forceinline__ Two<R> scal_lb(const PrmR<R>& Q, const ScalPlane<R>& f0, const ScalPlane<R>& f1,
                                          const ScalPlane<R>& f2, int s1, Two<R> corr)
{
    const Two<R> m0 = f1.mp(s1);
    Two<R> l{0, 0}, ad{0, 0};
#pragma unroll
    for (int i = 1; i < 7; ++i) {
        const ScalPlane<R>& f = cz(i) == 0 ? f1 : cz(i) > 0 ? f2 : f0;
        const int s = s1 + poff<kZ1X>(i), a = cx(i) != 0 ? 0 : cy(i) != 0 ? 1 : 2;
        const R u = cx(i) + cy(i) + cz(i) < 0 ? -f.u[a][s] : f.u[a][s];
        const Two<R> g = add2(f.gp(s), corr);
        l = add2(l, sub2(f.mp(s), m0));
        ad.a = fma_x(u, g.a, ad.a);
        ad.b = fma_x(u, g.b, ad.b);
    }
    return {fma_x((R)-0.5, ad.a, mul_x(Q.Mpsi, l.a)), fma_x((R)-0.5, ad.b, mul_x(Q.Mphi, l.b))};
}

// Whether (x, y, z) is fluid and not next to a particle, from the masks of this
// step: covering replaces the boundary flags while this kernel runs.
__device__ __forceinline__ bool free_node(const DevParams& P, const DevPtrs& D, int x, int y, int z)
{
    int nb[19];
    neighbours(P, x, y, z, nb);
    unsigned any = 0;
#pragma unroll
    for (int i = 0; i < 19; ++i) any |= D.mask[nb[i] >= 0 ? nb[i] : nb[0]];
    return any == 0;
}

// The march of one block: columns x0 .. x0 + 31, y0 .. y0 + 7, planes z0 ..
// z0 + nt - 1 (nt >= 1).  kQuiet: every plane the block stages is clear.  kLB:
// the lattice-Boltzmann scheme.
template <class C, bool kQuiet, bool kLB>
__device__ __forceinline__ void scal_march(const DevParams& P, const DevPtrs& D, int x0, int y0, int z0, int nt,
                                           bool xywall, ScalSmem<typename C::fld_t>& sm)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    const PrmR<R>& Q = prm<R>(P);
    ScalCols cols;
    scal_cols(P, x0, y0, cols);
    const int tx = threadIdx.x & (kZX - 1), ty = threadIdx.x / kZX;
    const int s1 = (tx + 1) + kZ1X * (ty + 1);
    const int x = x0 + tx, y = y0 + ty;
    const bool in = x < P.nx && y < P.ny;
    const int nxy = x + P.nx * y, sxy = P.nx * P.ny;
    const unsigned wxy = (!P.per[0] ? (x == 0 ? 1u : 0u) | (x == P.nx - 1 ? 2u : 0u) : 0u) |
                         (!P.per[1] ? (y == 0 ? 4u : 0u) | (y == P.ny - 1 ? 8u : 0u) : 0u);
    const Two<R> corr{corr_r<R>(D, 0), corr_r<R>(D, 1)};
    const R kdc = Q.C != (R)0 ? Q.kd / Q.C : (R)0;
    // Plane p in ring slot (p - z0 + 1) mod 5.  Iteration t takes in plane q =
    // z0 + t - 1 (with the column's values in q + 1), finishes plane q - 1 and
    // issues the copies of plane q + 2 into the slot of q - 3, last read in
    // iteration t - 1.  Bit k of win: plane q + 1 - k is not clear.
    unsigned win = 0;
    if (!kQuiet)
        win = ((unsigned)plane_solid(P, sm.sol, xywall, z0 - 2) << 1) |
              (unsigned)plane_solid(P, sm.sol, xywall, z0 - 1);
    scal_plane_async<F, kQuiet>(P, D, cols, z0 - 1, sm, 0);
    scal_plane_async<F, kQuiet>(P, D, cols, z0, sm, 1);
    cp_async_commit();
    ScalSums<R> prev, cur, next;
    ScalOwn<R> a, o;
    Two<R> mm;
    int r0 = 0;   // slot of plane q
#pragma unroll 1
    for (int t = 0; t <= nt + 1; ++t) {
        const int r1 = r0 + 1 == kScalRing ? 0 : r0 + 1;
        const int r2 = r1 + 1 == kScalRing ? 0 : r1 + 1;
        const int rm = r0 == 0 ? kScalRing - 1 : r0 - 1, rn = rm == 0 ? kScalRing - 1 : rm - 1;
        cp_async_wait<0>();   // this thread's copies of plane q + 1 have landed
        __syncthreads();
        if (t + 1 <= nt) scal_plane_async<F, kQuiet>(P, D, cols, z0 + t + 1, sm, r2);   // plane q + 2
        cp_async_commit();
        const int zo = z0 + t - 2;
        bool put = in && t >= 2, wall = false;
        if (!kQuiet) {
            win = (win << 1) | (unsigned)plane_solid(P, sm.sol, xywall, z0 + t);
            if (put && (win & 0xEu)) {   // planes q - 2 .. q
                put = free_node(P, D, x, y, zo);
                wall = wxy || (!P.per[2] && (zo == 0 || zo == P.nz - 1));
            }
        }
        Two<R> inc, old;   // increments of psi, phi (less the correction and the sink), old values
        R om;              // mu_phi
        if (kLB) {
            if (t >= 2) {
                const ScalPlane<R> f1 = scal_ring(sm, rm);
                inc = scal_lb<R>(Q, scal_ring(sm, rn), f1, scal_ring(sm, r0), s1, corr);
                old = f1.gp(s1);
                om = sm.mu[rm][s1][1];
            }
        } else {
            const ScalPlane<R> f = scal_ring(sm, r0);
            const Two<R> m0 = f.mp(s1);
            if (t == 0) {
                a = o = scal_own(f, s1);
                mm = m0;
                prev.ad = prev.lp = {0, 0};
                prev.dv = 0;
                cur = prev;
            }
            const ScalOwn<R> b = scal_own(scal_ring(sm, r1), s1);
            scal_plane<R>(f, s1, t >= 1 && t <= nt, a, o, b, mm, m0, prev, cur, next);
            old = a.g;
            om = mm.b;
            const Two<R> g = add2(old, corr);
            inc.a = fma_x((R)(-1.0 / 12.0), fma_x(g.a, prev.dv, prev.ad.a), mul_x((R)(1.0 / 6.0) * Q.Mpsi, prev.lp.a));
            inc.b = fma_x((R)(-1.0 / 12.0), fma_x(g.b, prev.dv, prev.ad.b), mul_x((R)(1.0 / 6.0) * Q.Mphi, prev.lp.b));
            prev = cur;
            cur = next;
            a = o;
            o = b;
            mm = m0;
        }
        if (put) {
            const int n = nxy + sxy * zo;
            if (!kQuiet && wall) {
                ZAccS<F> w;
                w.g[0] = sm.g[rn];
                w.g[1] = sm.g[rm];
                w.g[2] = sm.g[r0];
                w.mu[0] = sm.mu[rn];
                w.mu[1] = sm.mu[rm];
                w.mu[2] = sm.mu[r0];
                w.u[0] = sm.u[rn];
                w.u[1] = sm.u[rm];
                w.u[2] = sm.u[r0];
                w.s1 = s1;
                w.beyond = wxy | (!P.per[2] ? (zo == 0 ? 16u : 0u) | (zo == P.nz - 1 ? 32u : 0u) : 0u);
                scalars_compute_c<C, false>(P, D, x, y, zo, n, w, corr.a, corr.b);
            } else {
                // the stored value plus every increment of the step
                // (correction, fluxes, sink) summed first: one rounding of the
                // O(1) field
                const R sink = Q.C != (R)0 ? kdc * om
                                           : Q.kd * ((old.b + corr.b) - phi0_of(Q, old.a + corr.a));
                ((F*)D.psi_dst)[n] = (F)(old.a + (corr.a + inc.a));
                ((F*)D.phi_dst)[n] = (F)(old.b + ((corr.b + inc.b) - sink));
            }
        }
        r0 = r1;
    }
    cp_async_wait<0>();
}

// One block of kz_scalars, smem of scal_smem_bytes<C>() bytes.
template <class C>
__device__ __forceinline__ void kz_scalars_run(const DevParams& P, const DevPtrs& D, int x0, int y0, int z0, int nt,
                                               unsigned char* smem_raw)
{
    using F = typename C::fld_t;
    ScalSmem<F>& sm = *reinterpret_cast<ScalSmem<F>*>(smem_raw);
    // the positions of this step's particle update stand in the records by now,
    // and covering may be replacing the old ones: the old position lies within
    // one step's velocity of the new one
    find_solids<true>(P, D, x0, y0, 1, sm.sol, [](int, int, const DevPart&) {});
    const bool xywall = beyond_xy(P, x0, y0, 1);
    // planes any iteration looks at: z0 - 2 .. z0 + nt + 1
    bool quiet = !xywall && (P.per[2] || (z0 >= 2 && z0 + nt + 2 <= P.nz));
    for (int i = 0; i < sm.sol.n; ++i)
        quiet = quiet && !spans_meet(sm.sol.lo[i], sm.sol.len[i], z0 - 2, nt + 4, P.nz, P.per[2]);
    if (P.scheme) {
        if (quiet)
            scal_march<C, true, true>(P, D, x0, y0, z0, nt, xywall, sm);
        else
            scal_march<C, false, true>(P, D, x0, y0, z0, nt, xywall, sm);
    } else {
        if (quiet)
            scal_march<C, true, false>(P, D, x0, y0, z0, nt, xywall, sm);
        else
            scal_march<C, false, false>(P, D, x0, y0, z0, nt, xywall, sm);
    }
}

template <class C>
constexpr size_t scal_smem_bytes()
{
    return sizeof(ScalSmem<typename C::fld_t>);
}

// Resident blocks per SM of the transport: three in FP32 (80 registers), two
// in FP64.
template <class C>
constexpr int scal_blocks_per_sm()
{
    return sizeof(typename C::real) == 8 ? 2 : 3;
}

template <class C>
__global__ void __launch_bounds__(kZThreads, scal_blocks_per_sm<C>()) kz_scalars(const __grid_constant__ DevParams P,
                                                                                const __grid_constant__ DevPtrs D)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];   // scal_smem_bytes<C>()
    const int zc = zm_chunk(P.nz, gridDim.z);
    const int z0 = blockIdx.z * zc;
    const int nt = min(z0 + zc, P.nz) - z0;
    if (nt <= 0) return;   // block-uniform
    kz_scalars_run<C>(P, D, blockIdx.x * kZX, blockIdx.y * kZY, z0, nt, smem_raw);
}

}  // namespace lbdp
