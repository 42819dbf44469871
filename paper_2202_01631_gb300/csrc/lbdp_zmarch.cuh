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
//               three 34 x 10 planes of psi, phi, mu and u.
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

// shape of a one-halo plane for the paired field layout (tile_index_last)
struct ZPlane1 {
    static constexpr int slots = kZ1;
};

// Shared-memory place of field k of slot s in a plane of T::slots slots:
// fields 2j and 2j+1 interleave ([j][slot][2]), so a body that reads both
// gets them in one 64-bit load; an odd last field stands alone.
template <class T>
__host__ __device__ constexpr int tile_index(int k, int s)
{
    return (k & ~1) * T::slots + 2 * s + (k & 1);
}
template <int NF, class T>
__host__ __device__ constexpr int tile_index_last(int k, int s)
{
    return ((NF & 1) && k == NF - 1) ? (NF - 1) * T::slots + s : tile_index<T>(k, s);
}

// Nodes a thread of kz_fused works on together: the node of its column in each
// half of the block's z chunk.  Two in FP32 arithmetic (packed instructions,
// one set of column offsets, 64-bit shared loads); one in FP64, which has no
// packed form and no registers to spare.
template <class R>
__host__ __device__ constexpr int zm_halves()
{
    return sizeof(R) == 8 ? 1 : 2;
}

// Particles whose nodes may lie in the columns a block stages: the planes lo
// .. lo + len - 1 (before wrapping) hold them; slot[k] is where particle k
// stands in the list.  geo: what the wetting ghosts need of it.
struct GhostPart {
    Geo g;
    double Hk;
    float Hk_f;
};
struct SolidPlanes {
    int n;
    int lo[kMaxParticles], len[kMaxParticles];
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
    // nodes of the plane in hand that take the general body (NP slot + half),
    // and how many, for even and odd iterations
    uint16_t todo[NP * kZ1];
    int ntodo[2];
};

template <class F>
struct ScalSmem {
    F f[kScalRing][7 * kZ1];
    uint8_t mk[kScalRing][kZ1];
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
// positions the current mask was made from.
__device__ __forceinline__ void find_solids(const DevParams& P, const DevPtrs& D, int x0, int y0, int halo,
                                            SolidPlanes& sp)
{
    if (threadIdx.x == 0) sp.n = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < P.np; k += blockDim.x) {
        const DevPart& q = D.parts[k];
        // |x - X| < R lies strictly between floor(X) - ceil(R) and
        // floor(X) + ceil(R) + 1
        const int w = 2 * q.Rc + 2;
        if (spans_meet(q.g.Xi[0] - q.Rc, w, x0 - halo, kZX + 2 * halo, P.nx, P.per[0]) &&
            spans_meet(q.g.Xi[1] - q.Rc, w, y0 - halo, kZY + 2 * halo, P.ny, P.per[1])) {
            const int i = atomicAdd(&sp.n, 1);
            sp.lo[i] = q.g.Xi[2] - q.Rc;
            sp.len[i] = w;
            sp.slot[k] = (uint8_t)i;
            sp.geo[i].g = q.g;
            sp.geo[i].Hk = q.Hk;
            sp.geo[i].Hk_f = q.Hk_f;
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
    const SolidPlanes* sol;
    __device__ __forceinline__ const GhostPart& part(const DevPtrs&, int k) const { return sol->geo[sol->slot[k]]; }
    __device__ __forceinline__ uint8_t mask(int i) const { return nb[i] >= 0 ? mk[nb[i]] : kWallSlot; }
    template <int K>
    __device__ __forceinline__ F get(int i) const
    {
        if (K == 0) return ps[1 + cz(i)][o2 + NP * poff<kZ2X>(i)];
        return phi_own;   // field 1 is read at the node itself only
    }
};

// force body of a node next to a wall, in one half of the planes of kz_fused:
// the stress (p_iso, grad psi) of the one-halo planes.  Bit 2 a + s of beyond:
// the neighbours on side s (0 below, 1 above) of axis a lie beyond a wall.
template <class F, int NP>
struct ZAccP {
    const F* pa[3];
    const F* pb[3];
    int o1;   // 2 * NP * slot + half
    unsigned beyond;
    __device__ __forceinline__ uint8_t mask(int i) const
    {
        const unsigned c = (cx(i) < 0 ? 1u : cx(i) > 0 ? 2u : 0u) | (cy(i) < 0 ? 4u : cy(i) > 0 ? 8u : 0u) |
                           (cz(i) < 0 ? 16u : cz(i) > 0 ? 32u : 0u);
        return (beyond & c) ? kWallSlot : (uint8_t)0;
    }
    template <int K>
    __device__ __forceinline__ F get(int i) const
    {
        const F* p = K < 2 ? pa[1 + cz(i)] : pb[1 + cz(i)];
        return p[o1 + 2 * NP * poff<kZ1X>(i) + (K & 1) * NP];
    }
};

// transport body: psi, phi, mu_psi, mu_phi, u (one-halo planes, paired)
template <class F, bool kClear>
struct ZAccS {
    const F* f[3];
    const uint8_t* mk[3];
    int s1;
    __device__ __forceinline__ uint8_t mask(int i) const
    {
        return kClear ? (uint8_t)0 : mk[1 + cz(i)][s1 + poff<kZ1X>(i)];
    }
    template <int K>
    __device__ __forceinline__ F get(int i) const
    {
        return f[1 + cz(i)][tile_index_last<7, ZPlane1>(K, s1 + poff<kZ1X>(i))];
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
    static_assert(B == 4 || B == 8, "4- or 8-byte copies");
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

// Issue the copies of the seven transport fields of plane p into ring slot r.
template <class F>
__device__ __forceinline__ void scal_plane_async(const DevParams& P, const DevPtrs& D, const ScalCols& c, int p,
                                                 ScalSmem<F>& sm, int r)
{
    const size_t N = (size_t)P.N;
    const F* u = (const F*)D.u;
    const F* const src[7] = {(const F*)D.psi_src, (const F*)D.phi_src, (const F*)D.mupsi, (const F*)D.muphi,
                             u, u + N, u + 2 * N};
    const int gz = wrap_coord(p, P.nz, P.per[2]);
    const int base = gz * P.nx * P.ny;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int s = threadIdx.x + h * kZThreads;
        if (s < kZ1) {
            const bool ok = c.c[h] >= 0 && gz >= 0;
            const int g = ok ? base + c.c[h] : 0;
#pragma unroll
            for (int k = 0; k < 7; ++k)
                cp_async<(int)sizeof(F)>(&sm.f[r][tile_index_last<7, ZPlane1>(k, s)], src[k] + g, ok);
        }
    }
}

// The masks of a plane go through registers (their OR decides the mask-free
// body): m[h] for this thread's slots, kWallSlot beyond a wall.
struct ScalMask {
    uint8_t m[2];
};

__device__ __forceinline__ void scal_mask_fetch(const DevParams& P, const DevPtrs& D, const ScalCols& c, int p,
                                                ScalMask& M)
{
    const int gz = wrap_coord(p, P.nz, P.per[2]);
    const int base = gz * P.nx * P.ny;
#pragma unroll
    for (int h = 0; h < 2; ++h) M.m[h] = (c.c[h] >= 0 && gz >= 0) ? D.mask[base + c.c[h]] : kWallSlot;
}

// Store the masks into ring slot r; returns whether any is not fluid.
template <class F>
__device__ __forceinline__ bool scal_mask_store(ScalSmem<F>& sm, int r, const ScalMask& M)
{
    bool any = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int s = threadIdx.x + h * kZThreads;
        if (s < kZ1) {
            sm.mk[r][s] = M.m[h];
            any = any || M.m[h] != 0;
        }
    }
    return any;
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
    if (n >= 0) {
        ((F*)D.mupsi)[n] = (F)mps;
        ((F*)D.muphi)[n] = (F)mph;
    }
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
                    ((F*)D.mupsi)[n] = (F)mps.lane(h);
                    ((F*)D.muphi)[n] = (F)mph.lane(h);
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
        a.sol = &sm.sol;
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

// BGK collision with Guo forcing of NP nodes, as collide_store, with the
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
    find_solids(P, D, x0, y0, 2, sm.sol);
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
template <class C, bool kClear>
__device__ __forceinline__ void scal_stage(const DevParams& P, const DevPtrs& D,
                                           const ScalSmem<typename C::fld_t>& sm, int x0, int y0, int zs,
                                           const int (&r)[3], typename C::real dps, typename C::real dph)
{
    using F = typename C::fld_t;
    const int tx = threadIdx.x & (kZX - 1), ty = threadIdx.x / kZX;
    const int x = x0 + tx, y = y0 + ty;
    if (x >= P.nx || y >= P.ny) return;
    const int s1 = (tx + 1) + kZ1X * (ty + 1);
    if (sm.mk[r[1]][s1] != 0) return;   // inside a particle
    ZAccS<F, kClear> a;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a.f[k] = sm.f[r[k]];
        a.mk[k] = sm.mk[r[k]];
    }
    a.s1 = s1;
    scalars_compute_c<C, false>(P, D, x, y, zs, x + P.nx * (y + P.ny * zs), a, dps, dph);
}

// The march of one block, as kz_fused_run (smem of sizeof(ScalSmem<F>) bytes).
template <class C>
__device__ __forceinline__ void kz_scalars_run(const DevParams& P, const DevPtrs& D, int x0, int y0, int z0, int nt,
                                               unsigned char* smem_raw)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    ScalSmem<F>& sm = *reinterpret_cast<ScalSmem<F>*>(smem_raw);
    ScalCols cols;
    scal_cols(P, x0, y0, cols);
    const R dps = corr_r<R>(D, 0), dph = corr_r<R>(D, 1);
    // Plane p in ring slot (p - z0 + 1) mod 5.  Iteration t computes plane
    // z0 + t from planes z0 + t - 1 .. z0 + t + 1 and issues the copies of
    // plane z0 + t + 2 (into the slot of z0 + t - 3, last read at t - 2); the
    // masks of a plane are loaded one iteration before they are stored.
    unsigned hist = 0;
    ScalMask M;
    for (int k = 0; k < 2; ++k) {   // planes z0 - 1, z0
        scal_plane_async<F>(P, D, cols, z0 - 1 + k, sm, k);
        scal_mask_fetch(P, D, cols, z0 - 1 + k, M);
        hist = (hist << 1) | (unsigned)__syncthreads_or(scal_mask_store<F>(sm, k, M));
    }
    cp_async_commit();
    scal_plane_async<F>(P, D, cols, z0 + 1, sm, 2);
    cp_async_commit();
    scal_mask_fetch(P, D, cols, z0 + 1, M);
    int r0 = 0;   // slot of plane z0 + t - 1
    for (int t = 0; t < nt; ++t) {
        const int r1 = r0 + 1 == kScalRing ? 0 : r0 + 1;
        const int r2 = r1 + 1 == kScalRing ? 0 : r1 + 1;
        const int r3 = r2 + 1 == kScalRing ? 0 : r2 + 1;
        const bool any = scal_mask_store<F>(sm, r2, M);   // plane z0 + t + 1
        if (t + 2 <= nt) {
            scal_mask_fetch(P, D, cols, z0 + t + 2, M);
            scal_plane_async<F>(P, D, cols, z0 + t + 2, sm, r3);
        }
        cp_async_commit();
        cp_async_wait<1>();   // this thread's copies of plane z0 + t + 1 have landed
        hist = (hist << 1) | (unsigned)__syncthreads_or(any);
        const int r[3] = {r0, r1, r2};
        if ((hist & 7u) == 0u)
            scal_stage<C, true>(P, D, sm, x0, y0, z0 + t, r, dps, dph);
        else
            scal_stage<C, false>(P, D, sm, x0, y0, z0 + t, r, dps, dph);
        r0 = r1;
    }
    cp_async_wait<0>();
}

// Resident blocks per SM of the transport: three (80 registers) measured
// faster than four (64) on the 256^3 workload.
constexpr int kScalBlocksPerSM = 3;

template <class C>
__global__ void __launch_bounds__(kZThreads, kScalBlocksPerSM) kz_scalars(const __grid_constant__ DevParams P,
                                                                          const __grid_constant__ DevPtrs D)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];   // sizeof(ScalSmem<F>)
    const int zc = zm_chunk(P.nz, gridDim.z);
    const int z0 = blockIdx.z * zc;
    const int nt = min(z0 + zc, P.nz) - z0;
    if (nt <= 0) return;   // block-uniform
    kz_scalars_run<C>(P, D, blockIdx.x * kZX, blockIdx.y * kZY, z0, nt, smem_raw);
}

}  // namespace lbdp
