// lbdp_particles.cuh -- the kernels of the nodes next to particles, which run
// beside the bulk kernels on the side streams: stress and force there
// (k_pt_part, k_f_part), the link sums and the implicit particle update
// (k_links), the collide-stream (k_collide_particles) and the transport
// (k_scalars_particles).
//
// They are bound by latency -- a few hundred to a few thousand nodes, each a
// chain of dependent loads -- and on small boxes they are the step.  So a block
// first lists the nodes of its share of the particle's box that have work, in
// box order, and then gives one node to a thread: the warps that go through
// the long bodies are full instead of a tenth full, and the rest stop.  The
// bodies issue the loads of a node together and loop over the links a node
// has (a bit mask) with the particle's record in registers, instead of 18
// unrolled bodies each with its own loads.  The list is in box order and the
// split of the box over blocks is fixed, so every sum has one order.
#pragma once

#include "lbdp_kernels.cuh"
#include "lbdp_vec.cuh"
#include "lbdp_zmarch.cuh"

namespace lbdp {

// Blocks per SM the long bodies are compiled for: four in FP32 arithmetic (128
// registers), two in FP64, so that two or one fit in the place of a block of
// kz_fused and need not wait for an SM of their own.
template <class C>
constexpr int part_blocks_per_sm()
{
    return sizeof(typename C::real) == 8 ? 2 : 4;
}

// ---------------------------------------------------------------------------
// lists of nodes
// ---------------------------------------------------------------------------
constexpr int kScanWarps = kPartThreads / 32;
template <class C>
struct NodeList {
    static constexpr int kScanSlots = part_slots(sizeof(typename C::real) == 8);
    int n[kScanSlots * kPartThreads];   // node indices, in the order of the scan
    int wcount[kScanSlots][kScanWarps];
};

// List the nodes among the kScanSlots * blockDim.x box slots of block bi of
// nbi, round r (edges s, origin o), that pred(n, x, y, z) takes; returns their
// number.  Block-wide.  A block takes every nbi-th slot: consecutive ones would
// give the blocks that hold a polar cap of the sphere many times the nodes of
// the others.
template <class C, class Pred>
__device__ __forceinline__ int list_nodes(const DevParams& P, const int o[3], const int s[3], int r, int bi, int nbi,
                                          int tot, NodeList<C>& L, Pred pred)
{
    constexpr int kScanSlots = NodeList<C>::kScanSlots;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int n[kScanSlots];
    bool ok[kScanSlots];
#pragma unroll
    for (int j = 0; j < kScanSlots; ++j) {
        const int t = ((r * kScanSlots + j) * kPartThreads + (int)threadIdx.x) * nbi + bi;
        int x, y, z;
        n[j] = 0;
        ok[j] = t < tot && box_node(P, o, s, t, x, y, z);
        if (ok[j]) {
            n[j] = x + P.nx * (y + P.ny * z);
            ok[j] = pred(n[j], x, y, z);
        }
    }
    unsigned bal[kScanSlots];
#pragma unroll
    for (int j = 0; j < kScanSlots; ++j) bal[j] = __ballot_sync(0xffffffffu, ok[j]);
    __syncthreads();   // the list of the round before has been read
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < kScanSlots; ++j) L.wcount[j][warp] = __popc(bal[j]);
    __syncthreads();
    int total = 0;
#pragma unroll
    for (int j = 0; j < kScanSlots; ++j) {
        int base = total;
#pragma unroll
        for (int w = 0; w < kScanWarps; ++w) {
            const int c = L.wcount[j][w];
            base += w < warp ? c : 0;
            total += c;
        }
        if (ok[j]) L.n[base + __popc(bal[j] & ((1u << lane) - 1u))] = n[j];
    }
    __syncthreads();
    return total;
}

__device__ __forceinline__ void node_coords(const DevParams& P, int n, int& x, int& y, int& z)
{
    const int r = n / P.nx;
    x = n - r * P.nx;
    z = r / P.ny;
    y = r - z * P.ny;
}

// Masks around a node: mk[i] (kWallSlot beyond a wall); solid: directions into
// a particle; stop: directions into a particle or a wall; lo, hi: lowest and
// highest particle number + 1 (lo = 255 without one).
struct Around {
    int nb[19];
    uint8_t mk[19];
    unsigned solid, stop;
    int lo, hi;
};

__device__ __forceinline__ void look_around(const DevParams& P, const DevPtrs& D, int x, int y, int z, Around& a)
{
    neighbours(P, x, y, z, a.nb);
    a.mk[0] = 0;
#pragma unroll
    for (int i = 1; i < 19; ++i) a.mk[i] = a.nb[i] >= 0 ? D.mask[a.nb[i]] : kWallSlot;
    a.solid = a.stop = 0;
    a.lo = 255;
    a.hi = 0;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        if (a.mk[i]) a.stop |= 1u << i;
        if (a.mk[i] && a.mk[i] != kWallSlot) {
            a.solid |= 1u << i;
            a.lo = min(a.lo, (int)a.mk[i]);
            a.hi = max(a.hi, (int)a.mk[i]);
        }
    }
}

// The directions of a that lead into particle k (number + 1).
__device__ __forceinline__ unsigned links_into(const Around& a, int k)
{
    if (a.lo == a.hi) return k == a.lo ? a.solid : 0u;
    unsigned b = 0;
#pragma unroll
    for (int i = 1; i < 19; ++i) b |= a.mk[i] == k ? 1u << i : 0u;
    return b;
}

// grad phi of the node, 3 sum_i w_i c_i phi(x + c_i), from differences to its own value;
// stopped directions carry the node's own value.
template <class R, class F>
__device__ __forceinline__ void grad_phi_around(const Around& a, const F* phi, int n, R own, R dphi, R g[3])
{
    R pv[19];
#pragma unroll
    for (int i = 1; i < 19; ++i) pv[i] = (R)phi[a.nb[i] >= 0 ? a.nb[i] : n];
    g[0] = g[1] = g[2] = (R)0;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        const R v = (a.stop >> i & 1u) ? (R)0 : add_x(pv[i] + dphi, -own);
        const R w = wgt_r<R>(i);
        if (cx(i) != 0) g[0] = fma_x(cx(i) > 0 ? w : -w, v, g[0]);
        if (cy(i) != 0) g[1] = fma_x(cy(i) > 0 ? w : -w, v, g[1]);
        if (cz(i) != 0) g[2] = fma_x(cz(i) > 0 ? w : -w, v, g[2]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) g[k] = mul_x(g[k], (R)3);
}

// ---------------------------------------------------------------------------
// links of one node into one particle
// ---------------------------------------------------------------------------
template <class R>
struct NodeLinks {
    LinkPart q;
    int D[3];
    R r0[3];   // x - X
};

template <class R>
__device__ __forceinline__ void node_links(const DevParams& P, const DevPart& part, int x, int y, int z,
                                           NodeLinks<R>& l)
{
    l.q = link_part(part);
    int_offset(P, l.q.g, x, y, z, l.D);
    link_offset_r<R>(l.q.g, l.D, 0, l.r0);
}

// m . r <= 0 at the midpoint of link (c0, c1, c2), the oracle's decision.
template <class Q>
__device__ __forceinline__ bool cap_minus_at(const Q& q, const int D[3], int c0, int c1, int c2)
{
    const float r0 = ((float)D[0] + 0.5f * (float)c0) - q.g.fr[0];
    const float r1 = ((float)D[1] + 0.5f * (float)c1) - q.g.fr[1];
    const float r2 = ((float)D[2] + 0.5f * (float)c2) - q.g.fr[2];
    const float sd = dot_x(q.mf[0], q.mf[1], q.mf[2], r0, r1, r2);
    if (sd < -q.smarg) return true;
    if (sd > q.smarg) return false;
    const double e[3] = {__dsub_rn(__dadd_rn((double)D[0], 0.5 * c0), q.g.frd[0]),
                         __dsub_rn(__dadd_rn((double)D[1], 0.5 * c1), q.g.frd[1]),
                         __dsub_rn(__dadd_rn((double)D[2], 0.5 * c2), q.g.frd[2])};
    return dot3_rn(q.m, e) <= 0.0;
}

// c . v_s at the midpoint of link i, v_s = mu (1 - n n) . grad phi with mu =
// mu_- where m . r <= 0 else mu_+ (Eq. MuJ); r: the midpoint offset.
template <class R>
__device__ __forceinline__ R link_slip(const NodeLinks<R>& l, int i, const R gphi[3], R r[3])
{
    const int k0 = dir_comp<0>(i), k1 = dir_comp<1>(i), k2 = dir_comp<2>(i);
    const R c0 = (R)k0, c1 = (R)k1, c2 = (R)k2;
    r[0] = fma_x((R)0.5, c0, l.r0[0]);
    r[1] = fma_x((R)0.5, c1, l.r0[1]);
    r[2] = fma_x((R)0.5, c2, l.r0[2]);
    const R mp = PartR<R>::mu_p(l.q), mm = PartR<R>::mu_m(l.q);
    if (mp == (R)0 && mm == (R)0) return (R)0;
    const R mu = mp == mm ? mp : (cap_minus_at(l.q, l.D, k0, k1, k2) ? mm : mp);
    const InvNorm<R> in = inv_norm(dot_x(r[0], r[1], r[2], r[0], r[1], r[2]));
    const R n0 = in.times(r[0]), n1 = in.times(r[1]), n2 = in.times(r[2]);
    const R ng = dot_x(n0, n1, n2, gphi[0], gphi[1], gphi[2]);
    return dot_x(c0, c1, c2, mul_x(mu, fma_x(-n0, ng, gphi[0])), mul_x(mu, fma_x(-n1, ng, gphi[1])),
                 mul_x(mu, fma_x(-n2, ng, gphi[2])));
}

// c . u_b of link i, u_b = U + Omega x r + v_s.
template <class R>
__device__ __forceinline__ R link_cub(const NodeLinks<R>& l, int i, const R gphi[3])
{
    R r[3];
    const R s = link_slip<R>(l, i, gphi, r);
    const R c0 = (R)dir_comp<0>(i), c1 = (R)dir_comp<1>(i), c2 = (R)dir_comp<2>(i);
    const R U0 = PartR<R>::U(l.q, 0), U1 = PartR<R>::U(l.q, 1), U2 = PartR<R>::U(l.q, 2);
    const R W0 = PartR<R>::W(l.q, 0), W1 = PartR<R>::W(l.q, 1), W2 = PartR<R>::W(l.q, 2);
    const R v0 = add_x(U0, cross_x(W1, r[2], W2, r[1]));
    const R v1 = add_x(U1, cross_x(W2, r[0], W0, r[2]));
    const R v2 = add_x(U2, cross_x(W0, r[1], W1, r[0]));
    return add_x(dot_x(c0, c1, c2, v0, v1, v2), s);
}

// ---------------------------------------------------------------------------
// the pressure tensor and force next to particles
// ---------------------------------------------------------------------------
// The link box of particle p grown by one node.
__device__ __forceinline__ void pt_box(const DevParams& P, const DevPart& q, int o[3], int s[3])
{
    const int L[3] = {P.nx, P.ny, P.nz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        o[a] = q.g.Xi[a] - q.Rc - 3;
        s[a] = P.side1[a] + 2;
        if (P.per[a] && s[a] > L[a]) s[a] = L[a];
    }
}

// Blocks per particle of k_pt_part.
__host__ __device__ inline int pt_part_blocks(const DevParams& P, bool fp64)
{
    long long t = 1;
    const int L[3] = {P.nx, P.ny, P.nz};
    for (int a = 0; a < 3; ++a) {
        int s = P.side1[a] + 2;
        if (P.per[a] && s > L[a]) s = L[a];
        t *= s;
    }
    const int per = part_slots(fp64) * kPartThreads;
    const long long b = (t + per - 1) / per;
    return (int)(b < 1 ? 1 : (b > kMaxPartBlocks ? kMaxPartBlocks : b));
}

// Block bi of the nbi blocks of particle p: P at the fluid nodes next to the
// particle and their neighbours -- those within R + 2 sqrt 2 of its centre --
// into the pressure-tensor array.  Nodes near two particles are written twice
// with the same values.
template <class C>
__device__ __forceinline__ void pt_part_block(const DevParams& P, const DevPtrs& D, int p, int bi, int nbi,
                                              NodeList<C>& list)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    if (!P.thermo) return;
    const DevPart& q = D.parts[p];
    const Geo g = q.g;
    const float reach = (float)q.R + 2.84f;
    int o[3], sd[3];
    pt_box(P, q, o, sd);
    const int tot = sd[0] * sd[1] * sd[2];
    const size_t N = (size_t)P.N;
    for (int r = 0; (long long)r * NodeList<C>::kScanSlots * kPartThreads * nbi < tot; ++r) {
        const int cnt = list_nodes(P, o, sd, r, bi, nbi, tot, list, [&](int n, int x, int y, int z) {
            int Dn[3];
            int_offset(P, g, x, y, z, Dn);
            const float d0 = (float)Dn[0] - g.fr[0], d1 = (float)Dn[1] - g.fr[1], d2 = (float)Dn[2] - g.fr[2];
            return dot_x(d0, d1, d2, d0, d1, d2) < reach * reach && D.mask[n] == 0;
        });
        for (int e = threadIdx.x; e < cnt; e += kPartThreads) {
            const int n = list.n[e];
            int x, y, z;
            node_coords(P, n, x, y, z);
            GAcc<F, 2> a;
            neighbours(P, x, y, z, a.nb);
            a.n = n;
            a.mk = D.mask;
            a.f[0] = (const F*)D.psi_src;
            a.f[1] = (const F*)D.phi_src;
            R mps, mph, pt[kPtFields];
            mup_values<C>(P, D, x, y, z, a, corr_r<R>(D, 0), corr_r<R>(D, 1), mps, mph, pt);
            F* ptg = (F*)D.pt;
#pragma unroll
            for (int k = 0; k < kPtFields; ++k) ptg[k * N + n] = (F)pt[k];
        }
    }
}

template <class C>
__global__ void __launch_bounds__(kPartThreads) k_pt_part(const __grid_constant__ DevParams P,
                                                           const __grid_constant__ DevPtrs D)
{
    __shared__ NodeList<C> list;
    pt_part_block<C>(P, D, blockIdx.y, blockIdx.x, gridDim.x, list);
}

// The link box of particle p: it holds every fluid node within R + 2 of the
// centre (floor(X) - ceil(R) <= floor(X - R)).
__device__ __forceinline__ void link_box(const DevPart& q, int o[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) o[a] = q.g.Xi[a] - q.Rc - 2;
}

// F at the fluid nodes of particle p's link box that lie next to a particle, into
// the force array.
template <class C>
__device__ __forceinline__ void f_part_block(const DevParams& P, const DevPtrs& D, int p, int bi, int nbi,
                                             NodeList<C>& list)
{
    using F = typename C::fld_t;
    int o[3];
    link_box(D.parts[p], o);
    const int tot = P.side1[0] * P.side1[1] * P.side1[2];
    for (int r = 0; (long long)r * NodeList<C>::kScanSlots * kPartThreads * nbi < tot; ++r) {
        const int cnt = list_nodes(P, o, P.side1, r, bi, nbi, tot, list,
                                   [&](int n, int, int, int) { return D.mask[n] == 0 && D.bflag[n] != 0; });
        for (int e = threadIdx.x; e < cnt; e += kPartThreads) {
            const int n = list.n[e];
            int x, y, z;
            node_coords(P, n, x, y, z);
            // a node in the boxes of several particles: each of their blocks
            // writes the same force
            const size_t N = (size_t)P.N;
            const F* pt = (const F*)D.pt;
            GAcc<F, kPtFields> a;
            neighbours(P, x, y, z, a.nb);
            a.n = n;
            a.mk = D.mask;
#pragma unroll
            for (int k = 0; k < kPtFields; ++k) a.f[k] = pt + k * N;
            fdiv_compute<C>(P, D, n, a);
        }
    }
}

template <class C>
__global__ void __launch_bounds__(kPartThreads) k_f_part(const __grid_constant__ DevParams P,
                                                          const __grid_constant__ DevPtrs D)
{
    __shared__ NodeList<C> list;
    f_part_block<C>(P, D, blockIdx.y, blockIdx.x, gridDim.x, list);
}

// ---------------------------------------------------------------------------
// S5 + S6a: link sums and the implicit velocity update.  Grid (nb1, np): the
// blocks of a particle split its link box; the last block of the particle (a
// ticket counter) sums the partials in block order and solves
//   (Mdiag + zeta) V(t+1) = Mdiag V(t) + [F0; T0]
// (symmetric positive definite), then stores the new velocity and the
// position/orientation after the step.
//
// With a = 36 w_i (2 on axis links, 1 on diagonal ones), c = c_i, r = x - X and
// D = r + fr the node's integer offset from floor(X), the sums over a node's
// links into the particle are
//   A = sum a c c^T, B = sum a c          -- integers, from the link bits;
//   zeta: s sum a g g^T with g = (c, r_b x c) = (c, D x c - fr x c), s = rho0/6:
//     the integer sums A, sum a c (D x c)^T and sum a (D x c)(D x c)^T over all
//     nodes are exact, and the fraction fr enters once, in FP64;
//   F0: sum c (2 g_i - 6 w rho0 c.v_s) + (p B + kappa grad psi (grad psi . B))/6,
//   T0: r x (the node's F0) + kappa/12 (A grad psi) x grad psi -- the c/2 of a
//     link point is parallel to c, and the rest of c/2 x P.c is this;
//   the constant parts of both (2 w rho0 c of the bounced populations, 6 w
//     (A/4) c of the bulk pressure the stored stress leaves out) from the
//     integer sums of B and D x B;
//   the scalar flux into the surface, linear in V(t+1): psi, phi times
//     sum 6 w (c, r x c) = (B, r x B)/6 and sum 6 w c.v_s (finite differences),
//     or the same with weight 1 on the six D3Q7 links (lattice Boltzmann).
// So a link costs its slip velocity and nothing else.  Each node's values are
// one row of 26 numbers of the arithmetic precision and 27 integers; a thread
// per column and quarter of the rows adds them in FP64 and int64.  Two threads
// of different warps share a node, one for its stress and the force of it
// (columns 20 to 25), one for the rest: a block has fewer nodes than threads,
// and what bounds it is the length of one thread's work.
// Measured on GB300: FP32, one sphere R = 8, 56 us with 41 FP64 sums over the
// links (250 registers, 84 KB of shared memory), 33 with the rows; the rows'
// part of the block 16.5 thousand cycles with a thread per node, 10.0 with two
// (24^3; FP64 32^3 100 and 70), the kernels before the bulk 54.3 -> 48.6 us at
// 24^3, 160 -> 144 in FP64 at 32^3 (with the shared particle update).
// ---------------------------------------------------------------------------
constexpr int kRowP = 20, kRowF = kRowP + 6, kRowI = 27, kRow = kRowF + kRowI, kRowGroups = 4;
constexpr int kRowNodes = kPartThreads / 2;   // nodes of a round: two threads each
static_assert(kRowGroups * kRowF <= kPartThreads && kRowGroups * kRowI <= kPartThreads,
              "a thread per column and group of rows");

template <class C>
struct LinkSmem {
    using R = typename C::real;
    NodeList<C> list;
    DevPart part;
    R rf[kRowNodes][kRowF + 1];
    int ri[kRowNodes][kRowI];
    double col[kRowGroups][kRow];
    double red[kPartThreads];
    double tot[64];        // link totals
    bool last;
};

// Integer sums of the links in bits: A = sum a c c^T (xx yy zz xy xz yz), B =
// sum a c.
__device__ __forceinline__ void link_ints(unsigned bits, int (&A)[6], int (&B)[3])
{
#pragma unroll
    for (int k = 0; k < 6; ++k) A[k] = 0;
    B[0] = B[1] = B[2] = 0;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        const int k = (int)(bits >> i & 1u) * (i < 7 ? 2 : 1);
        A[0] += k * cx(i) * cx(i);
        A[1] += k * cy(i) * cy(i);
        A[2] += k * cz(i) * cz(i);
        A[3] += k * cx(i) * cy(i);
        A[4] += k * cx(i) * cz(i);
        A[5] += k * cy(i) * cz(i);
        B[0] += k * cx(i);
        B[1] += k * cy(i);
        B[2] += k * cz(i);
    }
}

// Node n of the link box of particle q (in shared memory): the force of its
// stress (the one the fluid's force uses this step, k_pt_part) on the links and
// its torque, columns kRowP to kRowP + 5 of the row.
template <class C>
__device__ __forceinline__ void link_stress(const DevParams& P, const DevPtrs& D, const DevPart& q, int p, int n,
                                            typename C::real (&rf)[kRowF + 1])
{
    using R = typename C::real;
    using F = typename C::fld_t;
    const PrmR<R>& Q = prm<R>(P);
    if (!P.thermo) {
#pragma unroll
        for (int k = 0; k < 6; ++k) rf[kRowP + k] = 0;
        return;
    }
    int x, y, z;
    node_coords(P, n, x, y, z);
    Around a;
    look_around(P, D, x, y, z, a);
    GAcc<F, 2> ga;
#pragma unroll
    for (int i = 0; i < 19; ++i) ga.nb[i] = a.nb[i];
    ga.n = n;
    ga.mk = D.mask;
    ga.f[0] = (const F*)D.psi_src;
    ga.f[1] = (const F*)D.phi_src;
    R m1, m2, pt[kPtFields];
    mup_values<C>(P, D, x, y, z, ga, corr_r<R>(D, 0), corr_r<R>(D, 1), m1, m2, pt);
#pragma unroll
    for (int k = 0; k < kPtFields; ++k) pt[k] = (R)(F)pt[k];
    int A[6], B[3];
    link_ints(links_into(a, p + 1), A, B);
    const R Bf[3] = {(R)B[0], (R)B[1], (R)B[2]};
    const R gB = mul_x(Q.kappa, dot_x(pt[1], pt[2], pt[3], Bf[0], Bf[1], Bf[2]));
    R m[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) m[k] = mul_x((R)(1.0 / 6.0), fma_x(gB, pt[1 + k], mul_x(pt[0], Bf[k])));
    NodeLinks<R> l;
    node_links<R>(P, q, x, y, z, l);
    const R Af[6] = {(R)A[0], (R)A[1], (R)A[2], (R)A[3], (R)A[4], (R)A[5]};
    const R Ag[3] = {dot_x(Af[0], Af[3], Af[4], pt[1], pt[2], pt[3]), dot_x(Af[3], Af[1], Af[5], pt[1], pt[2], pt[3]),
                     dot_x(Af[4], Af[5], Af[2], pt[1], pt[2], pt[3])};
    const R k = mul_x(Q.kappa, (R)(1.0 / 12.0));
    rf[kRowP] = m[0];
    rf[kRowP + 1] = m[1];
    rf[kRowP + 2] = m[2];
    rf[kRowP + 3] = fma_x(k, cross_x(Ag[1], pt[3], Ag[2], pt[2]), cross_x(l.r0[1], m[2], l.r0[2], m[1]));
    rf[kRowP + 4] = fma_x(k, cross_x(Ag[2], pt[1], Ag[0], pt[3]), cross_x(l.r0[2], m[0], l.r0[0], m[2]));
    rf[kRowP + 5] = fma_x(k, cross_x(Ag[0], pt[2], Ag[1], pt[1]), cross_x(l.r0[0], m[1], l.r0[1], m[0]));
}

// Node n of the link box of particle q (in shared memory): the rest of its row.
template <class C>
__device__ __forceinline__ void link_row(const DevParams& P, const DevPtrs& D, const DevPart& q, int p, int n,
                                         typename C::real (&rf)[kRowF + 1], int (&ri)[kRowI])
{
    using R = typename C::real;
    using F = typename C::fld_t;
    using S = typename C::pop_t;
    const PrmR<R>& Q = prm<R>(P);
    const int NN = (int)P.N;
    const S* fs = (const S*)D.f_src;
    const F* phi = (const F*)D.phi_src;
    const R dps = corr_r<R>(D, 0), dph = corr_r<R>(D, 1);
    int x, y, z;
    node_coords(P, n, x, y, z);
    Around a;
    look_around(P, D, x, y, z, a);
    const unsigned bits = links_into(a, p + 1);
    // populations as deviations g_i = f_i - w_i rho0: their constant part is
    // added exactly, so the link terms carry small numbers
    R fv[19];
#pragma unroll
    for (int i = 1; i < 19; ++i) fv[i] = (R)PopStore<S>::load_dev(fs, i * NN + n, i, Q.rho0);
    const R ps = (R)((const F*)D.psi_src)[n] + dps, ph = (R)phi[n] + dph;
    R gphi[3];
    grad_phi_around<R, F>(a, phi, n, ph, dph, gphi);
    // bounced populations, 2 sum c g_i
    R m[3] = {0, 0, 0};
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        const R f = (bits >> i & 1u) ? fv[i] : (R)0;
        if (cx(i) != 0) m[0] = cx(i) > 0 ? add_x(m[0], f) : add_x(m[0], -f);
        if (cy(i) != 0) m[1] = cy(i) > 0 ? add_x(m[1], f) : add_x(m[1], -f);
        if (cz(i) != 0) m[2] = cz(i) > 0 ? add_x(m[2], f) : add_x(m[2], -f);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) m[k] = add_x(m[k], m[k]);
    // slip: sum 6 w rho0 c (c . v_s) and the flux weight's sum of c . v_s
    NodeLinks<R> l;
    node_links<R>(P, q, x, y, z, l);
    R slip = 0;
    if (PartR<R>::mu_p(l.q) != (R)0 || PartR<R>::mu_m(l.q) != (R)0) {
        for (unsigned b = bits; b; b &= b - 1) {
            const int i = __ffs((int)b) - 1;
            R r[3];
            const R cvs = link_slip<R>(l, i, gphi, r);
            const R w6 = i < 7 ? (R)(1.0 / 3.0) : (R)(1.0 / 6.0);
            const R k = mul_x(mul_x(w6, Q.rho0), cvs);
            m[0] = fma_x((R)-dir_comp<0>(i), k, m[0]);
            m[1] = fma_x((R)-dir_comp<1>(i), k, m[1]);
            m[2] = fma_x((R)-dir_comp<2>(i), k, m[2]);
            slip = fma_x(P.scheme ? (i < 7 ? (R)1 : (R)0) : w6, cvs, slip);
        }
    }
    int A[6], B[3], B7[3] = {0, 0, 0};
    link_ints(bits, A, B);
#pragma unroll
    for (int i = 1; i < 7; ++i) {
        const int one = (int)(bits >> i & 1u);
        B7[0] += one * cx(i);
        B7[1] += one * cy(i);
        B7[2] += one * cz(i);
    }
    const R Bf[3] = {(R)B[0], (R)B[1], (R)B[2]};
    const R T[3] = {cross_x(l.r0[1], m[2], l.r0[2], m[1]), cross_x(l.r0[2], m[0], l.r0[0], m[2]),
                    cross_x(l.r0[0], m[1], l.r0[1], m[0])};
    R G[7];
    {
        const R w = P.scheme ? (R)1 : (R)(1.0 / 6.0);
        const R b0 = mul_x(w, P.scheme ? (R)B7[0] : Bf[0]), b1 = mul_x(w, P.scheme ? (R)B7[1] : Bf[1]),
                b2 = mul_x(w, P.scheme ? (R)B7[2] : Bf[2]);
        G[0] = b0;
        G[1] = b1;
        G[2] = b2;
        G[3] = cross_x(l.r0[1], b2, l.r0[2], b1);
        G[4] = cross_x(l.r0[2], b0, l.r0[0], b2);
        G[5] = cross_x(l.r0[0], b1, l.r0[1], b0);
        G[6] = slip;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        rf[k] = m[k];
        rf[3 + k] = T[k];
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        rf[6 + k] = mul_x(ps, G[k]);
        rf[13 + k] = mul_x(ph, G[k]);
    }
    // L = sum a c (D x c)^T, Qm = sum a (D x c)(D x c)^T
    const int d0 = l.D[0], d1 = l.D[1], d2 = l.D[2];
    const int Am[3][3] = {{A[0], A[3], A[4]}, {A[3], A[1], A[5]}, {A[4], A[5], A[2]}};
    int Lm[3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        Lm[i][0] = d1 * Am[i][2] - d2 * Am[i][1];
        Lm[i][1] = d2 * Am[i][0] - d0 * Am[i][2];
        Lm[i][2] = d0 * Am[i][1] - d1 * Am[i][0];
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) ri[k] = A[k];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) ri[6 + 3 * i + j] = Lm[i][j];
    // Qm_ab = (D x .)_a of the rows of L
    ri[15] = d1 * Lm[2][0] - d2 * Lm[1][0];
    ri[16] = d2 * Lm[0][1] - d0 * Lm[2][1];
    ri[17] = d0 * Lm[1][2] - d1 * Lm[0][2];
    ri[18] = d1 * Lm[2][1] - d2 * Lm[1][1];
    ri[19] = d1 * Lm[2][2] - d2 * Lm[1][2];
    ri[20] = d2 * Lm[0][2] - d0 * Lm[2][2];
    ri[21] = B[0];
    ri[22] = B[1];
    ri[23] = B[2];
    ri[24] = d1 * B[2] - d2 * B[1];
    ri[25] = d2 * B[0] - d0 * B[2];
    ri[26] = d0 * B[1] - d1 * B[0];
}

// Entry (a, b), a <= b, of zeta from the summed integers Z (A [6], L [9], Qm
// [6]) and the fraction f of the centre: with [f] c = f x c,
//   UU: s A,  UW: s (L - A [f]^T),  WW: s (Qm - L^T [f]^T - [f] L + [f] A [f]^T).
__device__ __forceinline__ double zeta_entry(int a, int b, const double* Z, const double f[3], double s)
{
    auto A = [&](int i, int j) { return Z[i == j ? i : 2 + i + j]; };
    auto L = [&](int i, int j) { return Z[6 + 3 * i + j]; };
    auto Qm = [&](int i, int j) { return Z[15 + (i == j ? i : 2 + i + j)]; };
    if (b < 3) return mul_x(s, A(a, b));
    const int j = b - 3, j1 = j == 2 ? 0 : j + 1, j2 = j == 0 ? 2 : j - 1;
    if (a < 3)   // (A [f]^T)_aj = f_j1 A_aj2 - f_j2 A_aj1
        return mul_x(s, add_x(L(a, j), -cross_x(f[j1], A(a, j2), f[j2], A(a, j1))));
    const int i = a - 3, i1 = i == 2 ? 0 : i + 1, i2 = i == 0 ? 2 : i - 1;
    const double u = cross_x(f[j1], L(j2, i), f[j2], L(j1, i));   // ([f] L)_ji
    const double v = cross_x(f[i1], L(i2, j), f[i2], L(i1, j));   // ([f] L)_ij
    const double w1 = cross_x(f[i1], A(i2, j2), f[i2], A(i1, j2)), w2 = cross_x(f[i1], A(i2, j1), f[i2], A(i1, j1));
    const double w = cross_x(f[j1], w1, f[j2], w2);              // ([f] A [f]^T)_ij
    return mul_x(s, add_x(add_x(Qm(i, j), w), -add_x(u, v)));
}

// links_block runs block bi of the nbi blocks of particle p; the block split
// (and with it the summation order) is the same in the single-box and the
// batched kernels, so both give identical bits.
template <class C>
__device__ __forceinline__ void links_block(const DevParams& P, const DevPtrs& D, int p, int bi, int nbi,
                                            LinkSmem<C>& sm)
{
    constexpr int K = kLinkK;
    {   // the particle's record, by the whole block
        static_assert(sizeof(DevPart) % 8 == 0, "copied in 64-bit words");
        const unsigned long long* src = (const unsigned long long*)(D.parts + p);
        unsigned long long* dst = (unsigned long long*)&sm.part;
        for (int k = threadIdx.x; k < (int)(sizeof(DevPart) / 8); k += kPartThreads) dst[k] = src[k];
    }
    __syncthreads();
    const DevPart& q = sm.part;
    int o[3];
    link_box(q, o);
    const int tot = P.side1[0] * P.side1[1] * P.side1[2];
    const int colf = threadIdx.x % kRowF, grpf = threadIdx.x / kRowF;
    const int coli = threadIdx.x % kRowI, grpi = threadIdx.x / kRowI;
    double accf = 0.0;
    long long acci = 0;
    for (int r = 0; (long long)r * NodeList<C>::kScanSlots * kPartThreads * nbi < tot; ++r) {
        const int cnt = list_nodes(P, o, P.side1, r, bi, nbi, tot, sm.list,
                                   [&](int n, int, int, int) { return D.mask[n] == 0 && D.bflag[n] != 0; });
        for (int s0 = 0; s0 < cnt; s0 += kRowNodes) {
            const int m = min(cnt - s0, kRowNodes);
            const int e = threadIdx.x % kRowNodes;
            if (e < m) {
                if ((int)threadIdx.x < kRowNodes)
                    link_row<C>(P, D, q, p, sm.list.n[s0 + e], sm.rf[e], sm.ri[e]);
                else
                    link_stress<C>(P, D, q, p, sm.list.n[s0 + e], sm.rf[e]);
            }
            __syncthreads();
            if (grpf < kRowGroups)
                for (int r = grpf; r < m; r += kRowGroups) accf += (double)sm.rf[r][colf];
            if (grpi < kRowGroups)
                for (int r = grpi; r < m; r += kRowGroups) acci += sm.ri[r][coli];
            __syncthreads();
        }
    }
    if (grpf < kRowGroups) sm.col[grpf][colf] = accf;
    if (grpi < kRowGroups) sm.col[grpi][kRowF + coli] = (double)acci;
    __syncthreads();
    if (threadIdx.x < kRow) {
        double s = 0.0;
#pragma unroll
        for (int g = 0; g < kRowGroups; ++g) s += sm.col[g][threadIdx.x];
        sm.tot[threadIdx.x] = s;
    }
    __syncthreads();
    double* part = D.link_part + ((size_t)p * kMaxPartBlocks + bi) * K;
    if (threadIdx.x < K) {
        // F0, T0, the integer sums of zeta, then the fluxes of psi and phi
        const int k = threadIdx.x;
        double v = k < 6 ? sm.tot[k] + sm.tot[kRowP + k] : (k < 27 ? sm.tot[kRowF + k - 6] : sm.tot[6 + k - 27]);
        if (k < 6) {
            const PrmR<double>& Qd = prm<double>(P);
            const double kc = (2.0 * Qd.rho0 + (P.thermo ? 1.5 * Qd.A : 0.0)) / 36.0;
            const double* B = sm.tot + kRowF + 21;
            const int a = k < 3 ? k : k - 3, a1 = a == 2 ? 0 : a + 1, a2 = a == 0 ? 2 : a - 1;
            const double c = k < 3 ? B[a] : add_x(B[3 + a], -cross_x(q.g.frd[a1], B[a2], q.g.frd[a2], B[a1]));
            v = fma_x(kc, c, v);
        }
        part[k] = v;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) sm.last = (atomicAdd(D.link_ticket + p, 1u) == (unsigned)nbi - 1u);
    __syncthreads();
    if (!sm.last) return;
    // last block of this particle: groups of threads add the blocks' partials
    // in block order
    __threadfence();
    constexpr int G = kPartThreads / K;
    {
        const int k = threadIdx.x % K, g = threadIdx.x / K;
        double s = 0.0;
        if (g < G) {
            // eight loads in flight (a loop of one at a time is a chain of L2
            // accesses: 10 of 54 thousand cycles with 42 blocks)
            const double* pb = D.link_part + (size_t)p * kMaxPartBlocks * K + k;
            for (int b0 = g; b0 < nbi; b0 += 8 * G) {
                double v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = b0 + j * G < nbi ? __ldcg(pb + (size_t)(b0 + j * G) * K) : 0.0;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (b0 + j * G < nbi) s += v[j];
            }
        }
        if (g < G) sm.red[g * K + k] = s;
        __syncthreads();
        if (threadIdx.x < K) {
            double v = 0.0;
#pragma unroll
            for (int gg = 0; gg < G; ++gg) v += sm.red[gg * K + threadIdx.x];
            sm.tot[threadIdx.x] = v;
        }
        __syncthreads();
    }
    {   // red is free again: zeta goes there, its three blocks on a warp each
        const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
        if (w < 3 && l < (w == 1 ? 9 : 6)) {
            const int i = w == 1 ? l / 3 : l < 3 ? 0 : l < 5 ? 1 : 2;   // row and column in the block
            const int j = w == 1 ? l % 3 : l < 3 ? l : l < 5 ? l - 2 : 2;
            const int a = w == 2 ? i + 3 : i, b = w == 0 ? j : j + 3;
            sm.red[a * 6 - (a * (a - 1)) / 2 + (b - a)] =
                zeta_entry(a, b, sm.tot + 6, q.g.frd, prm<double>(P).rho0 / 6.0);
        }
    }
    __syncthreads();
    particle_update(make_int3(P.nx, P.ny, P.nz), make_int3(P.per[0], P.per[1], P.per[2]), D.parts, D.link_ticket,
                    D.err, p, q, sm.tot, sm.red, sm.red + 32);   // totals in tot[0..K-1]
}

template <class C>
__global__ void __launch_bounds__(kPartThreads, part_blocks_per_sm<C>()) k_links(const __grid_constant__ DevParams P,
                                                         const __grid_constant__ DevPtrs D)
{
    __shared__ LinkSmem<C> sm;
    links_block<C>(P, D, blockIdx.y, blockIdx.x, gridDim.x, sm);
}

// ---------------------------------------------------------------------------
// S3 next to particles: halfway bounce-back on wall links, moving bounce-back
// with u_b = U + Omega x r + v_s on particle links.  A node next to several
// particles is collided by the lowest of them.
// ---------------------------------------------------------------------------
constexpr int kColNodes = kPartThreads;   // nodes of a round

template <class C>
struct ColSmem {
    using R = typename C::real;
    NodeList<C> list;
    R cub[19][kColNodes];   // 6 w rho0 c . u_b of the links of each node
};

template <class C>
__device__ __forceinline__ void collide_particles_block(const DevParams& P, const DevPtrs& D, int p, int bi, int nbi,
                                                        ColSmem<C>& sm)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    using S = typename C::pop_t;
    using V = Vec<R, 1>;
    const PrmR<R>& Q = prm<R>(P);
    const int NN = (int)P.N;
    const S* fs = (const S*)D.f_src;
    const F* phi = (const F*)D.phi_src;
    const F* force = (const F*)D.force;
    int o[3];
    link_box(D.parts[p], o);
    const int tot = P.side1[0] * P.side1[1] * P.side1[2];
    for (int r = 0; (long long)r * NodeList<C>::kScanSlots * kPartThreads * nbi < tot; ++r) {
        const int cnt = list_nodes(P, o, P.side1, r, bi, nbi, tot, sm.list,
                                   [&](int n, int, int, int) { return D.mask[n] == 0 && D.bflag[n] != 0; });
        for (int s0 = 0; s0 < cnt; s0 += kColNodes) {
            const int t = (int)threadIdx.x;
            if (s0 + t >= cnt) continue;
            const int n = sm.list.n[s0 + t];
            int x, y, z;
            node_coords(P, n, x, y, z);
            Around a;
            look_around(P, D, x, y, z, a);
            if (a.lo != p + 1) continue;
            // population j arrives from x - c_j = x + c_i (i = opp(j)); from a
            // wall or a particle it is the node's own population i, reflected
            V fl[19];
#pragma unroll
            for (int j = 0; j < 19; ++j) {
                const int i = opp(j);
                if (j == 0) {
                    fl[0].v = (R)PopStore<S>::load_dev(fs, n, 0, Q.rho0);
                    continue;
                }
                const bool st = a.stop >> i & 1u;
                const R raw = (R)PopStore<S>::load_dev(fs, st ? i * NN + n : j * NN + a.nb[i], i, Q.rho0);
                fl[j].v = raw;
            }
            const R dph = corr_r<R>(D, 1);
            R gphi[3];
            grad_phi_around<R, F>(a, phi, n, (R)phi[n] + dph, dph, gphi);
            const V f3[3] = {{(R)force[n]}, {(R)force[NN + n]}, {(R)force[2 * NN + n]}};
            for (int k = a.lo; k <= a.hi; ++k) {
                unsigned b = links_into(a, k);
                if (!b) continue;
                NodeLinks<R> l;
                node_links<R>(P, D.parts[k - 1], x, y, z, l);
                for (; b; b &= b - 1) {
                    const int i = __ffs((int)b) - 1;
                    const R w6 = i < 7 ? (R)(1.0 / 3.0) : (R)(1.0 / 6.0);
                    sm.cub[i][t] = mul_x(mul_x(w6, Q.rho0), link_cub<R>(l, i, gphi));
                }
            }
#pragma unroll
            for (int j = 1; j < 19; ++j) {
                const int i = opp(j);
                if (a.solid >> i & 1u) fl[j].v = add_x(fl[j].v, -sm.cub[i][t]);
            }
            V u[3];
            collide_values<R, 1>(Q, fl, f3, u);
            S* fd = (S*)D.f_dst;
            F* uo = (F*)D.u;
#pragma unroll
            for (int j = 0; j < 19; ++j) PopStore<S>::store_dev(fd, j * NN + n, j, Q.rho0, fl[j].v);
#pragma unroll
            for (int k = 0; k < 3; ++k) uo[k * NN + n] = (F)u[k].v;
        }
    }
}

template <class C>
__global__ void __launch_bounds__(kPartThreads, part_blocks_per_sm<C>()) k_collide_particles(const __grid_constant__ DevParams P,
                                                                     const __grid_constant__ DevPtrs D)
{
    __shared__ ColSmem<C> sm;
    collide_particles_block<C>(P, D, blockIdx.y, blockIdx.x, gridDim.x, sm);
}

// ---------------------------------------------------------------------------
// S4 next to particles, beside kz_scalars (which leaves those nodes out)
// ---------------------------------------------------------------------------
// Accessor of the transport body (scalars_compute_c) over global memory.
template <class F>
struct SAcc {
    int nb[19];
    int n, N;
    const uint8_t* mk;
    const F *psi, *phi, *mu, *u;
    __device__ __forceinline__ uint8_t mask(int i) const { return nb[i] >= 0 ? mk[nb[i]] : kWallSlot; }
    template <int K>
    __device__ __forceinline__ F get(int i) const
    {
        const int m = nb[i] >= 0 ? nb[i] : n;
        return K == 0 ? psi[m] : K == 1 ? phi[m] : K < 4 ? mu[2 * m + (K - 2)] : u[(K - 4) * N + m];
    }
};

template <class C>
__device__ __forceinline__ void scalars_particles_block(const DevParams& P, const DevPtrs& D, int p, int bi, int nbi,
                                                        NodeList<C>& list)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    int o[3];
    link_box(D.parts[p], o);
    const int tot = P.side1[0] * P.side1[1] * P.side1[2];
    for (int r = 0; (long long)r * NodeList<C>::kScanSlots * kPartThreads * nbi < tot; ++r) {
        const int cnt = list_nodes(P, o, P.side1, r, bi, nbi, tot, list,
                                   [&](int n, int, int, int) { return D.mask[n] == 0 && D.bflag[n] != 0; });
        for (int e = threadIdx.x; e < cnt; e += kPartThreads) {
            const int n = list.n[e];
            int x, y, z;
            node_coords(P, n, x, y, z);
            Around a;
            look_around(P, D, x, y, z, a);
            if (a.lo != p + 1) continue;
            SAcc<F> g;
#pragma unroll
            for (int i = 0; i < 19; ++i) g.nb[i] = a.nb[i];
            g.n = n;
            g.mk = D.mask;
            g.psi = (const F*)D.psi_src;
            g.phi = (const F*)D.phi_src;
            g.mu = (const F*)D.mu;
            g.u = (const F*)D.u;
            g.N = (int)P.N;
            const R dps = corr_r<R>(D, 0), dph = corr_r<R>(D, 1);
            const R ps = (R)g.psi[n] + dps, ph = (R)g.phi[n] + dph;
            // links into particles: no diffusive flux; the scalars leave with the
            // boundary velocity of the bounce-back rule, c.u_b g(x) -- weighted
            // w_i on the D3Q19 links of the finite-difference scheme, 1 on the six
            // D3Q7 links of the lattice-Boltzmann one; Janus production on the
            // m.(x - X) <= 0 side of each adjacent particle (any of the 18)
            R gphi[3];
            grad_phi_around<R, F>(a, g.phi, n, ph, dph, gphi);
            R out = 0, src = 0;   // sum of w c.u_b
            for (int k = a.lo; k <= a.hi; ++k) {
                unsigned b = links_into(a, k);
                if (!b) continue;
                const DevPart& q = D.parts[k - 1];
                NodeLinks<R> l;
                node_links<R>(P, q, x, y, z, l);
                if (cap_minus_at(l.q, l.D, 0, 0, 0)) src += PartR<R>::alpha(q);
                if (P.scheme) b &= 0x7Eu;
                for (; b; b &= b - 1) {
                    const int i = __ffs((int)b) - 1;
                    const R w = P.scheme ? (R)1 : (i < 7 ? (R)(1.0 / 18.0) : (R)(1.0 / 36.0));
                    out = fma_x(w, link_cub<R>(l, i, gphi), out);
                }
            }
            scalars_compute_c<C, true>(P, D, x, y, z, n, g, dps, dph, mul_x(-out, ps), mul_x(-out, ph), src);
        }
    }
}

template <class C>
__global__ void __launch_bounds__(kPartThreads, part_blocks_per_sm<C>()) k_scalars_particles(const __grid_constant__ DevParams P,
                                                                     const __grid_constant__ DevPtrs D)
{
    __shared__ NodeList<C> list;
    release_next_grid();   // k_cover_apply reads masks and positions beside this kernel
    scalars_particles_block<C>(P, D, blockIdx.y, blockIdx.x, gridDim.x, list);
}

}  // namespace lbdp
