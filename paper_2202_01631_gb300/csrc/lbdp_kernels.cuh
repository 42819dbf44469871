// lbdp_kernels.cuh -- the node and particle bodies of the lattice update and
// the particle kernels, templated on the precision configuration.  One step
// of a single box is
//   k_pt_part, k_f_part   per particle: chemical stress and force at the fluid
//                  nodes next to the particle (Eqs. chem_potentials,
//                  free_energy; the link-form divergence)
//   k_links        per particle: bounce-back and chemical-stress momentum sums
//                  over its boundary links, implicit velocity update, new
//                  position and orientation (Sec. "Particles")
//   k_collide_particles  collide-stream of the nodes next to particles: moving
//                  bounce-back plus phoretic slip on their particle links
//   kz_fused       (lbdp_zmarch.cuh) chemical potentials, stress, force and
//                  D3Q19 pull collide-stream of every other fluid node
//   k_scalars_particles  psi/phi transport next to particles, with Janus
//                  production (Eq. activity) and the flux into the moving
//                  surfaces
//   kz_scalars     (lbdp_zmarch.cuh) psi/phi transport (Eq.
//                  diffusion_reaction) and the k_d sink of every other node
//   k_cover_mark   per particle: solid mask at the new positions
//   k_cover_apply  per particle: covering/uncovering and boundary flags; the
//                  last block folds the psi/phi deficits into the uniform
//                  correction and moves the particles
// Every kernel is stencil or streaming work: no tensor cores.  Each body is a
// __device__ function of (parameters, pointers, node), so the single-box
// kernels and the batched kernels (lbdp_batch_kernels.cuh) run the same
// arithmetic.
//
// Precision: node and link arithmetic runs in the mode's real type R.  FP64
// is kept where the method needs it in every mode -- the solid/fluid and
// active-cap decisions (exact, unfused products and sums, as in the CPU
// oracle), the force/torque/conservation sums and the particle solve -- and
// nowhere else, because GB300 executes FP64 (and FP64 conversions) on a narrow
// pipe.
#pragma once

#include "lbdp_lattice.cuh"

namespace lbdp {

template <class Pop, class Fld, class Real>
struct Cfg {
    using pop_t = Pop;
    using fld_t = Fld;
    using real = Real;
};
using CfgF64 = Cfg<double, double, double>;
using CfgF32 = Cfg<float, float, float>;
using CfgF16 = Cfg<__half, float, float>;
using CfgBF16 = Cfg<__nv_bfloat16, float, float>;

// Threads of the kernels next to particles and of the covering kernels, and
// the box slots a thread of the former looks at.  About a tenth of a sphere's
// box lies next to it: a block of 128 threads finds the nodes of a full warp or
// two and takes a quarter of the registers of an SM.  FP64 takes fewer blocks:
// what they compute is taken from the bulk kernels on the same SM's FP64 pipe.
constexpr int kPartThreads = 128, kCoverThreads = 256;
__host__ __device__ constexpr int part_slots(bool fp64) { return fp64 ? 8 : 2; }

constexpr uint8_t kWallSlot = 0xFF;    // slot beyond a non-periodic wall

// ---------------------------------------------------------------------------
// precision accessors
// ---------------------------------------------------------------------------
template <class R>
__device__ __forceinline__ R corr_r(const DevPtrs& D, int k);
template <>
__device__ __forceinline__ float corr_r<float>(const DevPtrs& D, int k) { return D.corr_f[k]; }
template <>
__device__ __forceinline__ double corr_r<double>(const DevPtrs& D, int k) { return D.corr[k]; }

template <class R>
struct PartR;
template <>
struct PartR<float> {
    template <class Q>
    static __device__ __forceinline__ float U(const Q& q, int a) { return q.Uf[a]; }
    template <class Q>
    static __device__ __forceinline__ float W(const Q& q, int a) { return q.Wf[a]; }
    template <class Q>
    static __device__ __forceinline__ float mu_m(const Q& q) { return q.mu_mf; }
    template <class Q>
    static __device__ __forceinline__ float mu_p(const Q& q) { return q.mu_pf; }
    template <class Q>
    static __device__ __forceinline__ float Hk(const Q& q) { return q.Hk_f; }
    template <class Q>
    static __device__ __forceinline__ float alpha(const Q& q) { return q.alpha_f; }
};
template <>
struct PartR<double> {
    template <class Q>
    static __device__ __forceinline__ double U(const Q& q, int a) { return q.U[a]; }
    template <class Q>
    static __device__ __forceinline__ double W(const Q& q, int a) { return q.W[a]; }
    template <class Q>
    static __device__ __forceinline__ double mu_m(const Q& q) { return q.mu_m; }
    template <class Q>
    static __device__ __forceinline__ double mu_p(const Q& q) { return q.mu_p; }
    template <class Q>
    static __device__ __forceinline__ double Hk(const Q& q) { return q.Hk; }
    template <class Q>
    static __device__ __forceinline__ double alpha(const Q& q) { return q.alpha; }
};

// The fields of one particle that its boundary links use, copied from the
// device record into registers with independent loads (one memory round
// trip), for a kernel that reads them for many links of one node.
struct LinkPart {
    Geo g;
    float mf[3], smarg;
    float Uf[3], Wf[3], mu_pf, mu_mf;
    double m[3], U[3], W[3], mu_p, mu_m;
};

__device__ __forceinline__ LinkPart link_part(const DevPart& q)
{
    LinkPart l;
    l.g = q.g;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        l.mf[a] = q.mf[a];
        l.Uf[a] = q.Uf[a];
        l.Wf[a] = q.Wf[a];
        l.m[a] = q.m[a];
        l.U[a] = q.U[a];
        l.W[a] = q.W[a];
    }
    l.smarg = q.smarg;
    l.mu_pf = q.mu_pf;
    l.mu_mf = q.mu_mf;
    l.mu_p = q.mu_p;
    l.mu_m = q.mu_m;
    return l;
}

// ---------------------------------------------------------------------------
// shared device helpers
// ---------------------------------------------------------------------------

// c_i . (a, b, c) with the zero components of c_i dropped at compile time
// once the direction loop is unrolled (x + (-0) folds to x; a product with 0
// could not be removed because of NaN and signed-zero rules).
template <class R>
__device__ __forceinline__ R cdot(int i, R a, R b, R c)
{
    const R ta = cx(i) == 0 ? (R)-0.0 : (cx(i) > 0 ? a : -a);
    const R tb = cy(i) == 0 ? (R)-0.0 : (cy(i) > 0 ? b : -b);
    const R tc = cz(i) == 0 ? (R)-0.0 : (cz(i) > 0 ? c : -c);
    return ta + tb + tc;
}

// ---------------------------------------------------------------------------
// geometric decisions.  The oracle takes them in FP64 from exact offsets
// (|x - X|^2 < R^2 for solid nodes, m . r <= 0 for the cap side).  Here they
// are taken in FP32 from the integer/fraction split of the centre (Geo) and
// fall back to the oracle's FP64 arithmetic only when the FP32 value lies
// within its error bound of the threshold, so every decision is the oracle's
// while FP64 (a narrow pipe on GB300) is almost never executed.
// ---------------------------------------------------------------------------

// Integer offsets D of node (x, y, z) from centre g: x - X = D - fr.
__device__ __forceinline__ void int_offset(const DevParams& P, const Geo& g, int x, int y, int z, int D[3])
{
    D[0] = min_image_int(x, g.Xi[0], g.fl[0], P.nx, P.per[0]);
    D[1] = min_image_int(y, g.Xi[1], g.fl[1], P.ny, P.per[1]);
    D[2] = min_image_int(z, g.Xi[2], g.fl[2], P.nz, P.per[2]);
}

// FP32 error margins (host and device): the offset d = D - fr in FP32 is off
// by at most 2^-24 (1 + |d|), so |d|^2 near R^2 is off by less than
// 2^-24 (6 R^2 + 4 R + 1) including the rounding of R^2; m . r is off by less
// than 2^-24 (7 |r| + 2) for |r| <= R + 3.  The margins carry 8x of slack.
__host__ __device__ inline float solid_margin(double R) { return (float)(ldexp(1.0, -21) * (R * R + R + 1.0)); }
__host__ __device__ inline float side_margin(double R) { return (float)(ldexp(1.0, -21) * (R + 4.0)); }

// |x - X|^2 < R^2, the oracle's decision.
__device__ __forceinline__ bool solid_test(const Geo& g, const int D[3], float R2f, float marg, double R2)
{
    const float d0 = (float)D[0] - g.fr[0], d1 = (float)D[1] - g.fr[1], d2 = (float)D[2] - g.fr[2];
    const float q = dot_x(d0, d1, d2, d0, d1, d2);
    if (q < R2f - marg) return true;
    if (q > R2f + marg) return false;
    const double e[3] = {__dsub_rn((double)D[0], g.frd[0]), __dsub_rn((double)D[1], g.frd[1]),
                         __dsub_rn((double)D[2], g.frd[2])};
    return dot3_rn(e, e) < R2;
}

// Link midpoint offset r_b = (x - X) + c_i/2 in the arithmetic precision:
// exact in FP64, within 2^-24 (1 + |r|) in FP32.
template <class R>
__device__ __forceinline__ void link_offset_r(const Geo& g, const int D[3], int i, R r[3]);
template <>
__device__ __forceinline__ void link_offset_r<float>(const Geo& g, const int D[3], int i, float r[3])
{
    r[0] = ((float)D[0] + 0.5f * (float)cx(i)) - g.fr[0];
    r[1] = ((float)D[1] + 0.5f * (float)cy(i)) - g.fr[1];
    r[2] = ((float)D[2] + 0.5f * (float)cz(i)) - g.fr[2];
}
template <>
__device__ __forceinline__ void link_offset_r<double>(const Geo& g, const int D[3], int i, double r[3])
{
    r[0] = __dsub_rn(__dadd_rn((double)D[0], 0.5 * cx(i)), g.frd[0]);
    r[1] = __dsub_rn(__dadd_rn((double)D[1], 0.5 * cy(i)), g.frd[1]);
    r[2] = __dsub_rn(__dadd_rn((double)D[2], 0.5 * cz(i)), g.frd[2]);
}

// Wetting ghost of psi at the solid neighbour x + c_i of fluid node x,
// psi(x) + (H/kappa) c_i . n_hat at the link midpoint, as its difference
// from psi(x).
template <class R>
__device__ __forceinline__ R psi_ghost_diff(const DevParams& P, const DevPart& q, int x, int y, int z, int i)
{
    if (PartR<R>::Hk(q) == (R)0) return (R)0;
    int D[3];
    int_offset(P, q.g, x, y, z, D);
    R r[3];
    link_offset_r<R>(q.g, D, i, r);
    const R rn = sqrt(dot_x(r[0], r[1], r[2], r[0], r[1], r[2]));
    const R cn = cdot<R>(i, r[0], r[1], r[2]) / rn;
    return mul_x(PartR<R>::Hk(q), cn);
}

// The sums of the differences d that the Laplacian and the gradient need, per
// weight class: sa, sd = sum d over the axis and the diagonal directions,
// ga, gd = sum c d over them.
template <class R>
struct PsiSums {
    R sa, sd, ga[3], gd[3];
};

// Component k (0 x, 1 y, 2 z) of c_i for an i known only at run time: two bits
// per direction, c + 1, in one constant.
__host__ __device__ constexpr unsigned long long dir_code(int k)
{
    unsigned long long t = 0;
    for (int i = 0; i < 19; ++i) t |= (unsigned long long)((k == 0 ? cx(i) : k == 1 ? cy(i) : cz(i)) + 1) << (2 * i);
    return t;
}
template <int K>
__device__ __forceinline__ int dir_comp(int i)
{
    constexpr unsigned long long t = dir_code(K);
    return (int)((t >> (2 * i)) & 3ull) - 1;
}

// d / sqrt(a) rounded once (within 0.5001 ulp), for components of a unit vector:
// y is CUDA's FP32 inverse square root, e = 1 - a y^2 its residual, taken with
// the rounding of a y as a second term, and 1 / sqrt(a) = y (1 - e)^(-1/2) =
// y (1 + c) by the binomial series (|e| < 2^-20: two terms in FP64, one in FP32);
// the quotient adds d y's rounding and c d y to d y.  An IEEE square root and a
// division round twice and take longer: measured on GB300, a step with one
// sphere, FP32 24^3 46.7 us (IEEE 49.8), 128^3 188.5 (196.9); FP64 32^3 175.9
// (180.3), 96^3 1448 (1469).  Errors over random link points, largest and mean,
// in units of the rounding: ghost FP32 4.69, 0.393 (IEEE 5.38, 0.445), FP64 4.54,
// 0.391 (4.89, 0.437); slip FP32 8.14, 0.461 (10.16, 0.519), FP64 6.10, 0.458
// (7.85, 0.511).
template <class R>
struct InvNorm {
    R y, c;
    __device__ __forceinline__ R times(R d) const
    {
        const R q = mul_x(d, y);
        return add_x(q, fma_x(c, q, fma_x(d, y, -q)));
    }
};
template <class R>
__device__ __forceinline__ InvNorm<R> inv_norm(R a)
{
    const R y = (R)rsqrtf((float)a), t = mul_x(a, y), tl = fma_x(a, y, -t);
    const R e = fma_x(-tl, y, fma_x(-t, y, (R)1));
    return {y, sizeof(R) == 4 ? mul_x((R)0.5, e) : mul_x(e, fma_x((R)0.375, e, (R)0.5))};
}

// The wetting ghosts of fluid node (x, y, z) on its links into particle q (bit
// i of bits: direction i), added to the sums of the psi differences.  A loop
// over the links a node has, not over the 18 directions: the lanes of a warp
// at a sphere's surface hold different links, and a body per direction, taken
// by whichever lane needs it, made the blocks of kz_fused next to a sphere
// run twice as long as the rest of the grid (latency of its square root,
// division and particle loads, 18 times per slot).
// Measured on GB300, FP32, loop against unrolled bodies: kz_fused 201 -> 131
// us with one sphere R = 8 in 128^3, 66 -> 42 us in 24^3.
template <class R, class Q>
__device__ __forceinline__ void psi_ghosts(const DevParams& P, const Q& q, int x, int y, int z, unsigned bits,
                                           PsiSums<R>& s)
{
    const R Hk = PartR<R>::Hk(q);
    if (Hk == (R)0) return;
    int D[3];
    int_offset(P, q.g, x, y, z, D);
    R r0[3];   // x - X
    link_offset_r<R>(q.g, D, 0, r0);
    for (; bits; bits &= bits - 1) {
        const int i = __ffs((int)bits) - 1;
        const R c0 = (R)dir_comp<0>(i), c1 = (R)dir_comp<1>(i), c2 = (R)dir_comp<2>(i);
        const R r[3] = {fma_x((R)0.5, c0, r0[0]), fma_x((R)0.5, c1, r0[1]), fma_x((R)0.5, c2, r0[2])};
        const R gd = mul_x(Hk, inv_norm(dot_x(r[0], r[1], r[2], r[0], r[1], r[2]))
                                   .times(dot_x(c0, c1, c2, r[0], r[1], r[2])));
        const R ax = i < 7 ? gd : (R)0, dg = i < 7 ? (R)0 : gd;
        s.sa += ax;
        s.sd += dg;
        s.ga[0] = fma_x(c0, ax, s.ga[0]);
        s.ga[1] = fma_x(c1, ax, s.ga[1]);
        s.ga[2] = fma_x(c2, ax, s.ga[2]);
        s.gd[0] = fma_x(c0, dg, s.gd[0]);
        s.gd[1] = fma_x(c1, dg, s.gd[1]);
        s.gd[2] = fma_x(c2, dg, s.gd[2]);
    }
}

// Equilibrium population i of (rho, u) as its deviation from the rest
// equilibrium, f_eq - w_i rho0 =
// w_i [(rho - rho0) + rho (3 c.u + 4.5 (c.u)^2 - 1.5 u^2)], rounding written out.
template <class Real>
__device__ __forceinline__ Real geq_i(int i, Real rho, Real rho0, Real ux, Real uy, Real uz)
{
    const Real cu = cdot<Real>(i, ux, uy, uz);
    const Real uu = dot_x(ux, uy, uz, ux, uy, uz);
    const Real t = fma_x((Real)-1.5, uu, fma_x(mul_x((Real)4.5, cu), cu, mul_x((Real)3, cu)));
    return mul_x(wgt_r<Real>(i), fma_x(rho, t, add_x(rho, -rho0)));
}

__device__ __forceinline__ float tanh_r(float v) { return tanhf(v); }
__device__ __forceinline__ double tanh_r(double v) { return tanh(v); }

// phi0 = phi_b + E tanh psi (Eq. free_energy); with E = 0 it is phi_b and tanh
// is not evaluated.
template <class R>
__device__ __forceinline__ R phi0_of(const PrmR<R>& Q, R ps)
{
    return Q.E != (R)0 ? Q.phib + Q.E * tanh_r(ps) : Q.phib;
}

// Chemical potentials and (optionally) the chemical stress at one fluid node
// from ps = psi(x), d[i] = psi(x + c_i) - psi(x) (ghost-resolved; d[0] is not
// read) and ph = phi(x):
//   mu_psi = A(psi^3 - psi) - kappa lap psi - C E (phi - phi0)/cosh^2 psi,
//   mu_phi = C (phi - phi0),  phi0 = phi_b + E tanh psi          (Eq. chem_potentials)
//   P = p_iso I + kappa grad psi grad psi,
//   p_iso = psi mu_psi + phi mu_phi - f - kappa |grad psi|^2/2,
//   f = A psi^4/4 - A psi^2/2 + C (phi - phi0)^2/2.               (Eq. free_energy)
// P is returned by its four independent numbers: pt = (p_iso, grad psi).
// 1/cosh^2 is taken as 1 - tanh^2; with E = 0, phi0 = phi_b and the
// coupling term vanish, and tanh is not evaluated.  The 19-point Laplacian
// 6 sum_i w_i (psi(x+c_i) - psi(x)) sums the differences per weight class;
// the gradient 3 sum_i w_i c_i psi(x+c_i) sums the differences of opposite
// neighbours.
// Written for FP32: A psi (psi^2 - 1) and f + A/4 = A (psi^2 - 1)^2 / 4 + ...
// do not cancel in the bulk phases, the stencils act on differences, and
// p_iso is returned less the bulk pressure A/4.  A constant part of P exerts
// no force: the link-form divergence sums w_i c_i over all 18 directions of a
// node, and the particle stress sums w_i c_i and w_i r_b x c_i over the
// boundary links of a sphere, which vanish for the same reason.

template <class R>
__device__ __forceinline__ PsiSums<R> psi_sums(const R d[19])
{
    PsiSums<R> q;
    // the two weight classes summed in two halves each (shorter chains)
    q.sa = (d[1] + d[2] + d[3]) + (d[4] + d[5] + d[6]);
    q.sd = ((d[7] + d[8]) + (d[9] + d[10]) + (d[11] + d[12])) +
           ((d[13] + d[14]) + (d[15] + d[16]) + (d[17] + d[18]));
#pragma unroll
    for (int a = 0; a < 3; ++a) q.ga[a] = q.gd[a] = (R)0;
    // opposite pairs (j, j + 1), j odd: c_j = -c_{j+1}
#pragma unroll
    for (int j = 1; j < 19; j += 2) {
        const R df = d[j] - d[j + 1];
        R* acc = j < 7 ? q.ga : q.gd;
        if (cx(j) != 0) acc[0] += cx(j) > 0 ? df : -df;
        if (cy(j) != 0) acc[1] += cy(j) > 0 ? df : -df;
        if (cz(j) != 0) acc[2] += cz(j) > 0 ? df : -df;
    }
    return q;
}

template <class R>
__device__ __forceinline__ void mu_pressure(const PrmR<R>& Q, R ps, const PsiSums<R>& s, R ph, bool want_p, R& mps,
                                            R& mph, R pt[kPtFields])
{
    const R lap = fma_x(s.sa, (R)(1.0 / 3.0), s.sd * (R)(1.0 / 6.0));
    const R g0 = fma_x(s.ga[0], (R)(1.0 / 6.0), s.gd[0] * (R)(1.0 / 12.0));
    const R g1 = fma_x(s.ga[1], (R)(1.0 / 6.0), s.gd[1] * (R)(1.0 / 12.0));
    const R g2 = fma_x(s.ga[2], (R)(1.0 / 6.0), s.gd[2] * (R)(1.0 / 12.0));
    const R t = fma_x(ps, ps, (R)-1);   // psi^2 - 1
    R dphi;
    if (Q.E != (R)0) {
        const R th = tanh_r(ps);
        dphi = ph - (Q.phib + Q.E * th);
        mps = Q.A * ps * t - Q.kappa * lap - Q.C * Q.E * dphi * ((R)1 - th * th);
    } else {
        dphi = ph - Q.phib;
        mps = Q.A * ps * t - Q.kappa * lap;
    }
    mph = Q.C * dphi;
    if (!want_p) return;
    const R fs = (R)0.25 * Q.A * t * t + (R)0.5 * Q.C * dphi * dphi;   // f + A/4
    const R gg = g0 * g0 + g1 * g1 + g2 * g2;
    pt[0] = ps * mps + ph * mph - fs - (R)0.5 * Q.kappa * gg;   // less A/4
    pt[1] = g0;
    pt[2] = g1;
    pt[3] = g2;
}

// P . c_i of the stress pt = (p_iso, grad psi): p_iso c_i + kappa g (g . c_i).
template <class R>
__device__ __forceinline__ void pt_dot_c(int i, R kappa, const R pt[kPtFields], R out[3])
{
    const R ks = kappa * cdot<R>(i, pt[1], pt[2], pt[3]);
    out[0] = fma_x(ks, pt[1], cx(i) == 0 ? (R)0 : (cx(i) > 0 ? pt[0] : -pt[0]));
    out[1] = fma_x(ks, pt[2], cy(i) == 0 ? (R)0 : (cy(i) > 0 ? pt[0] : -pt[0]));
    out[2] = fma_x(ks, pt[3], cz(i) == 0 ? (R)0 : (cz(i) > 0 ? pt[0] : -pt[0]));
}

// psi(x) (with the correction) and the 18 ghost-resolved differences
// psi(x + c_i) - psi(x) of fluid node n, from global memory.
template <class R, class F>
__device__ __forceinline__ R gather_psi(const DevParams& P, const DevPtrs& D, const F* psi, int x, int y, int z,
                                        const int nb[19], R d[19])
{
    const R p0 = (R)psi[nb[0]];
    d[0] = (R)0;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        const int m = nb[i];
        if (m < 0) {
            d[i] = (R)0;
        } else {
            const uint8_t q = D.mask[m];
            d[i] = q ? psi_ghost_diff<R>(P, D.parts[q - 1], x, y, z, i) : (R)psi[m] - p0;
        }
    }
    return p0 + corr_r<R>(D, 0);
}

// FP64 block reduction: sums K values per thread over the block in a fixed
// order (warp shuffles, then warps in index order); the result is valid in
// thread 0.
template <int K>
__device__ void block_sum(double (&v)[K], double* smem /* [32*K] */)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    }
    if (lane == 0)
        for (int k = 0; k < K; ++k) smem[warp * K + k] = v[k];
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
        for (int w = 0; w < nw; ++w) s += smem[w * K + threadIdx.x];
        smem[32 * K - K + threadIdx.x] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int k = 0; k < K; ++k) v[k] = smem[32 * K - K + k];
    __syncthreads();
}

// FP64 block reduction over the threads whose values are not all zero (in the
// particle kernels most threads of a box hold none): those threads write
// their K values as rows, in thread order, into shared memory; G threads per
// value add rows g, g + G, ..., and thread k adds its G partials in order.
// The order depends only on which threads contribute, so the result is
// deterministic.  It is left in sm[0..K-1]; sm holds
// block_rows_bytes<K>(blockDim.x) bytes (results, 32 warp counts and the G x K
// partials below sm[256], rows from there).  blockDim.x >= G K.
template <int K>
__host__ __device__ constexpr size_t block_rows_bytes(int threads)
{
    return (size_t)(256 + threads * K) * sizeof(double);
}

template <int K>
__device__ void block_sum_rows(const double (&v)[K], double* sm)
{
    constexpr int G = 16;
    static_assert(G * K <= 176, "reduction layout");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int* wcount = (int*)(sm + 64);
    double* part = sm + 80;
    double* rows = sm + 256;
    bool nz = false;
#pragma unroll
    for (int k = 0; k < K; ++k) nz = nz || (v[k] != 0.0);
    const unsigned bal = __ballot_sync(0xffffffffu, nz);
    if (lane == 0) wcount[warp] = __popc(bal);
    __syncthreads();
    int base = 0, total = 0;
    for (int w = 0; w < nw; ++w) {
        const int c = wcount[w];
        base += w < warp ? c : 0;
        total += c;
    }
    if (nz) {
        double* row = rows + (size_t)(base + __popc(bal & ((1u << lane) - 1u))) * K;
#pragma unroll
        for (int k = 0; k < K; ++k) row[k] = v[k];
    }
    __syncthreads();
    const int t = threadIdx.x;
    if (t < G * K) {
        const int k = t % K, g = t / K;
        double s = 0.0;
        for (int r = g; r < total; r += G) s += rows[(size_t)r * K + k];
        part[g * K + k] = s;
    }
    __syncthreads();
    if (t < K) {
        double s = 0.0;
#pragma unroll
        for (int g = 0; g < G; ++g) s += part[g * K + t];
        sm[t] = s;
    }
    __syncthreads();
}

// Lattice node of slot t in a box of edges s[3] starting at o[3]; false when
// the node falls beyond a wall.
__device__ __forceinline__ bool box_node(const DevParams& P, const int o[3], const int s[3], int t, int& x, int& y,
                                         int& z)
{
    x = wrap_coord(o[0] + t % s[0], P.nx, P.per[0]);
    y = wrap_coord(o[1] + (t / s[0]) % s[1], P.ny, P.per[1]);
    z = wrap_coord(o[2] + t / (s[0] * s[1]), P.nz, P.per[2]);
    return x >= 0 && y >= 0 && z >= 0;
}

// ---------------------------------------------------------------------------
// neighbour access of the stencil bodies.  A body sees node x through an
// accessor: mask(i) is the mask of neighbour x + c_i (kWallSlot beyond a
// wall) and get<k>(i) the value of field k there (own(k) = get<k>(0)).  Where
// mask(i) is not 0 the bodies do not use get<k>(i) except multiplied by 0.
// GAcc reads global memory through the D3Q19 neighbour indices; the
// accessors of lbdp_zmarch.cuh read planes staged in shared memory.  All hand
// the same values to the same arithmetic.
// ---------------------------------------------------------------------------
template <class F, int NF>
struct GAcc {
    int nb[19];
    int n;
    const uint8_t* mk;
    const F* f[NF];
    __device__ __forceinline__ const DevPart& part(const DevPtrs& D, int k) const { return D.parts[k]; }
    __device__ __forceinline__ int at(int i) const { return nb[i] >= 0 ? nb[i] : n; }
    __device__ __forceinline__ uint8_t mask(int i) const { return nb[i] >= 0 ? mk[at(i)] : kWallSlot; }
    template <int K>
    __device__ __forceinline__ F get(int i) const
    {
        return f[K][at(i)];
    }
};

// Whether node (x, y, z) lies next to a wall (a non-periodic box face).
__device__ __forceinline__ bool near_wall(const DevParams& P, int x, int y, int z)
{
    return (!P.per[0] && (x == 0 || x == P.nx - 1)) || (!P.per[1] && (y == 0 || y == P.ny - 1)) ||
           (!P.per[2] && (z == 0 || z == P.nz - 1));
}

// ---------------------------------------------------------------------------
// S1: chemical potentials and pressure tensor, one thread per node.  Every
// neighbour load is issued before any decision (walls clamp to the node
// itself), so the loads overlap instead of waiting behind mask branches.
// ---------------------------------------------------------------------------
// Fields of the chemical-potential body: 0 psi, 1 phi.  mup_values returns
// mu_psi, mu_phi and (when P.thermo) the pressure tensor of fluid node
// (x, y, z).
// dps, dph: the uniform psi/phi correction still to be added (corr_r); a
// kernel that loops over many nodes reads them once.
template <class C, class A>
__device__ __forceinline__ void mup_values(const DevParams& P, const DevPtrs& D, int x, int y, int z, const A& a,
                                           typename C::real dps, typename C::real dph, typename C::real& mps,
                                           typename C::real& mph, typename C::real (&pt)[kPtFields])
{
    using R = typename C::real;
    const PrmR<R>& Q = prm<R>(P);
    // differences from psi(x): the uniform correction cancels in them; 0
    // towards a wall (neutral) or, until psi_ghosts adds it, a particle
    R d[19];
    uint8_t mk[19];
    const R p0 = (R)a.template get<0>(0);
    d[0] = (R)0;
    unsigned ids = 0;   // bit i: neighbour i lies inside a particle
    int lo = 255, hi = 0;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        mk[i] = a.mask(i);
        d[i] = (R)a.template get<0>(i) - p0;
    }
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        if (mk[i]) d[i] = (R)0;
        if (mk[i] && mk[i] != kWallSlot) {
            ids |= 1u << i;
            lo = min(lo, (int)mk[i]);
            hi = max(hi, (int)mk[i]);
        }
    }
    PsiSums<R> s = psi_sums<R>(d);
    for (int k = lo; k <= hi; ++k) {   // the particles next to this node: one, nearly always
        unsigned bits = ids;
        if (lo != hi) {
            bits = 0;
#pragma unroll
            for (int i = 1; i < 19; ++i) bits |= mk[i] == k ? 1u << i : 0u;
        }
        if (bits) psi_ghosts<R>(P, a.part(D, k - 1), x, y, z, bits, s);
    }
    mu_pressure<R>(Q, p0 + dps, s, (R)a.template get<1>(0) + dph, P.thermo != 0, mps, mph, pt);
}

// ---------------------------------------------------------------------------
// S2: force on the fluid, F = g - div P in the link form
//   -6 sum_i w_i [(P(x) + P~_i)/2] . c_i = -3 sum_i w_i P~_i . c_i
// (sum_i w_i c_i = 0), with P~_i = P(x) at solid and wall neighbours, and
// P~_i . c_i = p_iso c_i + kappa g (g . c_i) from the stress (p_iso, g) of
// mu_pressure.
// ---------------------------------------------------------------------------
// fdiv_values returns the force of a fluid node (rounded to the field type, as
// stored); fdiv_compute stores it.  Fields of the accessor: the stress
// (p_iso, g_x, g_y, g_z).
template <class C, class A>
__device__ __forceinline__ void fdiv_values(const DevParams& P, const A& a, typename C::real& Fxo,
                                            typename C::real& Fyo, typename C::real& Fzo)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    const PrmR<R>& Q = prm<R>(P);
    R Fx = Q.g[0], Fy = Q.g[1], Fz = Q.g[2];
    if (P.thermo) {
        const R o0 = (R)a.template get<0>(0), o1 = (R)a.template get<1>(0), o2 = (R)a.template get<2>(0);
        const R o3 = (R)a.template get<3>(0);
        R d0 = 0, d1 = 0, d2 = 0;   // sum_i w_i (g . c_i) g
        R e0 = 0, e1 = 0, e2 = 0;   // sum_i w_i c_i p_iso
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const bool own = a.mask(i) != 0;
            const R pi = own ? o0 : (R)a.template get<0>(i);
            const R gx = own ? o1 : (R)a.template get<1>(i);
            const R gy = own ? o2 : (R)a.template get<2>(i);
            const R gz = own ? o3 : (R)a.template get<3>(i);
            const R w = wgt_r<R>(i);
            const R ws = w * cdot<R>(i, gx, gy, gz);
            d0 = fma_x(ws, gx, d0);
            d1 = fma_x(ws, gy, d1);
            d2 = fma_x(ws, gz, d2);
            if (cx(i) != 0) e0 = fma_x(cx(i) > 0 ? w : -w, pi, e0);
            if (cy(i) != 0) e1 = fma_x(cy(i) > 0 ? w : -w, pi, e1);
            if (cz(i) != 0) e2 = fma_x(cz(i) > 0 ? w : -w, pi, e2);
        }
        Fx -= (R)3 * fma_x(Q.kappa, d0, e0);
        Fy -= (R)3 * fma_x(Q.kappa, d1, e1);
        Fz -= (R)3 * fma_x(Q.kappa, d2, e2);
    }
    Fxo = (R)(F)Fx;
    Fyo = (R)(F)Fy;
    Fzo = (R)(F)Fz;
}

template <class C, class A>
__device__ __forceinline__ void fdiv_compute(const DevParams& P, const DevPtrs& D, int n, const A& a)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    const size_t N = (size_t)P.N;
    R Fx, Fy, Fz;
    fdiv_values<C>(P, a, Fx, Fy, Fz);
    F* force = (F*)D.force;
    force[n] = (F)Fx;
    force[N + n] = (F)Fy;
    force[2 * N + n] = (F)Fz;
}

// Rotate the unit vector m by the angle |w| about w (Rodrigues):
//   m' = m cos|w| + (w x m) sin|w|/|w| + w (w . m)(1 - cos|w|)/|w|^2,
// then renormalise.  For |w| < 0.1 both ratios are their Taylor series in
// |w|^2, exact to double precision with six terms; the renormalisation is one
// Newton step of 1/sqrt around 1 (|m'| = 1 up to rounding).
// By one warp (all lanes call it): lanes 0, 1 and 2 hold the components of m, w
// and the result, and one evaluates each series.
__device__ __forceinline__ double rotate_unit(const double (&m)[3], const double (&w)[3], int lane)
{
    const double w2 = dot_x(w[0], w[1], w[2], w[0], w[1], w[2]);
    double s1, c1, cw;
    if (w2 < 0.01) {
        // s1 = 1 - w2/6 (1 - w2/20 (...)) in the even lanes, 2 c1 = 1 - w2/12 (1 -
        // w2/30 (...)) in the odd ones.  The ten quotients w2 / (k + 2)(k + 3) are
        // a lane's each: one division instead of a chain of five
        const double d = -w2 / (double)((lane + 2) * (lane + 3));
        double t = 1.0;
#pragma unroll
        for (int k = 4; k >= 0; --k) t = fma_x(__shfl_sync(0xffffffffu, d, 2 * k + (lane & 1)), t, 1.0);
        s1 = __shfl_sync(0xffffffffu, t, 0);
        c1 = 0.5 * __shfl_sync(0xffffffffu, t, 1);
        cw = fma_x(-w2, c1, 1.0);
    } else {
        const double wn = sqrt(w2);
        s1 = sin(wn) / wn;
        cw = cos(wn);
        c1 = (1.0 - cw) / w2;
    }
    const int a = lane < 3 ? lane : 0, a1 = a == 2 ? 0 : a + 1, a2 = a == 0 ? 2 : a - 1;
    auto at = [](const double (&v)[3], int k) { return k == 0 ? v[0] : k == 1 ? v[1] : v[2]; };
    const double wxm = cross_x(at(w, a1), at(m, a2), at(w, a2), at(m, a1));
    const double wm = mul_x(dot_x(w[0], w[1], w[2], m[0], m[1], m[2]), c1);
    const double r = fma_x(at(w, a), wm, fma_x(wxm, s1, mul_x(at(m, a), cw)));
    const double r0 = __shfl_sync(0xffffffffu, r, 0), r1 = __shfl_sync(0xffffffffu, r, 1), r2 = __shfl_sync(0xffffffffu, r, 2);
    const double nn2 = dot_x(r0, r1, r2, r0, r1, r2);
    return mul_x(r, fma_x(-0.5, nn2, 1.5));
}

// Implicit particle update of particle p by the whole last block (at least
// four warps), from the link totals tot[0..5] (F0[3], T0[3]), the upper
// triangle z[21] of zeta and the surface fluxes tot[kLinkGpsi...]:
//   (Mdiag + zeta) V(t+1) = Mdiag V(t) + [F0 + impulses + loads; T0 + ...]
// (symmetric positive definite), force and torque F0 - zeta V, then the
// position and orientation after the step.  FP64 throughout.  A warp issues one
// FP64 instruction in 64 cycles whether it depends on the one before or not, so
// what counts is the longest instruction stream of a warp: a thread per element
// of the matrix, eliminated above and below the pivot at once (a reciprocal, a
// product and an update per pivot, no substitution afterwards), then the rest
// shared by four warps.  By Cholesky in one warp with everything after it in
// lanes of that warp it took 16 thousand cycles of k_links, 25 thousand with a
// spinning sphere; so 9 and 13 thousand (24^3 FP32: 54 -> 48 us a step, with the
// block sums loaded eight at a time).
// G is scratch for 48 doubles.
static __device__ __noinline__ void particle_update(int3 L3, int3 per3, DevPart* parts, unsigned* ticket, int* err, int p,
                                             const DevPart& q, const double* tot, const double* z, double* G)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* V = G + 42;   // velocity and spin after the step
    // element (a, c) of [Mdiag + zeta | b] at G[7 a + c]
    auto zeta = [&](int a, int c) {
        const int lo = min(a, c), hi = max(a, c);
        return z[lo * 6 - (lo * (lo - 1)) / 2 + (hi - lo)];
    };
    auto load = [&](int a) {   // F0 + impulses + loads
        return a < 3 ? add_x(add_x(tot[a], q.imp_f[a]), q.ext_f[a])
                     : add_x(add_x(tot[a], q.imp_t[a - 3]), q.ext_t[a - 3]);
    };
    auto vel = [&](int a) { return a < 3 ? q.U[a] : q.W[a - 3]; };
    if (q.fixed) {
        if (threadIdx.x < 6) V[threadIdx.x] = vel(threadIdx.x);
    } else {
        const int e = threadIdx.x, a = e / 7, c = e % 7;
        const bool mine = e < 42;
        double x = 0.0;
        if (mine) {
            const double M = a < 3 ? q.M : q.I;
            x = c == 6 ? fma_x(M, vel(a), load(a)) : a == c ? add_x(zeta(a, c), M) : zeta(a, c);
            G[e] = x;
        }
        __syncthreads();
        bool ok = true;
        double ra = 0.0;   // reciprocal of the pivot of row a
#pragma unroll 1
        for (int j = 0; j < 6; ++j) {
            const double piv = G[8 * j];
            double f = 0.0, g = 0.0;
            if (mine) {
                f = G[7 * a + j];
                g = G[7 * j + c];
            }
            __syncthreads();
            if (mine) {
                ok = ok && (unsigned)__double2hiint(piv) - 1u < 0x7ff00000u;   // positive, not NaN
                const double r = __drcp_rn(fmax(piv, 1e-300));
                // the pivot row keeps its elements; columns up to j are never read again
                if (a == j)
                    ra = r;
                else
                    G[e] = x = fma_x(-mul_x(f, r), g, x);
            }
            __syncthreads();
        }
        if (mine && c == 6) V[a] = mul_x(x, ra);
        if (!ok && e == 0) atomicOr(err, kErrSolve);
    }
    __syncthreads();
    DevPart& dp = parts[p];
    if (warp == 0) {
        if (lane == 0) ticket[p] = 0u;
        if (lane < 6) {
            double zv = 0.0;
#pragma unroll 1
            for (int c = 0; c < 6; ++c) zv = fma_x(zeta(lane, c), V[c], zv);
            const double f = add_x(load(lane), -zv);
            if (lane < 3)
                dp.force[lane] = f;
            else
                dp.torque[lane - 3] = f;
        }
    } else if (warp == 1) {
        if (lane < 3) {
            const int a = lane;
            const int L = a == 0 ? L3.x : (a == 1 ? L3.y : L3.z);
            const int per = a == 0 ? per3.x : (a == 1 ? per3.y : per3.z);
            const double v = V[a], w = V[3 + a];
            dp.U[a] = v;
            dp.W[a] = w;
            dp.Uf[a] = (float)v;
            dp.Wf[a] = (float)w;
            dp.imp_f[a] = 0.0;
            dp.imp_t[a] = 0.0;
            double X = add_x(q.X[a], v);
            if (per) {
                if (X >= L)
                    X -= L;
                else if (X < 0.0)
                    X += L;
            } else if (X - q.R < 1.0 || X + q.R > L - 2.0) {
                atomicOr(err, kErrWall);
            }
            dp.Xn[a] = X;
            const double f = floor(X);
            const double fr = X - f;
            dp.gn.Xi[a] = (int)f;
            dp.gn.frd[a] = fr;
            dp.gn.fr[a] = (float)fr;
            dp.gn.fl[a] = (fr > 0.0 ? kFrPos : 0) | (fr < 0.5 ? kFrBelowHalf : 0) | (fr > 0.5 ? kFrAboveHalf : 0);
        }
    } else if (warp == 2) {
        const double w3[3] = {V[3], V[4], V[5]}, m[3] = {q.m[0], q.m[1], q.m[2]};
        double mn = lane == 0 ? m[0] : lane == 1 ? m[1] : m[2];
        if (w3[0] != 0.0 || w3[1] != 0.0 || w3[2] != 0.0) mn = rotate_unit(m, w3, lane);   // uniform in the warp
        if (lane < 3) dp.mn[lane] = mn;
    } else if (warp == 3 && lane < 2) {
        // psi, phi carried into the surface: sum 6 w g c.u_b with u_b at V(t+1)
        const double* g = tot + (lane == 0 ? kLinkGpsi : kLinkGphi);
        double s = g[6];
#pragma unroll 1
        for (int c = 0; c < 6; ++c) s = fma_x(g[c], V[c], s);
        (lane == 0 ? dp.wall_psi : dp.wall_phi) = s;
    }
}

// Halfway bounce-back of a bulk node next to a wall: a link whose source lies
// beyond a wall brings back the node's own population of the opposite
// direction.
template <class C>
__device__ __forceinline__ void bulk_wall_links(const DevParams& P, const DevPtrs& D, int x, int y, int z,
                                                typename C::real (&fl)[19])
{
    using R = typename C::real;
    using S = typename C::pop_t;
    const int n = x + P.nx * (y + P.ny * z);
    const int NN = (int)P.N;
    const S* fs = (const S*)D.f_src;
    const bool wx[3] = {!P.per[0] && x == 0, false, !P.per[0] && x == P.nx - 1};
    const bool wy[3] = {!P.per[1] && y == 0, false, !P.per[1] && y == P.ny - 1};
    const bool wz[3] = {!P.per[2] && z == 0, false, !P.per[2] && z == P.nz - 1};
#pragma unroll
    for (int j = 1; j < 19; ++j)
        if (wx[1 - cx(j)] || wy[1 - cy(j)] || wz[1 - cz(j)])
            fl[j] = (R)PopStore<S>::load_dev(fs, opp(j) * NN + n, opp(j), prm<R>(P).rho0);
}

// ---------------------------------------------------------------------------
// S4: psi and phi transport, production and sink, one thread per node
// ---------------------------------------------------------------------------
// psi and phi side by side: on sm_100-class GPUs two FP32 values go through
// one packed instruction (each lane rounds as the scalar operation does);
// FP64 keeps two scalar operations.
template <class R>
struct alignas(2 * sizeof(R)) Two {
    R a, b;
};
__device__ __forceinline__ Two<float> fma2(Two<float> x, Two<float> y, Two<float> z)
{
    const float2 r = __ffma2_rn(make_float2(x.a, x.b), make_float2(y.a, y.b), make_float2(z.a, z.b));
    return {r.x, r.y};
}
__device__ __forceinline__ Two<double> fma2(Two<double> x, Two<double> y, Two<double> z)
{
    return {fma_x(x.a, y.a, z.a), fma_x(x.b, y.b, z.b)};
}
__device__ __forceinline__ Two<float> add2(Two<float> x, Two<float> y)
{
    const float2 r = __fadd2_rn(make_float2(x.a, x.b), make_float2(y.a, y.b));
    return {r.x, r.y};
}
__device__ __forceinline__ Two<double> add2(Two<double> x, Two<double> y) { return {add_x(x.a, y.a), add_x(x.b, y.b)}; }
__device__ __forceinline__ Two<double> sub2(Two<double> x, Two<double> y)
{
    return {add_x(x.a, -y.a), add_x(x.b, -y.b)};
}
__device__ __forceinline__ Two<float> sub2(Two<float> x, Two<float> y)
{
    Two<float> r;
    asm("{.reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n sub.rn.f32x2 c, a, b;\n"
        " mov.b64 {%0, %1}, c;}"
        : "=f"(r.a), "=f"(r.b)
        : "f"(x.a), "f"(x.b), "f"(y.a), "f"(y.b));
    return r;
}

// Lattice-Boltzmann transport (scalar_scheme 1): D3Q7, weights 1/4 (rest)
// and 1/8, c_s^2 = 1/4, relaxation time 1, Gamma = 2M.  The post-collision
// distributions are then the equilibrium of the node's own fields,
//   h_i* = M mu + g c_i.u / 2   (i = 1..6),   h_0* = g - 6 M mu (+ sources),
// so the pull stream needs no stored distributions: the node's new total is
//   g'(x) = h_0*(x) + sum_i  h_i*(x - c_i)          (fluid source)
//                          | h_ibar*(x)              (wall: bounce-back)
//                          | h_ibar*(x) - g(x) c_ibar.u_b   (moving surface)
// with ibar the direction from x to the source.  Written per link from x
// towards y = x + c_j (j = ibar), after taking M mu(x) from each of the six
// terms of h_0*:
//   fluid y: M (mu(y) - mu(x)) - g(y) c_j.u(y) / 2,   otherwise g(x) c_j.u(x) / 2
// and -g(x) c_j.u_b more on a particle link (k_scalars_particles).
template <class C, bool kBoundary, class A>
__device__ __forceinline__ void scalars_compute_lb(const DevParams& P, const DevPtrs& D, int x, int y, int z,
                                                   int n, const A& a, typename C::real dps, typename C::real dph,
                                                   typename C::real eps, typename C::real eph, typename C::real src)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    const PrmR<R>& Q = prm<R>(P);
    const R ps = (R)a.template get<0>(0) + dps, ph = (R)a.template get<1>(0) + dph;
    const R a0 = (R)a.template get<2>(0), b0 = (R)a.template get<3>(0);
    const R ux = (R)a.template get<4>(0), uy = (R)a.template get<5>(0), uz = (R)a.template get<6>(0);
    const R ma0 = Q.Mpsi * a0, mb0 = Q.Mphi * b0;
    const R hps = (R)0.5 * ps, hph = (R)0.5 * ph;
    R sps = 0, sph = 0;
    bool solid_nb = false;
#pragma unroll
    for (int i = 1; i < 7; ++i) {
        const uint8_t mk = a.mask(i);
        const R cu0 = cdot<R>(i, ux, uy, uz);
        const R cu1 = cdot<R>(i, (R)a.template get<4>(i), (R)a.template get<5>(i), (R)a.template get<6>(i));
        const R psm = (R)a.template get<0>(i) + dps, phm = (R)a.template get<1>(i) + dph;
        const R tps = mk ? mul_x(hps, cu0) : fma_x(Q.Mpsi, (R)a.template get<2>(i), -ma0) - (R)0.5 * mul_x(psm, cu1);
        const R tph = mk ? mul_x(hph, cu0) : fma_x(Q.Mphi, (R)a.template get<3>(i), -mb0) - (R)0.5 * mul_x(phm, cu1);
        sps += tps;
        sph += tph;
        solid_nb = solid_nb || (mk != 0 && mk != kWallSlot);
    }
#pragma unroll
    for (int i = 7; i < 19; ++i) {
        const uint8_t mk = a.mask(i);
        solid_nb = solid_nb || (mk != 0 && mk != kWallSlot);
    }
    R hn_src = 0;
    if (kBoundary) {
        sps = add_x(sps, eps);
        sph = add_x(sph, eph);
        hn_src = src;
    } else if (solid_nb) {
        return;   // left to k_scalars_particles
    }
    // the stored value plus every increment of the step (correction, fluxes,
    // sink, source) summed first: one rounding of the O(1) field per step
    const R ps0 = (R)a.template get<0>(0), ph0 = (R)a.template get<1>(0);
    const R pn = ps0 + (dps + sps);
    const R hn = ph0 + (((dph + sph) - Q.kd * (ph - phi0_of(Q, ps))) + hn_src);
    ((F*)D.psi_dst)[n] = (F)pn;
    ((F*)D.phi_dst)[n] = (F)hn;
}

// Fields of the transport body: 0 psi, 1 phi, 2 mu_psi, 3 mu_phi, 4..6 u.
// kBoundary: a node next to a particle, whose links there carry eps, eph
// (before the factor 6 of the finite-difference scheme) and whose production
// is src; otherwise such nodes are left to k_scalars_particles.
// dps, dph as for mup_values.
template <class C, bool kBoundary, class A>
__device__ __forceinline__ void scalars_compute_c(const DevParams& P, const DevPtrs& D, int x, int y, int z, int n,
                                                  const A& a, typename C::real dps, typename C::real dph,
                                                  typename C::real eps = 0, typename C::real eph = 0,
                                                  typename C::real src = 0)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    if (P.scheme) {
        scalars_compute_lb<C, kBoundary>(P, D, x, y, z, n, a, dps, dph, eps, eph, src);
        return;
    }
    const PrmR<R>& Q = prm<R>(P);
    const R ps = (R)a.template get<0>(0) + dps, ph = (R)a.template get<1>(0) + dph;
    const R a0 = (R)a.template get<2>(0), b0 = (R)a.template get<3>(0);
    const R ux = (R)a.template get<4>(0), uy = (R)a.template get<5>(0), uz = (R)a.template get<6>(0);
    const R ma0 = Q.Mpsi * a0, mb0 = Q.Mphi * b0;
    const Two<R> g0{ps, ph}, corr{dps, dph}, mob{Q.Mpsi, Q.Mphi}, nmu0{-ma0, -mb0};
    Two<R> sg{0, 0};
    bool solid_nb = false;
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        const uint8_t mk = a.mask(i);
        const R cu0 = cdot<R>(i, ux, uy, uz);
        const R cu1 = cdot<R>(i, (R)a.template get<4>(i), (R)a.template get<5>(i), (R)a.template get<6>(i));
        const R ub = (R)0.5 * (cu0 + cu1);
        const Two<R> gm = add2(Two<R>{(R)a.template get<0>(i), (R)a.template get<1>(i)}, corr);
        // donor-cell upwind advection, diffusion M (mu(x + c) - mu(x)), for
        // psi and phi together
        // -ub g_upwind = -ua g(x) - ud g(x + c) with ua = max(ub, 0), ud = ub - ua:
        // one of the two products is zero, so this is the single rounding of
        // the upwind term, with a max instead of a compare and two selects
        const R ua = ub > (R)0 ? ub : (R)0, ud = ub - ua;
        Two<R> t = fma2(mob, Two<R>{(R)a.template get<2>(i), (R)a.template get<3>(i)}, nmu0);
        t = fma2(Two<R>{-ud, -ud}, gm, t);
        t = fma2(Two<R>{-ua, -ua}, g0, t);
        // links to walls and particles carry no flux here (particle links are
        // handled below)
        const R w = wgt_r<R>(i);
        sg = fma2(Two<R>{w, w}, mk ? Two<R>{0, 0} : t, sg);
        solid_nb = solid_nb || (mk != 0 && mk != kWallSlot);
    }
    R sps = sg.a, sph = sg.b;
    R hn_src = 0;
    if (kBoundary) {
        sps = add_x(sps, eps);
        sph = add_x(sph, eph);
        hn_src = src;
    } else if (solid_nb) {
        return;   // left to k_scalars_particles
    }
    // the stored value plus every increment of the step (correction, fluxes,
    // sink, source) summed first: one rounding of the O(1) field per step
    const R ps0 = (R)a.template get<0>(0), ph0 = (R)a.template get<1>(0);
    const R pn = ps0 + fma_x((R)6, sps, dps);
    const R hn = ph0 + ((fma_x((R)6, sph, dph) - Q.kd * (ph - phi0_of(Q, ps))) + hn_src);
    ((F*)D.psi_dst)[n] = (F)pn;
    ((F*)D.phi_dst)[n] = (F)hn;
}

// ---------------------------------------------------------------------------
// S7: covering / uncovering.  The cover box of particle p holds its old and
// new position with a margin that contains every neighbour of a node that can
// change.  k_cover_mark writes the new mask of the box (ownership over all
// particles at their new positions, first match); k_cover_apply moves the
// fields of the changed nodes, refreshes the boundary flags of the box and
// sums what the moving surfaces carried out of the fluid.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cover_origin(const DevParams& P, const DevPart& q, int o[3])
{
    for (int a = 0; a < 3; ++a) {
        const int L = a == 0 ? P.nx : (a == 1 ? P.ny : P.nz);
        const int i0 = q.g.Xi[a], i1 = q.gn.Xi[a];
        int lo = min(i0, i1);
        // on a periodic axis the two centres may sit on opposite sides of the
        // wrap; take the lower end of the shorter arc
        if (P.per[a] && abs(i0 - i1) > L / 2) lo = max(i0, i1);
        // floor(lo) - ceil(R) <= floor(lo - R): the box starts at or below the
        // lowest node that can change or neighbour a change
        o[a] = lo - q.Rc - 3;
    }
}

template <class C>
__device__ __forceinline__ void cover_mark_block(const DevParams& P, const DevPtrs& D, int p, int bi, int nbi)
{
    const DevPart& q = D.parts[p];
    int o[3];
    cover_origin(P, q, o);
    const int tot = P.side2[0] * P.side2[1] * P.side2[2];
    for (int t = bi * blockDim.x + threadIdx.x; t < tot; t += nbi * blockDim.x) {
        int x, y, z;
        if (!box_node(P, o, P.side2, t, x, y, z)) continue;
        uint8_t own = 0;
        for (int k = 0; k < P.np; ++k) {
            const DevPart& qk = D.parts[k];
            int Dk[3];
            int_offset(P, qk.gn, x, y, z, Dk);
            if (solid_test(qk.gn, Dk, qk.R2f, qk.rmarg, qk.R2)) {
                own = (uint8_t)(k + 1);
                break;
            }
        }
        D.mask_next[x + P.nx * (y + P.ny * z)] = own;
    }
}

// A kernel launched with programmatic stream serialization starts once every
// block of the kernel before it in the stream has called release_next_grid (or
// has ended), and may run its first part beside it; wait_for_prior_grid
// returns when that kernel has ended and its writes are visible.  Both do
// nothing in a kernel launched without the attribute.
__device__ __forceinline__ void release_next_grid() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

//
// cover_apply_block runs block bi of the nbi blocks of particle p; the last of
// the np * nbi blocks of the box (a ticket) finishes the step for all
// particles of the box.  smem holds block_rows_bytes<kCoverK>(blockDim.x)
// bytes.
// Bound by latency: few nodes, a chain of dependent loads.  In most steps no node
// of a block changes, and then it adds nothing up; the last block gives each
// particle a warp instead of taking one after the other with all its threads
// (alone: 11.1 -> 9.5 us with one sphere at 24^3, 29.1 -> 14.7 us with eight at
// 256^3).
template <class C>
__device__ __forceinline__ void cover_apply_block(const DevParams& P, const DevPtrs& D, int p, int bi, int nbi,
                                                  double* smem, bool& last)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    using S = typename C::pop_t;
    constexpr int K = kCoverK;
    const DevPart& q = D.parts[p];
    const size_t N = (size_t)P.N;
    int o[3];
    cover_origin(P, q, o);
    const int tot = P.side2[0] * P.side2[1] * P.side2[2];
    S* f = (S*)D.f_dst;
    F* psi = (F*)D.psi_dst;
    F* phi = (F*)D.phi_dst;
    F* u = (F*)D.u;
    const R rho0 = prm<R>(P).rho0;
    double acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.0;
    bool changed = false;
    for (int t = bi * blockDim.x + threadIdx.x; t < tot; t += nbi * blockDim.x) {
        int x, y, z;
        if (!box_node(P, o, P.side2, t, x, y, z)) continue;
        const int n = x + P.nx * (y + P.ny * z);
        const uint8_t ob = D.mask[n], nw = D.mask_next[n];
        int nb[19];
        neighbours(P, x, y, z, nb);
        // boundary flag for the next step (fluid node with a solid neighbour);
        // all mask loads first
        bool adj = false;
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const int m = nb[i] >= 0 ? nb[i] : n;
            adj = adj || (nb[i] >= 0 && D.mask_next[m]);
        }
        wait_for_prior_grid();   // k_scalars_particles reads the old flags and writes the fields
        D.bflag[n] = (!nw && adj) ? 1 : 0;
        if (ob == nw) continue;
        changed = true;
        if (ob == 0 && nw == p + 1) {
            // covered: the particle takes the momentum the node's populations
            // carry; psi, phi are removed
            R jr[3] = {0, 0, 0};
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                const R fi = (R)PopStore<S>::load_dev(f, (size_t)i * N + n, i, rho0);   // sum c f = sum c g
                if (cx(i) != 0) jr[0] = cx(i) > 0 ? add_x(jr[0], fi) : add_x(jr[0], -fi);
                if (cy(i) != 0) jr[1] = cy(i) > 0 ? add_x(jr[1], fi) : add_x(jr[1], -fi);
                if (cz(i) != 0) jr[2] = cz(i) > 0 ? add_x(jr[2], fi) : add_x(jr[2], -fi);
            }
            const double j[3] = {(double)jr[0], (double)jr[1], (double)jr[2]};
            int Dn[3];
            int_offset(P, q.gn, x, y, z, Dn);
            const double r[3] = {__dsub_rn((double)Dn[0], q.gn.frd[0]), __dsub_rn((double)Dn[1], q.gn.frd[1]),
                                 __dsub_rn((double)Dn[2], q.gn.frd[2])};
            acc[0] += j[0];
            acc[1] += j[1];
            acc[2] += j[2];
            acc[3] += cross_x(r[1], j[2], r[2], j[1]);
            acc[4] += cross_x(r[2], j[0], r[0], j[2]);
            acc[5] += cross_x(r[0], j[1], r[1], j[0]);
            acc[6] += (double)psi[n];
            acc[7] += (double)phi[n];
            acc[8] -= 1.0;
        } else if (ob == p + 1 && nw == 0) {
            // uncovered: equilibrium at the boundary velocity with the mean
            // density of neighbours fluid before and after; psi, phi = means
            R rb = 0, pb = 0, hb = 0;
            int cnt = 0;
            for (int i = 1; i < 19; ++i) {
                const int m = nb[i];
                if (m < 0 || D.mask[m] || D.mask_next[m]) continue;
                R rm = 0;   // rho - rho0 = sum g
#pragma unroll
                for (int k = 0; k < 19; ++k) rm = add_x(rm, (R)PopStore<S>::load_dev(f, (size_t)k * N + m, k, rho0));
                rb = add_x(rb, add_x(rho0, rm));
                pb = add_x(pb, (R)psi[m]);
                hb = add_x(hb, (R)phi[m]);
                ++cnt;
            }
            if (cnt == 0) {
                atomicOr(D.err, kErrOverlap);
                rb = rho0;
                pb = hb = 0;
            } else {
                rb = rb / (R)cnt;
                pb = pb / (R)cnt;
                hb = hb / (R)cnt;
            }
            int Dn[3];
            int_offset(P, q.gn, x, y, z, Dn);
            R r[3];
            link_offset_r<R>(q.gn, Dn, 0, r);
            const R U0 = PartR<R>::U(q, 0), U1 = PartR<R>::U(q, 1), U2 = PartR<R>::U(q, 2);
            const R W0 = PartR<R>::W(q, 0), W1 = PartR<R>::W(q, 1), W2 = PartR<R>::W(q, 2);
            const R ub[3] = {add_x(U0, cross_x(W1, r[2], W2, r[1])), add_x(U1, cross_x(W2, r[0], W0, r[2])),
                             add_x(U2, cross_x(W0, r[1], W1, r[0]))};
#pragma unroll
            for (int i = 0; i < 19; ++i)
                PopStore<S>::store_dev(f, (size_t)i * N + n, i, rho0, geq_i<R>(i, rb, rho0, ub[0], ub[1], ub[2]));
            u[n] = (F)ub[0];
            u[N + n] = (F)ub[1];
            u[2 * N + n] = (F)ub[2];
            psi[n] = (F)pb;
            phi[n] = (F)hb;
            const double j[3] = {(double)mul_x(rb, ub[0]), (double)mul_x(rb, ub[1]), (double)mul_x(rb, ub[2])};
            const double rd[3] = {(double)r[0], (double)r[1], (double)r[2]};
            acc[0] -= j[0];
            acc[1] -= j[1];
            acc[2] -= j[2];
            acc[3] -= cross_x(rd[1], j[2], rd[2], j[1]);
            acc[4] -= cross_x(rd[2], j[0], rd[0], j[2]);
            acc[5] -= cross_x(rd[0], j[1], rd[1], j[0]);
            acc[6] -= (double)psi[n];
            acc[7] -= (double)phi[n];
            acc[8] += 1.0;
        } else if (ob == p + 1) {
            atomicOr(D.err, kErrOverlap);   // passed straight into another sphere
        }
    }
    wait_for_prior_grid();   // threads without a node
    double* part = D.cover_part + ((size_t)p * kMaxPartBlocks + bi) * K;
    const int any = __syncthreads_or(changed);
    if (any) block_sum_rows<K>(acc, smem);
    // a block without changes stores one +0, its node count; one with changes
    // but as many nodes covered as uncovered stores -0 there
    if ((int)threadIdx.x < (any ? K - 1 : 0)) part[threadIdx.x] = smem[threadIdx.x];
    if (threadIdx.x == K - 1) part[K - 1] = !any ? 0.0 : smem[K - 1] == 0.0 ? -0.0 : smem[K - 1];
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = (atomicAdd(D.cover_ticket, 1u) == (unsigned)(nbi * P.np) - 1u);
    }
    __syncthreads();
    if (!last) return;
    // last block of the grid, one warp per particle: lane l adds the partials
    // of blocks l, l + 32, ..., the lanes' sums meet in a fixed tree; impulses
    // go to their particles, deficits into the uniform correction, particles
    // move
    __threadfence();
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int k = threadIdx.x >> 5; k < P.np; k += nw) {
        DevPart& dk = D.parts[k];
        double s[K];
#pragma unroll
        for (int c = 0; c < K; ++c) s[c] = 0.0;
        // nothing changed: one load a block and no FP64 instruction (64 cycles
        // each)
        bool nz = false;
        for (int b = lane; b < nbi; b += 32) {
            const double* cp = D.cover_part + ((size_t)k * kMaxPartBlocks + b) * K;
            const double d = __ldcg(cp + K - 1);
            if (__double_as_longlong(d) == 0) continue;
            nz = true;
#pragma unroll
            for (int c = 0; c < K - 1; ++c) s[c] += __ldcg(cp + c);
            s[K - 1] += d;
        }
        if (__any_sync(0xffffffffu, nz)) {
            for (int w = 16; w > 0; w >>= 1)
#pragma unroll
                for (int c = 0; c < K; ++c) s[c] += __shfl_xor_sync(0xffffffffu, s[c], w);
        }
        if (lane == 0) {
            // all loads first: a store after each load would wait for it
            const Geo gn = dk.gn;
            double X[3], m[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                X[a] = dk.Xn[a];
                m[a] = dk.mn[a];
            }
            const double wp = dk.wall_psi, wh = dk.wall_phi;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                dk.imp_f[a] = s[a];
                dk.imp_t[a] = s[3 + a];
                dk.X[a] = X[a];
                dk.m[a] = m[a];
                dk.mf[a] = (float)m[a];
            }
            dk.g = gn;
            smem[3 * k] = s[6] + wp;
            smem[3 * k + 1] = s[7] + wh;
            smem[3 * k + 2] = s[8];
        }
    }
    __syncthreads();
    if (threadIdx.x >= 2) return;
    // thread 0: psi, thread 1: phi
    double dsum = 0.0, dcnt = 0.0;
    for (int k = 0; k < P.np; ++k) {
        dsum += smem[3 * k + threadIdx.x];
        dcnt += smem[3 * k + 2];
    }
    const long long nf = *D.nfluid + (long long)dcnt;
    const double c = dsum / (double)nf;
    D.corr_next[threadIdx.x] = c;
    D.corr_f_next[threadIdx.x] = (float)c;
    __syncwarp(3u);
    if (threadIdx.x != 0) return;
    *D.nfluid = nf;
    *D.cover_ticket = 0u;
}

// ---------------------------------------------------------------------------
// covering kernels of the single box: grid (blocks per particle, particles)
// (the other particle kernels are in lbdp_particles.cuh, the bulk kernels in
// lbdp_zmarch.cuh)
// ---------------------------------------------------------------------------
template <class C>
__global__ void __launch_bounds__(kCoverThreads) k_cover_mark(DevParams P, DevPtrs D)
{
    cover_mark_block<C>(P, D, blockIdx.y, blockIdx.x, gridDim.x);
}

template <class C>
__global__ void __launch_bounds__(kCoverThreads) k_cover_apply(DevParams P, DevPtrs D)
{
    __shared__ double smem[block_rows_bytes<kCoverK>(kCoverThreads) / sizeof(double)];
    __shared__ bool last;
    cover_apply_block<C>(P, D, blockIdx.y, blockIdx.x, gridDim.x, smem, last);
}

// ---------------------------------------------------------------------------
// host <-> device field conversion and diagnostics
// ---------------------------------------------------------------------------

// Populations to equilibrium of (rho, u) from FP64 staging; fields from
// staging where given, else the current value plus any pending uniform
// correction.  Solid nodes are left untouched.
template <class C>
__global__ void k_set_fields(DevParams P, DevPtrs D, const double* rho_in, const double* u_in, const double* psi_in,
                             const double* phi_in)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    using S = typename C::pop_t;
    const size_t N = (size_t)P.N;
    const R rho0 = prm<R>(P).rho0;
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N; n += (size_t)gridDim.x * blockDim.x) {
        if (D.mask[n]) continue;
        F* psi = (F*)D.psi_dst;
        F* phi = (F*)D.phi_dst;
        F* u = (F*)D.u;
        S* f = (S*)D.f_dst;
        psi[n] = psi_in ? (F)psi_in[n] : (F)((double)psi[n] + D.corr[0]);
        phi[n] = phi_in ? (F)phi_in[n] : (F)((double)phi[n] + D.corr[1]);
        if (u_in) {
            u[n] = (F)u_in[n];
            u[N + n] = (F)u_in[N + n];
            u[2 * N + n] = (F)u_in[2 * N + n];
        }
        double rho;
        if (rho_in) {
            rho = rho_in[n];
        } else {
            R s = 0;   // rho - rho0
#pragma unroll
            for (int i = 0; i < 19; ++i) s += (R)PopStore<S>::load_dev(f, (size_t)i * N + n, i, rho0);
            rho = P.rho0 + (double)s;
        }
        const double ux = (double)u[n], uy = (double)u[N + n], uz = (double)u[2 * N + n];
#pragma unroll
        for (int i = 0; i < 19; ++i)
            PopStore<S>::store_dev(f, (size_t)i * N + n, i, rho0, (R)geq_i<double>(i, rho, P.rho0, ux, uy, uz));
    }
}

// Chemical potentials of the current fields (for the readout only).
template <class C>
__global__ void k_mu_now(DevParams P, DevPtrs D)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    const size_t N = (size_t)P.N;
    const F* psi = (const F*)D.psi_src;
    const F* phi = (const F*)D.phi_src;
    const R dph = corr_r<R>(D, 1);
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N; n += (size_t)gridDim.x * blockDim.x) {
        R mps = 0, mph = 0;
        if (!D.mask[n]) {
            const int x = (int)(n % P.nx), y = (int)((n / P.nx) % P.ny), z = (int)(n / ((size_t)P.nx * P.ny));
            int nb[19];
            neighbours(P, x, y, z, nb);
            R d[19], pt[kPtFields];
            const R ps = gather_psi<R, F>(P, D, psi, x, y, z, nb, d);
            mu_pressure<R>(prm<R>(P), ps, psi_sums<R>(d), (R)phi[n] + dph, false, mps, mph, pt);
        }
        ((F*)D.mupsi)[n] = (F)mps;
        ((F*)D.muphi)[n] = (F)mph;
    }
}

// Fields to FP64 staging (zeros at solid nodes).  which: bit0 rho, bit1 u,
// bit2 psi, bit3 phi, bit4 mu (mu_psi to out_rho, mu_phi to out_psi).
template <class C>
__global__ void k_get_fields(DevParams P, DevPtrs D, int which, double* out_rho, double* out_u, double* out_psi,
                             double* out_phi)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    using S = typename C::pop_t;
    const size_t N = (size_t)P.N;
    const R rho0 = prm<R>(P).rho0;
    const S* f = (const S*)D.f_src;
    const F* psi = (const F*)D.psi_src;
    const F* phi = (const F*)D.phi_src;
    const F* u = (const F*)D.u;
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N; n += (size_t)gridDim.x * blockDim.x) {
        const bool solid = D.mask[n] != 0;
        if (which & 1) {
            R s = 0;   // rho - rho0
            if (!solid)
#pragma unroll
                for (int i = 0; i < 19; ++i) s += (R)PopStore<S>::load_dev(f, (size_t)i * N + n, i, rho0);
            out_rho[n] = solid ? 0.0 : P.rho0 + (double)s;
        }
        if (which & 2)
            for (int a = 0; a < 3; ++a) out_u[a * N + n] = solid ? 0.0 : (double)u[a * N + n];
        if (which & 4) out_psi[n] = solid ? 0.0 : (double)psi[n] + D.corr[0];
        if (which & 8) out_phi[n] = solid ? 0.0 : (double)phi[n] + D.corr[1];
        if (which & 16) {
            out_rho[n] = solid ? 0.0 : (double)((const F*)D.mupsi)[n];
            out_psi[n] = solid ? 0.0 : (double)((const F*)D.muphi)[n];
        }
    }
}

template <class C>
__global__ void k_get_pops(DevParams P, DevPtrs D, double* out, int i)
{
    using R = typename C::real;
    using S = typename C::pop_t;
    const size_t N = (size_t)P.N;
    const S* f = (const S*)D.f_src;
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N; n += (size_t)gridDim.x * blockDim.x) {
        double v = 0.0;
        if (!D.mask[n]) v = (double)PopStore<S>::load(f, (size_t)i * N + n, i, prm<R>(P).rho0);
        out[n] = v;
    }
}

// Conservation sums, pass 1: per-block FP64 partials of rho, psi, phi over
// fluid nodes.
template <class C>
__global__ void __launch_bounds__(256) k_sums(DevParams P, DevPtrs D, double* part)
{
    using R = typename C::real;
    using F = typename C::fld_t;
    using S = typename C::pop_t;
    __shared__ double smem[32 * 3];
    const size_t N = (size_t)P.N;
    const R rho0 = prm<R>(P).rho0;
    const S* f = (const S*)D.f_src;
    const F* psi = (const F*)D.psi_src;
    const F* phi = (const F*)D.phi_src;
    double v[3] = {0.0, 0.0, 0.0};
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N; n += (size_t)gridDim.x * blockDim.x) {
        if (D.mask[n]) continue;
        double s = 0.0;
#pragma unroll
        for (int i = 0; i < 19; ++i) s += (double)PopStore<S>::load(f, (size_t)i * N + n, i, rho0);
        v[0] += s;
        v[1] += (double)psi[n] + D.corr[0];
        v[2] += (double)phi[n] + D.corr[1];
    }
    block_sum<3>(v, smem);
    if (threadIdx.x == 0)
        for (int k = 0; k < 3; ++k) part[blockIdx.x * 3 + k] = v[k];
}

// pass 2: one thread sums the partials in block order
static __global__ void k_sums_final(const double* part, int nblocks, double* out)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double s[3] = {0.0, 0.0, 0.0};
    for (int b = 0; b < nblocks; ++b)
        for (int k = 0; k < 3; ++k) s[k] += part[b * 3 + k];
    for (int k = 0; k < 3; ++k) out[k] = s[k];
}

// New sphere q as particle p: its record, and the fluid nodes strictly inside it
// claimed in both mask buffers and taken off the fluid node count.
static __global__ void k_claim(DevParams P, uint8_t* m0, uint8_t* m1, DevPart* parts, int p,
                               const __grid_constant__ DevPart q, long long* nfluid)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) parts[p] = q;
    const size_t N = (size_t)P.N;
    int claimed = 0;
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N; n += (size_t)gridDim.x * blockDim.x) {
        if (m0[n]) continue;
        const int x = (int)(n % P.nx), y = (int)((n / P.nx) % P.ny), z = (int)(n / ((size_t)P.nx * P.ny));
        if (inside_sphere(P, q, x, y, z)) {
            m0[n] = (uint8_t)(p + 1);
            m1[n] = (uint8_t)(p + 1);
            ++claimed;
        }
    }
    if (claimed) atomicAdd((unsigned long long*)nfluid, (unsigned long long)(-(long long)claimed));
}

// Staging of a new box: rho0 at every node, and the fluid node count.
static __global__ void k_rest(double* rho, double rho0, long long N, long long* nfluid)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *nfluid = N;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N; n += (long long)gridDim.x * blockDim.x)
        rho[n] = rho0;
}

// Boundary flags of every node from a mask: fluid node with a solid neighbour.
static __global__ void k_bflag_all(DevParams P, const uint8_t* mask, uint8_t* bflag)
{
    const size_t N = (size_t)P.N;
    for (size_t n = blockIdx.x * (size_t)blockDim.x + threadIdx.x; n < N; n += (size_t)gridDim.x * blockDim.x) {
        const int x = (int)(n % P.nx), y = (int)((n / P.nx) % P.ny), z = (int)(n / ((size_t)P.nx * P.ny));
        bool adj = false;
        if (!mask[n]) {
            int nb[19];
            neighbours(P, x, y, z, nb);
            for (int i = 1; i < 19; ++i) adj = adj || (nb[i] >= 0 && mask[nb[i]]);
        }
        bflag[n] = adj ? 1 : 0;
    }
}

}  // namespace lbdp
