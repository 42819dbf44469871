// lbdp_ops.cuh -- launch wrappers of one precision configuration; included by
// exactly one lbdp_prec_*.cu translation unit each, so the four precision
// modes compile in parallel.
#pragma once

#include "lbdp_batch_kernels.cuh"
#include "lbdp_internal.h"
#include "lbdp_kernels.cuh"
#include "lbdp_zmarch.cuh"

namespace lbdp {

// Launch of a side-stream kernel with the side streams' priority as a launch
// attribute, so that it keeps the priority inside captured graphs too.
template <class... A>
inline void side_launch_with(cudaLaunchAttribute* at, int nat, cudaStream_t st, void (*k)(A...), dim3 grid,
                             int threads, const SideStream* side, A... args)
{
    at[0].id = cudaLaunchAttributePriority;
    at[0].val.priority = side->prio;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = nat;
    cudaLaunchKernelEx(&cfg, k, args...);
}

template <class... A>
inline void side_launch_on(cudaStream_t st, void (*k)(A...), dim3 grid, int threads, const SideStream* side,
                           A... args)
{
    cudaLaunchAttribute at[1];
    side_launch_with(at, 1, st, k, grid, threads, side, args...);
}

template <class... A>
inline void side_launch(void (*k)(A...), dim3 grid, int threads, const SideStream* side, A... args)
{
    side_launch_on(side->s, k, grid, threads, side, args...);
}

// The same for a kernel that may start beside the end of the kernel before it
// in the stream, which calls release_next_grid; it calls wait_for_prior_grid.
template <class... A>
inline void side_launch_early(void (*k)(A...), dim3 grid, int threads, const SideStream* side, A... args)
{
    cudaLaunchAttribute at[2];
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    side_launch_with(at, 2, side->s, k, grid, threads, side, args...);
}

// Blocks of kz_scalars (at most one on each SM) up to which k_cover_apply is
// launched early.
constexpr unsigned kEarlyCoverBlocks = kSMs;

template <class C>
struct Ops {
    using R = typename C::real;
    using F = typename C::fld_t;

    static constexpr size_t kFusedSmem = fused_smem_bytes<C>();
    static constexpr size_t kZScalSmem = scal_smem_bytes<C>();

    // Opt the kernels that use more than 48 KiB of shared memory in, once per
    // device.
    static cudaError_t prepare()
    {
        static bool done[64] = {false};
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
        e = cudaFuncSetAttribute(kz_fused<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFusedSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kz_scalars<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kZScalSmem);
        if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
        return e;
    }

    static dim3 pt_grid(const DevParams& P) { return dim3(pt_part_blocks(P, sizeof(R) == 8), P.np); }

    // One time step.  With particles and side streams: the particle kernels
    // (pressure tensor and force next to the particles, link sums and the
    // particle update with the new mask on a stream of their own, then the
    // collide-stream of the nodes next to particles) run beside kz_fused; the
    // transport of the bulk waits for the boundary collide-stream (it reads u
    // there), and the boundary transport and covering wait for kz_fused and
    // run beside it.
    // ev (optional, 6 events): the same kernels in sequence, an event before
    // the first and after each kernel class.
    static cudaError_t launch_step(const DevParams& P, const DevPtrs& D, const RowGrid& g, cudaStream_t s,
                                   cudaEvent_t* ev, const SideStream* side)
    {
        cudaError_t e = prepare();
        if (e != cudaSuccess) return e;
        const dim3 pg1(P.nb1, P.np), pg2(P.nb2, P.np), pgt = pt_grid(P);
        if (P.np > 0 && side && !ev) {
            cudaEventRecord(side->fork, s);
            cudaStreamWaitEvent(side->s2, side->fork, 0);
            side_launch_on(side->s2, k_links<C>, pg1, kPartThreads, side, P, D);
            cudaEventRecord(side->links_done, side->s2);
            side_launch_on(side->s2, k_cover_mark<C>, pg2, kCoverThreads, side, P, D);
            cudaEventRecord(side->mark_done, side->s2);
            cudaStreamWaitEvent(side->s, side->fork, 0);
            side_launch(k_pt_part<C>, pgt, kPartThreads, side, P, D);
            side_launch(k_f_part<C>, pg1, kPartThreads, side, P, D);
            cudaStreamWaitEvent(side->s, side->links_done, 0);
            side_launch(k_collide_particles<C>, pg1, kPartThreads, side, P, D);
            cudaEventRecord(side->bnd_done, side->s);
            kz_fused<C><<<g.zgrid, kZThreads, kFusedSmem, s>>>(P, D);
            cudaEventRecord(side->collide_done, s);
            // covering touches only nodes next to particles, whose fields the
            // side-stream kernels wrote, and leaves the next step's uniform
            // correction in the other buffer: it runs beside the transport.
            // Where the transport leaves room on every SM it starts beside
            // k_scalars_particles (24^3 FP32: 56.1 -> 51.8 us a step); its
            // waiting blocks would hold up a transport that fills the chip
            // (96^3 FP64: 1351 -> 1417 us)
            const bool early = g.zgrid_s.x * g.zgrid_s.y * g.zgrid_s.z <= kEarlyCoverBlocks;
            if (early) cudaStreamWaitEvent(side->s, side->mark_done, 0);
            cudaStreamWaitEvent(side->s, side->collide_done, 0);
            side_launch(k_scalars_particles<C>, pg1, kPartThreads, side, P, D);
            if (early) {
                side_launch_early(k_cover_apply<C>, pg2, kCoverThreads, side, P, D);
            } else {
                cudaStreamWaitEvent(side->s, side->mark_done, 0);
                side_launch(k_cover_apply<C>, pg2, kCoverThreads, side, P, D);
            }
            cudaEventRecord(side->scal_done, side->s);
            cudaStreamWaitEvent(s, side->bnd_done, 0);
            kz_scalars<C><<<g.zgrid_s, kZThreads, kZScalSmem, s>>>(P, D);
            cudaStreamWaitEvent(s, side->scal_done, 0);   // the step ends with the side stream
            return cudaGetLastError();
        }
        if (ev) cudaEventRecord(ev[0], s);
        if (P.np > 0) {
            k_pt_part<C><<<pgt, kPartThreads, 0, s>>>(P, D);
            k_f_part<C><<<pg1, kPartThreads, 0, s>>>(P, D);
            k_links<C><<<pg1, kPartThreads, 0, s>>>(P, D);
            k_collide_particles<C><<<pg1, kPartThreads, 0, s>>>(P, D);
        }
        if (ev) cudaEventRecord(ev[1], s);
        kz_fused<C><<<g.zgrid, kZThreads, kFusedSmem, s>>>(P, D);
        if (ev) cudaEventRecord(ev[2], s);
        kz_scalars<C><<<g.zgrid_s, kZThreads, kZScalSmem, s>>>(P, D);
        if (ev) cudaEventRecord(ev[3], s);
        if (P.np > 0) k_scalars_particles<C><<<pg1, kPartThreads, 0, s>>>(P, D);
        if (ev) cudaEventRecord(ev[4], s);
        if (P.np > 0) {
            k_cover_mark<C><<<pg2, kCoverThreads, 0, s>>>(P, D);
            k_cover_apply<C><<<pg2, kCoverThreads, 0, s>>>(P, D);
        }
        if (ev) cudaEventRecord(ev[5], s);
        return cudaGetLastError();
    }

    static cudaError_t step(const DevParams& P, const DevPtrs& D, const RowGrid& g, cudaStream_t s,
                            const SideStream* side)
    {
        return launch_step(P, D, g, s, nullptr, side);
    }

    // sequential order with events around the kernel classes (the per-kernel
    // split; no overlap, so each class is timed alone)
    static cudaError_t step_events(const DevParams& P, const DevPtrs& D, const RowGrid& g, cudaStream_t s,
                                   cudaEvent_t* ev)
    {
        return launch_step(P, D, g, s, ev, nullptr);
    }

    static cudaError_t bulk(int which, const DevParams& P, const DevPtrs& D, dim3 grid, cudaStream_t s)
    {
        cudaError_t e = prepare();
        if (e != cudaSuccess) return e;
        if (which == 0)
            kz_fused<C><<<grid, kZThreads, kFusedSmem, s>>>(P, D);
        else
            kz_scalars<C><<<grid, kZThreads, kZScalSmem, s>>>(P, D);
        return cudaGetLastError();
    }

    static int grid1d(const DevParams& P)
    {
        long long b = (P.N + 255) / 256;
        return (int)(b < kSMs * 16 ? b : kSMs * 16);
    }

    static cudaError_t set_fields(const DevParams& P, const DevPtrs& D, cudaStream_t s, const double* rho,
                                  const double* u, const double* psi, const double* phi)
    {
        k_set_fields<C><<<grid1d(P), 256, 0, s>>>(P, D, rho, u, psi, phi);
        return cudaGetLastError();
    }

    static cudaError_t get_fields(const DevParams& P, const DevPtrs& D, cudaStream_t s, int which, double* a,
                                  double* u, double* b, double* c)
    {
        if (which & 16) k_mu_now<C><<<grid1d(P), 256, 0, s>>>(P, D);
        k_get_fields<C><<<grid1d(P), 256, 0, s>>>(P, D, which, a, u, b, c);
        return cudaGetLastError();
    }

    static cudaError_t get_pop(const DevParams& P, const DevPtrs& D, cudaStream_t s, double* out, int i)
    {
        k_get_pops<C><<<grid1d(P), 256, 0, s>>>(P, D, out, i);
        return cudaGetLastError();
    }

    static cudaError_t sums(const DevParams& P, const DevPtrs& D, cudaStream_t s, double* part, int nblocks,
                            double* out)
    {
        k_sums<C><<<nblocks, 256, 0, s>>>(P, D, part);
        k_sums_final<<<1, 32, 0, s>>>(part, nblocks, out);
        return cudaGetLastError();
    }

    static PrecOps table()
    {
        PrecOps t;
        t.pop_bytes = (int)sizeof(typename C::pop_t);
        t.fld_bytes = (int)sizeof(typename C::fld_t);
        t.prepare = &prepare;
        t.step = &step;
        t.step_events = &step_events;
        t.bulk = &bulk;
        t.set_fields = &set_fields;
        t.get_fields = &get_fields;
        t.get_pop = &get_pop;
        t.sums = &sums;
        return t;
    }
};

// Launchers of the batched kernels of one precision configuration.
template <class C>
struct BOps {
    using F = typename C::fld_t;
    using KFn = void (*)(BoxLaunch);

    static KFn fn(int nc, int cfg)
    {
        static_assert(kNumBatchCfgs == 3, "configuration table");
        if (nc == 0) {
            switch (cfg) {
                case 0: return kbz_fused<C, kZChunks[0]>;
                case 1: return kbz_fused<C, kZChunks[1]>;
                default: return kbz_fused<C, kZChunks[2]>;
            }
        }
        switch (cfg) {
            case 0: return kbz_scalars<C, kZChunks[0]>;
            case 1: return kbz_scalars<C, kZChunks[1]>;
            default: return kbz_scalars<C, kZChunks[2]>;
        }
    }

    static size_t smem(int nc) { return nc == 0 ? fused_smem_bytes<C>() : scal_smem_bytes<C>(); }

    static cudaError_t prepare()
    {
        static bool done[64] = {false};
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
        for (int nc = 0; nc < kNumBatchClasses && e == cudaSuccess; ++nc)
            for (int k = 0; k < kNumBatchCfgs && e == cudaSuccess; ++k)
                e = cudaFuncSetAttribute((const void*)fn(nc, k), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem(nc));
        if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
        return e;
    }

    static cudaError_t node(int nc, int cfg, const LaunchPlan* L, cudaStream_t s)
    {
        if (nc < 0 || nc >= kNumBatchClasses || cfg < 0 || cfg >= kNumBatchCfgs) return cudaErrorInvalidValue;
        void* args[] = {(void*)&L->L};
        return cudaLaunchKernel((const void*)fn(nc, cfg), L->zgrid[cfg], dim3(kZThreads), args, smem(nc), s);
    }

    // The single-box step over each launch's boxes, in the single-box order:
    // the particle kernels on the side stream beside the fused bulk kernel,
    // the bulk transport after the boundary collide-stream, the boundary
    // transport and covering beside it.
    static cudaError_t step(const int cfg[kNumBatchClasses], LaunchPlan* Ls, int nl, int par, long long* left,
                            int nbox, cudaStream_t s, const SideStream* side)
    {
        cudaError_t e = prepare();
        if (e != cudaSuccess) return e;
        for (int l = 0; l < nl; ++l) {
            LaunchPlan* L = Ls + l;
            L->L.par = par;   // copied into each launch's parameters at the call
            if (side) {
                // the single-box stream order: link sums and the new mask on
                // s2 beside the force and boundary collide on s
                cudaEventRecord(side->fork, s);
                cudaStreamWaitEvent(side->s2, side->fork, 0);
                side_launch_on(side->s2, kb_links<C>, L->link, kPartThreads, side, L->L);
                cudaEventRecord(side->links_done, side->s2);
                side_launch_on(side->s2, kb_cover_mark<C>, L->cover, kCoverThreads, side, L->L);
                cudaEventRecord(side->mark_done, side->s2);
                cudaStreamWaitEvent(side->s, side->fork, 0);
                side_launch(kb_pt_part<C>, L->ptg, kPartThreads, side, L->L);
                side_launch(kb_f_part<C>, L->link, kPartThreads, side, L->L);
                cudaStreamWaitEvent(side->s, side->links_done, 0);
                side_launch(kb_collide_particles<C>, L->link, kPartThreads, side, L->L);
                cudaEventRecord(side->bnd_done, side->s);
                if ((e = node(0, cfg[0], L, s)) != cudaSuccess) return e;
                cudaEventRecord(side->collide_done, s);
                cudaStreamWaitEvent(side->s, side->collide_done, 0);
                side_launch(kb_scalars_particles<C>, L->link, kPartThreads, side, L->L);
                cudaStreamWaitEvent(side->s, side->mark_done, 0);
                side_launch(kb_cover_apply<C>, L->cover, kCoverThreads, side, L->L);
                cudaEventRecord(side->scal_done, side->s);
                cudaStreamWaitEvent(s, side->bnd_done, 0);
                if ((e = node(1, cfg[1], L, s)) != cudaSuccess) return e;
                cudaStreamWaitEvent(s, side->scal_done, 0);
            } else {
                kb_pt_part<C><<<L->ptg, kPartThreads, 0, s>>>(L->L);
                kb_f_part<C><<<L->link, kPartThreads, 0, s>>>(L->L);
                kb_links<C><<<L->link, kPartThreads, 0, s>>>(L->L);
                kb_collide_particles<C><<<L->link, kPartThreads, 0, s>>>(L->L);
                if ((e = node(0, cfg[0], L, s)) != cudaSuccess) return e;
                if ((e = node(1, cfg[1], L, s)) != cudaSuccess) return e;
                kb_scalars_particles<C><<<L->link, kPartThreads, 0, s>>>(L->L);
                kb_cover_mark<C><<<L->cover, kCoverThreads, 0, s>>>(L->L);
                kb_cover_apply<C><<<L->cover, kCoverThreads, 0, s>>>(L->L);
            }
        }
        kb_advance<<<(nbox + 255) / 256, 256, 0, s>>>(left, nbox);
        return cudaGetLastError();
    }

    static BatchOps table()
    {
        BatchOps t;
        t.prepare = &prepare;
        t.node = &node;
        t.step = &step;
        return t;
    }
};

}  // namespace lbdp
