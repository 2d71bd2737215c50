// walk_ordered.cuh -- the tree walk of runs with block time steps: one warp per
// group from the root to the end, in one order of operations.
//
// The steps of a block step are long (dt itself on level 0), so the FP32
// rounding of the accelerations reaches the FP64 positions through the FP32
// velocities: Plummer spheres of 2,000 to 100,000 particles at dt = 1/8, walked
// in this order and cooperatively, part by 5e-10 of the positions (2-norm) in
// one call and by 1.5e-9 in two, and a level decision that falls the other way
// by up to 4e-7.  A run followed with block steps is therefore walked, from its
// first forces on, in an order that depends on the group alone -- not on how
// many groups are active, nor on quotas and parts: the list is filled round by
// round (accepted nodes, then the particles of opened leaves, 32 at a time) and
// flushed when the next append would not fit, and an interaction is
// (m / r) / r / r.
//
// Bound by the longest group's own chain with the few active groups of most
// ticks (one warp, 40 to 80 ns per list entry): a Hernquist sphere of 65,539
// particles takes 6.2 ms per call (8 ticks), 3.4 with the cooperative walk.
#pragma once

#include "walk_impl.cuh"

namespace nb {

template <int IPL, bool PHI, bool COMP, bool SAFE, bool QUAD>
__global__ void __maxnreg__((walk_regs<IPL, QUAD || COMP>())) ordered_walk_kernel(WalkArgs a, int geometric) {
    extern __shared__ __align__(16) unsigned char walk_smem[];
    const int D = a.list_depth, S = a.stack_depth;
    const int DQ = QUAD ? walk_quad_depth(D) : 0;
    const unsigned lane = lane_id(), w = threadIdx.x >> 5;
    const size_t per_warp = walk_smem_per_warp(D, S, QUAD);
    float4 *LA = reinterpret_cast<float4 *>(walk_smem + w * per_warp);
    float4 *LQ = LA + D;
    uint32_t *stk = reinterpret_cast<uint32_t *>(walk_smem + w * per_warp + (size_t)D * sizeof(float4) +
                                                 (size_t)DQ * 40);
    int *scr = reinterpret_cast<int *>(stk + S);
    DevState *ds = a.ds;
    const int ng = a.nactive ? *a.nactive : ds->ngroups;
    const int nnodes = ds->nnodes;
    const int npart = (int)a.n;
    const unsigned lt = lanemask_lt();
    int max_sp = 0;
    unsigned long long warp_entries = 0, warp_inter = 0, warp_quad = 0;
    bool overflow = false, bad = false;

    for (;;) {
        int qi = 0;
        if (lane == 0) qi = atomicAdd(&ds->queue.head, 1);
        qi = __shfl_sync(NB_FULL, qi, 0);
        if (qi >= ng) break;
        const int g = a.order ? a.order[qi] : qi;
        const int first = a.grp_first[g], cnt = a.grp_count[g];
        const float4 sph = a.grp_sphere[g];
        const float alpha = geometric ? 0.0f : a.grp_alpha[g];
        const int sys = a.grp_sys[g];
        const float eps2 = a.sys_eps2[sys];

        if (cnt > 32 * IPL) bad = true;  // larger than the group size allows
        const Tiling tile = lane_tiling<IPL>(cnt);
        ISlots<IPL> I;
        load_slots<IPL>(tile, a.pos4, first, cnt, sph, I);

        if (lane == 0) stk[0] = (uint32_t)a.sys_root[sys] << 3;  // one node: the system's root
        int sp = 1, nl = 0, nq = 0;
        int entries = 0, qentries = 0;  // at most particles + nodes of the system
        auto flush = [&]() {
            __syncwarp();
            flush_runs<0, 0, IPL, PHI, COMP, SAFE, false, 1, true>(tile, LA, nl, eps2, I);
            entries += nl;
            nl = 0;
            __syncwarp();
        };
        auto flush_nodes = [&]() {
            __syncwarp();
            flush_runs<0, 0, IPL, PHI, COMP, SAFE, true>(tile, LQ, nq, eps2, I);
            qentries += nq;
            nq = 0;
            __syncwarp();
        };
        __syncwarp();
        while (sp > 0) {
            // ---- pop and MAC as in walk_kernel
            const int take = sp < 4 ? sp : 4;
            const int rr = (int)(lane >> 3), jj = (int)(lane & 7);
            uint32_t e = 0;
            if (rr < take) e = stk[sp - 1 - rr];
            const int node = (int)(e >> 3) + jj;
            const bool slot = rr < take && jj <= (int)(e & 7u);
            const bool in_range = (unsigned)node < (unsigned)nnodes;
            if (slot && !in_range) bad = true;
            const bool has = slot && in_range;
            sp -= take;
            __syncwarp();
            const int nd = has ? node : 0;
            const float4 A = __ldg(&a.nodeA[nd]), B = __ldg(&a.nodeB[nd]);
            const float dx = A.x - sph.x, dy = A.y - sph.y, dz = A.z - sph.z;
            const float d = sqrt_fast(fmaf(dz, dz, fmaf(dy, dy, dx * dx))) - sph.w;
            bool accept;
            if (geometric) {
                accept = has && d > B.x && B.x <= a.theta * d;
            } else {
                const float d2 = d * d;
                accept = has && d > B.x && B.y <= alpha * (d2 * d2);
            }
            const int link = __float_as_int(B.z), meta = __float_as_int(B.w);
            const bool leaf = (meta & 1) != 0;
            const int mcount = meta >> 1;
            const bool open_leaf = has && !accept && leaf;
            const bool bad_link = has && !accept && !leaf &&
                                  (link <= node || (unsigned)(mcount - 1) > 7u || link + mcount > nnodes);
            if (bad_link) bad = true;
            const bool open_node = has && !accept && !leaf && !bad_link;

            // ---- push the child ranges of opened internal nodes
            const unsigned om = __ballot_sync(NB_FULL, open_node);
            if (open_node) {
                const int pos = sp + __popc(om & lt);
                if (pos < S) stk[pos] = ((uint32_t)link << 3) | (uint32_t)(mcount - 1);
            }
            sp += __popc(om);
            if (sp > S) {
                overflow = true;
                sp = S;
            }
            if (sp > max_sp) max_sp = sp;

            // ---- accepted nodes join the list (with quadrupoles: the node list)
            const unsigned am = __ballot_sync(NB_FULL, accept);
            const int na = __popc(am);
            if constexpr (QUAD) {
                if (nq + na > DQ) flush_nodes();
                if (accept)
                    quad_put(LQ, nq + __popc(am & lt), A, __ldg(&a.nodeQ[2 * node]),
                             __ldg(&a.nodeQ[2 * node + 1]));
                nq += na;
            } else {
                if (nl + na > D) flush();
                if (accept) list_put(LA, nl + __popc(am & lt), A);
                nl += na;
            }

            // ---- particles of opened leaves join the list, 32 at a time
            const bool leaf_ok = open_leaf && (unsigned)link < (unsigned)npart &&
                                 (unsigned)(mcount - 1) < (unsigned)(npart - link);
            if (open_leaf && !leaf_ok) bad = true;
            const unsigned lm = __ballot_sync(NB_FULL, leaf_ok);
            if (lm) {
                const int nlf = __popc(lm);
                if (leaf_ok) scr[__popc(lm & lt)] = (int)lane;
                __syncwarp();
                const int src = (int)lane < nlf ? scr[lane] : 0;
                const int lf = __shfl_sync(NB_FULL, link, src);
                const int lcs = __shfl_sync(NB_FULL, mcount, src);
                const int lc = (int)lane < nlf ? lcs : 0;
                const int lincl = warp_incl_scan(lc);
                const int lexcl = lincl - lc;
                const int total = __shfl_sync(NB_FULL, lincl, 31);
                for (int base = 0; base < total; base += 32) {
                    const int c = min(32, total - base);
                    if (nl + c > D) flush();
                    // the owner of slot base + lane is the last leaf starting at
                    // or before it (counts >= 1, starts increasing)
                    const bool starts = lc > 0 && lexcl >= base && lexcl < base + 32;
                    const unsigned smap = __reduce_or_sync(NB_FULL, starts ? 1u << (lexcl - base) : 0u);
                    const int before = __popc(__ballot_sync(NB_FULL, lc > 0 && lexcl < base));
                    const int k = before + __popc(smap & (0xffffffffu >> (31 - lane))) - 1;
                    const int of = __shfl_sync(NB_FULL, lf, k & 31);
                    const int oex = __shfl_sync(NB_FULL, lexcl, k & 31);
                    if ((int)lane < c) list_put(LA, nl + (int)lane, __ldg(&a.pos4[of + base + (int)lane - oex]));
                    nl += c;
                }
            }
            __syncwarp();
        }
        if (nl > 0) flush();
        if constexpr (QUAD) {
            if (nq > 0) flush_nodes();
        }
        __syncwarp();

        const float self = SAFE ? 0.0f : rsqrt_fast(eps2);
        group_sums<IPL, PHI, COMP>(tile, cnt, I, [&](int idx, const float (&r)[4], float mi) {
            store_force<PHI>(a, first + idx, r, mi, a.G, self);
        });
        entries += qentries;
        if (lane == 0 && a.grp_cost) a.grp_cost[g] = entries;
        warp_entries += (unsigned long long)entries;
        warp_inter += (unsigned long long)entries * (unsigned long long)cnt;
        warp_quad += (unsigned long long)qentries * (unsigned long long)cnt;
    }
    if (lane == 0) {
        atomicMax(&ds->max_stack, max_sp);
        if (warp_entries) {
            atomicAdd(&ds->list_entries, warp_entries);
            atomicAdd(&ds->interactions, warp_inter);
        }
        if (QUAD && warp_quad) atomicAdd(&ds->quad_entries, warp_quad);
        if (overflow) atomicOr(&ds->status, kStatusStackOverflow);
    }
    if (bad) atomicOr(&ds->status, kStatusBadTree);
}

template <int IPL, bool QUAD>
cudaError_t launch_ordered_ipl(cudaStream_t s, const WalkArgs &a, const WalkShape &sh, int nsm) {
    const int threads = 32 * sh.warps_per_block;
    const size_t smem =
        (size_t)sh.warps_per_block * walk_smem_per_warp(a.list_depth, a.stack_depth, QUAD);
    void (*k)(WalkArgs, int);
    if (sh.potential) {
        if (sh.compensated) k = sh.safe ? ordered_walk_kernel<IPL, true, true, true, QUAD> : ordered_walk_kernel<IPL, true, true, false, QUAD>;
        else k = sh.safe ? ordered_walk_kernel<IPL, true, false, true, QUAD> : ordered_walk_kernel<IPL, true, false, false, QUAD>;
    } else {
        if (sh.compensated) k = sh.safe ? ordered_walk_kernel<IPL, false, true, true, QUAD> : ordered_walk_kernel<IPL, false, true, false, QUAD>;
        else k = sh.safe ? ordered_walk_kernel<IPL, false, false, true, QUAD> : ordered_walk_kernel<IPL, false, false, false, QUAD>;
    }
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem);
    if (err != cudaSuccess) return err;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    if (sh.warps_launched) *sh.warps_launched = nsm * per_sm * sh.warps_per_block;
    k<<<nsm * per_sm, threads, smem, s>>>(a, sh.geometric ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace nb
