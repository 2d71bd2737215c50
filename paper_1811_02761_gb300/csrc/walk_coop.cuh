// walk_coop.cuh -- the tree walk with a CTA (or several) per i-group.
//
// One warp per group (walk_impl.cuh) is the efficient shape when there are
// many more groups than resident warps.  With fewer, most of the chip idles
// while each group is a serial chain of one warp, and a group whose list is
// far longer than the others' (its smallest |a_old| is nearly zero, so Eq. 2
// opens almost every node) is such a chain in any launch.  Here kCoopWarps
// warps of a CTA walk one group together:
//   * one stack in shared memory: each round the warps take the top
//     4 * kCoopWarps child ranges (one warp as in the one-warp walk), and the
//     pushes and list entries of all warps are placed by a scan of the warps'
//     counts, so every order is fixed;
//   * one interaction list, filled by all warps and flushed by all warps: lane
//     split u of warp w takes the entry pairs w s + u, + kCoopWarps s, ...;
//   * when there are few groups, P CTAs take one group: each expands the tree
//     from the top down to nodes of at most 1 / (kCoopFine P) of the system's
//     particles (a few rounds, whose list entries only part 0 keeps) and
//     walks every P-th of the child ranges found; the CTA that finishes last
//     adds the P partial sums in part order.
// It runs in two stages.  The first takes every group (where coop_walk, api.cu,
// says so), or the groups the one-warp walk cut at its quota; a part whose own
// list passes a.cut_quota entries is cut again, its open ranges recorded.  The
// second stage walks those records, again with P CTAs each, to the end: however
// uneven the groups are, no CTA works much longer than the others.
// The MAC is evaluated exactly as in the one-warp walk, so the list of every
// group holds the same entries; only the order of the sums differs, and it
// depends on the counts of groups and cuts alone, never on timing: which
// record or slot a part gets is up to the atomics, the order in which its
// sums are added is not.  No CTA waits for another.
//
// Bound by latency (rounds of two barriers and two loads from L2 each), and
// by the FP32 pipe once every SM has its three CTAs.  Walk alone, one warp per
// group / this: Plummer N = 4096 (107 groups) 0.192 / 0.039 ms, galaxy 100003
// (2253) 0.252 / 0.201, Hernquist 30011 at delta_acc = 2^-20 2.0 / 0.71, and
// Plummer 262147 without |a_old| (one group of 167,663 entries) 9.1 / 0.71.
#pragma once

#include "walk_impl.cuh"

namespace nb {

// Exclusive prefix over the kCoopWarps per-warp counts and their total.
__device__ __forceinline__ int coop_prefix(int v, int w, int &total) {
    // v: lane l < kCoopWarps holds warp l's count
    int incl = v;
#pragma unroll
    for (int o = 1; o < kCoopWarps; o <<= 1) {
        const int t = __shfl_up_sync(NB_FULL, incl, o);
        if ((int)lane_id() >= o) incl += t;
    }
    total = __shfl_sync(NB_FULL, incl, kCoopWarps - 1);
    return __shfl_sync(NB_FULL, incl - v, w);
}

__host__ __device__ inline size_t coop_smem(int list_depth, int stack_depth, bool quad) {
    return (size_t)coop_list_depth(list_depth) * 16 + (quad ? (size_t)kCoopQuadDepth * 40 : 0) +
           (size_t)coop_stack_depth(stack_depth) * 4 + (size_t)kCoopWarps * (32 * 4 + 16) +
           (size_t)kCoopFront * 4 + 16;
}

template <int IPL, bool PHI, bool COMP, bool SAFE, bool QUAD>
__global__ void __maxnreg__((walk_regs<IPL, QUAD || COMP>()))
    coop_walk_kernel(WalkArgs a, int geometric, int second) {
    constexpr int W = kCoopWarps;
    extern __shared__ __align__(16) unsigned char walk_smem[];
    const int DC = coop_list_depth(a.list_depth), SC = coop_stack_depth(a.stack_depth);
    float4 *LA = reinterpret_cast<float4 *>(walk_smem);
    float4 *LQ = LA + DC;
    int4 *s_cnt = reinterpret_cast<int4 *>(walk_smem + (size_t)DC * 16 + (QUAD ? (size_t)kCoopQuadDepth * 40 : 0));
    uint32_t *stk = reinterpret_cast<uint32_t *>(s_cnt + W);
    uint32_t *front = stk + SC;  // ranges the parts of a group share out
    int *scr = reinterpret_cast<int *>(front + kCoopFront) + 32 * (threadIdx.x >> 5);
    __shared__ int s_task, s_last, s_cut;
    DevState *ds = a.ds;
    const int ng = a.nactive ? *a.nactive : ds->ngroups;
    const int nnodes = ds->nnodes;
    const int npart = (int)a.n;
    const int lane = (int)lane_id(), w = (int)(threadIdx.x >> 5), tid = (int)threadIdx.x;
    const unsigned lt = lanemask_lt();
    bool overflow = false, bad = false;
    int max_sp = 0;
    unsigned long long cta_entries = 0, cta_inter = 0, cta_quad = 0;

    const bool all = !second && a.coop_all;
    const int T = second ? ds->queue.ncut : (all ? ng : min(ds->queue.nheavy, a.heavy_cap));
    const int P = T > 0 ? max(1, min(kCoopParts, a.coop_target[second] / T)) : 1;
    const bool may_cut = !second && T <= kCutTasks / P;

    for (int task = blockIdx.x; task < T * P;) {
        const int rec_i = P > 1 ? task / P : task, part = P > 1 ? task % P : 0;
        const uint32_t *rec = second ? a.cut + (size_t)rec_i * kCutWords
                              : all  ? nullptr
                                     : a.heavy + (size_t)rec_i * kHeavyWords;
        const int g = all ? (a.order ? a.order[rec_i] : rec_i) : (int)rec[0];
        const int first = a.grp_first[g], cnt = a.grp_count[g];
        const float4 sph = a.grp_sphere[g];
        const float alpha = geometric ? 0.0f : a.grp_alpha[g];
        const int sys = a.grp_sys[g];
        const float eps2 = a.sys_eps2[sys];
        if (cnt > 32 * IPL) bad = true;
        const Tiling tile = lane_tiling<IPL, W>(cnt, w);
        ISlots<IPL> I;
        load_slots<IPL>(tile, a.pos4, first, cnt, sph, I);

        int sp = 1, nl = 0, nq = 0;
        if (all) {
            if (tid == 0) stk[0] = (uint32_t)a.sys_root[sys] << 3;
        } else {
            sp = min((int)rec[1], min(second ? kCutStack : kHeavyStack, SC));
            for (int k = tid; k < sp; k += 32 * W) stk[k] = rec[kHeavyHead + k];
        }
        if (tid == 0)  // read after the walk
            s_task = (int)gridDim.x + atomicAdd(&ds->queue.coop_head[second], 1);
        long long entries = 0, qentries = 0;
        bool shared = P > 1;  // the top of the tree, expanded by every part of the group
        int nf = 0;
        const int thr = shared ? a.node_count[a.sys_root[sys]] / (kCoopFine * P) : 0;
        __syncthreads();
        for (;;) {
            if (shared && (sp == 0 || nf + sp + 32 * W > kCoopFront)) {
                // this part's ranges: every P-th of those found (and of what
                // is still on the stack when there are that many)
                const int left = min(sp, kCoopFront - nf);
                for (int k = tid; k < left; k += 32 * W) front[nf + k] = stk[k];
                __syncthreads();
                const int found = nf + left;
                sp = found > part ? (found - part + P - 1) / P : 0;
                for (int k = tid; k < sp; k += 32 * W) stk[k] = front[part + k * P];
                shared = false;
                __syncthreads();
            }
            if (sp == 0) break;
            if (may_cut && !shared && entries + qentries >= a.cut_quota && sp <= kCutStack) break;
            // ---- pop: warp w takes ranges 4 w .. 4 w + 3 from the top, fewer
            // warps when the stack could overflow (a range opens at most 8)
            const int room = (SC - sp) / 7;
            const int take = min(sp, min(4 * W, max(4, room)));
            const int rr = 4 * w + (lane >> 3), jj = lane & 7;
            uint32_t e = 0;
            if (rr < take) e = stk[sp - 1 - rr];
            const int node = (int)(e >> 3) + jj;
            const bool slot = rr < take && jj <= (int)(e & 7u);
            const bool in_range = (unsigned)node < (unsigned)nnodes;
            if (slot && !in_range) bad = true;
            const bool has = slot && in_range;

            // ---- MAC (Eq. 2), as in the one-warp walk
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
            const bool leaf_ok = open_leaf && (unsigned)link < (unsigned)npart &&
                                 (unsigned)(mcount - 1) < (unsigned)(npart - link);
            if (open_leaf && !leaf_ok) bad = true;
            // while the parts of a group share the top of the tree, its list
            // entries are part 0's
            const bool keep = !shared || part == 0;

            // ---- this warp's counts
            const bool fine = shared && open_node && a.node_count[node] <= thr;
            const unsigned fm = __ballot_sync(NB_FULL, fine);
            const unsigned om = __ballot_sync(NB_FULL, open_node && !fine);
            const unsigned am = keep ? __ballot_sync(NB_FULL, accept) : 0u;
            const unsigned lm = keep ? __ballot_sync(NB_FULL, leaf_ok) : 0u;
            const int na = __popc(am), nlf = __popc(lm);
            int lf = 0, lc = 0, lincl = 0, ltotal = 0;
            if (lm) {  // opened leaves compacted to lanes 0..nlf-1, counts scanned
                if (leaf_ok) scr[__popc(lm & lt)] = lane;
                __syncwarp();
                const int src = lane < nlf ? scr[lane] : 0;
                lf = __shfl_sync(NB_FULL, link, src);
                const int lcs = __shfl_sync(NB_FULL, mcount, src);
                lc = lane < nlf ? lcs : 0;
                lincl = warp_incl_scan(lc);
                ltotal = __shfl_sync(NB_FULL, lincl, 31);
            }
            const int lexcl = lincl - lc;
            const int nadd = (QUAD ? 0 : na) + ltotal;
            if (lane == 0) s_cnt[w] = make_int4(__popc(om), nadd, na, __popc(fm));
            __syncthreads();  // counts visible; every popped range has been read

            // ---- places of this warp's pushes and entries
            const int4 c4 = lane < W ? s_cnt[lane] : make_int4(0, 0, 0, 0);
            int tpush, tadd, tquad = 0, qoff = 0;
            const int poff = coop_prefix(c4.x, w, tpush);
            const int aoff = coop_prefix(c4.y, w, tadd);
            if constexpr (QUAD) qoff = coop_prefix(c4.z, w, tquad);
            sp -= take;
            const uint32_t range = ((uint32_t)link << 3) | (uint32_t)(mcount - 1);
            if (om >> lane & 1u) {
                const int pos = sp + poff + __popc(om & lt);
                if (pos < SC) stk[pos] = range;
            }
            if (shared) {  // nf + sp + 32 W <= kCoopFront: room for every push
                int tfine;
                const int foff = coop_prefix(c4.w, w, tfine);
                if (fine) front[nf + foff + __popc(fm & lt)] = range;
                nf += tfine;
            }
            sp += tpush;
            if (sp > SC) {
                overflow = true;
                sp = SC;
            }
            max_sp = max(max_sp, sp);

            if constexpr (QUAD) {  // accepted nodes join the node list
                if (nq + tquad > kCoopQuadDepth) {
                    if ((nq & 1) && tid == 0)
                        quad_put(LQ, nq, make_float4(1e18f, 1e18f, 1e18f, 0.0f),
                                 make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f));
                    __syncthreads();
                    flush_runs<0, 0, IPL, PHI, COMP, SAFE, true, W>(tile, LQ, (nq + 1) & ~1, eps2, I);
                    qentries += nq;
                    nq = 0;
                    __syncthreads();
                }
                if (am >> lane & 1u)
                    quad_put(LQ, nq + qoff + __popc(am & lt), A, __ldg(&a.nodeQ[2 * node]),
                             __ldg(&a.nodeQ[2 * node + 1]));
                nq += tquad;
            }
            // ---- entries aoff .. aoff + nadd - 1 of this round's tadd: accepted
            // nodes, then the particles of opened leaves.  Written in windows
            // of what the list still holds (one, unless a leaf is larger than
            // the list)
            const int nacc = QUAD ? 0 : na;
            for (int done = 0;;) {
                const int hi = min(tadd, done + (DC - nl));
                if (!QUAD && (am >> lane & 1u)) {
                    const int p = aoff + __popc(am & lt);
                    if (p >= done && p < hi) list_put(LA, nl + p - done, A);
                }
                const int l0 = max(0, done - aoff - nacc), l1 = min(ltotal, hi - aoff - nacc);
                for (int base = l0; base < l1; base += 32) {
                    const bool starts = lc > 0 && lexcl >= base && lexcl < base + 32;
                    const unsigned smap = __reduce_or_sync(NB_FULL, starts ? 1u << (lexcl - base) : 0u);
                    const int before = __popc(__ballot_sync(NB_FULL, lc > 0 && lexcl < base));
                    const int k = before + __popc(smap & (0xffffffffu >> (31 - lane))) - 1;
                    const int of = __shfl_sync(NB_FULL, lf, k & 31);
                    const int oex = __shfl_sync(NB_FULL, lexcl, k & 31);
                    const int s = base + lane;
                    if (s < l1) list_put(LA, nl + aoff + nacc + s - done, __ldg(&a.pos4[of + s - oex]));
                }
                nl += hi - done;
                done = hi;
                if (done == tadd) break;
                __syncthreads();
                flush_runs<0, 0, IPL, PHI, COMP, SAFE, false, W>(tile, LA, nl, eps2, I);  // DC: even
                entries += nl;
                nl = 0;
                __syncthreads();
            }
            __syncthreads();  // pushes and entries visible to every warp
        }
        if (nl > 0) {
            if ((nl & 1) && tid == 0) list_put(LA, nl, make_float4(1e18f, 1e18f, 1e18f, 0.0f));
            __syncthreads();
            flush_runs<0, 0, IPL, PHI, COMP, SAFE, false, W>(tile, LA, (nl + 1) & ~1, eps2, I);
            entries += nl;
        }
        if constexpr (QUAD) {
            if (nq > 0) {
                if ((nq & 1) && tid == 0)
                    quad_put(LQ, nq, make_float4(1e18f, 1e18f, 1e18f, 0.0f),
                             make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f));
                __syncthreads();
                flush_runs<0, 0, IPL, PHI, COMP, SAFE, true, W>(tile, LQ, (nq + 1) & ~1, eps2, I);
                qentries += nq;
            }
        }
        __syncthreads();  // the list's memory now takes the warps' sums

        float4 *red = LA;  // [W][32 IPL], at most DC
        group_sums<IPL, PHI, COMP>(tile, cnt, I, [&](int idx, const float (&r)[4], float) {
            red[w * (32 * IPL) + idx] = make_float4(r[0], r[1], r[2], r[3]);
        });
        __syncthreads();
        const long long total = entries + qentries;
        // sums of the values v(0) .. v(m - 1), in order
        auto add_up = [&](int m, float (&r)[4], auto v) {
            float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            for (int k = 0; k < m; k++) {
                const float4 x = v(k);
                const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    if constexpr (COMP) neumaier_add(r[q], c[q], xs[q]);
                    else r[q] += xs[q];
                }
            }
            if constexpr (COMP) {
#pragma unroll
                for (int q = 0; q < 4; q++) r[q] += c[q];
            }
        };
        const int m = min(cnt, 32 * IPL);
        // the group's bookkeeping: the index of its first part
        const int owner = second ? (int)rec[2] : rec_i * P;
        if (sp > 0) {  // cut: the open ranges become a record of the second stage
            if (tid == 0) {
                const int k = s_cut = atomicAdd(&ds->queue.ncut, 1);  // k < T P <= kCutTasks
                a.cut_of[task] = k;
                atomicAdd(&a.cut_count[owner], 1);
            }
            __syncthreads();
            uint32_t *cr = a.cut + (size_t)s_cut * kCutWords;
            if (tid == 0) {
                cr[0] = (uint32_t)g;
                cr[1] = (uint32_t)sp;
                cr[2] = (uint32_t)owner;
                cr[3] = (uint32_t)P;
            }
            for (int k = tid; k < sp; k += 32 * W) cr[kHeavyHead + k] = stk[k];
        }
        // several parts: this one's sums go to its slot, and the CTA that
        // finishes the group's last part adds them up
        bool finish = true;
        if (second || P > 1) {
            for (int i = tid; i < m; i += 32 * W) {
                float r[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                add_up(W, r, [&](int k) { return red[k * (32 * IPL) + i]; });
                __stcg(&a.part[(size_t)task * kPartStride + i], make_float4(r[0], r[1], r[2], r[3]));
            }
            if (tid == 0) a.part_entries[task] = (int32_t)total;
            // the fences are the counting thread's, inside the barriers: they
            // cover the writes of the whole CTA before and its reads after
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                s_last = atomicAdd(&a.part_arrive[owner], 1) == P * (second ? a.cut_count[owner] : 1) - 1;
                __threadfence();
            }
            __syncthreads();
            finish = s_last != 0;
        }
        if (finish) {
            // parts of the group: slots rec_i P + k; in the second stage those
            // of its cut parts' records, in the order of the parts
            const int P1 = second ? (int)rec[3] : 1;
            const int cuts = second ? 0 : (P > 1 ? __ldcg(&a.cut_count[owner]) : (sp > 0 ? 1 : 0));
            const float G = cuts > 0 ? 1.0f : a.G;
            const float self = SAFE || cuts > 0 ? 0.0f : rsqrt_fast(eps2);
            for (int i = tid; i < m; i += 32 * W) {
                float r[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (!all) load_sums<PHI>(a, first + i, r);
                if (second) {
                    for (int u = 0; u < P1; u++) {
                        const int c = a.cut_of[owner + u];
                        if (c >= 0)
                            add_up(P, r, [&](int k) { return __ldcg(&a.part[((size_t)c * P + k) * kPartStride + i]); });
                    }
                } else if (P > 1) {
                    add_up(P, r, [&](int k) { return __ldcg(&a.part[((size_t)rec_i * P + k) * kPartStride + i]); });
                } else {
                    add_up(W, r, [&](int k) { return red[k * (32 * IPL) + i]; });
                }
                store_force<PHI>(a, first + i, r, PHI ? a.pos4[first + i].w : 0.0f, G, self);
            }
            if (second) __syncthreads();  // cut_of has been read
            if (tid == 0) {
                long long sum = 0;
                if (second) {
                    sum = a.grp_cost ? a.grp_cost[g] : 0;
                    for (int u = 0; u < P1; u++) {
                        const int c = a.cut_of[owner + u];
                        for (int k = 0; c >= 0 && k < P; k++) sum += __ldcg(&a.part_entries[c * P + k]);
                        a.cut_of[owner + u] = -1;
                    }
                    a.cut_count[owner] = 0;
                } else {
                    sum = all ? 0 : (long long)rec[2];
                    if (P > 1)
                        for (int k = 0; k < P; k++) sum += __ldcg(&a.part_entries[rec_i * P + k]);
                    else
                        sum += total;
                }
                if (second || P > 1) a.part_arrive[owner] = 0;
                if (a.grp_cost) a.grp_cost[g] = (int32_t)sum;
            }
        }
        cta_entries += (unsigned long long)total;
        cta_inter += (unsigned long long)total * (unsigned long long)cnt;
        cta_quad += (unsigned long long)qentries * (unsigned long long)cnt;
        task = s_task;
        __syncthreads();  // s_task, the list and the stack are free for the next group
    }
    if (tid == 0) {
        if (max_sp) atomicMax(&ds->max_stack, max_sp);
        if (cta_entries) {
            atomicAdd(&ds->list_entries, cta_entries);
            atomicAdd(&ds->interactions, cta_inter);
        }
        if (QUAD && cta_quad) atomicAdd(&ds->quad_entries, cta_quad);
        if (overflow) atomicOr(&ds->status, kStatusStackOverflow);
    }
    if (bad) atomicOr(&ds->status, kStatusBadTree);
}

template <int IPL, bool QUAD>
cudaError_t launch_coop_ipl(cudaStream_t s, const WalkArgs &a, const WalkShape &sh, int nsm) {
    const size_t smem = coop_smem(a.list_depth, a.stack_depth, QUAD);
    void (*k)(WalkArgs, int, int);
    if (sh.potential) {
        if (sh.compensated) k = sh.safe ? coop_walk_kernel<IPL, true, true, true, QUAD> : coop_walk_kernel<IPL, true, true, false, QUAD>;
        else k = sh.safe ? coop_walk_kernel<IPL, true, false, true, QUAD> : coop_walk_kernel<IPL, true, false, false, QUAD>;
    } else {
        if (sh.compensated) k = sh.safe ? coop_walk_kernel<IPL, false, true, true, QUAD> : coop_walk_kernel<IPL, false, true, false, QUAD>;
        else k = sh.safe ? coop_walk_kernel<IPL, false, false, true, QUAD> : coop_walk_kernel<IPL, false, false, false, QUAD>;
    }
    cudaError_t err = cudaSuccess;
    // (the kernel's static words count towards the 48 KB that need no asking)
    if (smem > 47 * 1024) err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    // resident CTAs, from the register and shared-memory budgets (no CTA waits
    // for another, so a grid larger than that would only queue); an occupancy
    // query on every launch costs more host time than the launch
    constexpr int by_regs = 65536 / (32 * kCoopWarps * walk_regs<IPL, QUAD>());
    const int more = 65536 / (32 * kCoopWarps * walk_regs<IPL, true>());
    int per_sm = sh.compensated ? more : by_regs;
    per_sm = per_sm > kCoopTarget ? kCoopTarget : per_sm;
    const int by_smem = (int)(227 * 1024 / (smem + 1024));
    if (per_sm > by_smem) per_sm = by_smem;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    if (sh.warps_launched && sh.coop_only) *sh.warps_launched = nsm * per_sm * kCoopWarps;
    k<<<nsm * per_sm, 32 * kCoopWarps, smem, s>>>(a, sh.geometric ? 1 : 0, 0);
    // a list no longer than the quota is never cut
    if (a.longest > a.cut_quota) k<<<nsm * per_sm, 32 * kCoopWarps, smem, s>>>(a, sh.geometric ? 1 : 0, 1);
    return cudaGetLastError();
}

}  // namespace nb
