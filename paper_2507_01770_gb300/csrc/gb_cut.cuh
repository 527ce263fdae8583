// The children of a large fan-out (one child per thread): groups cut off as a
// whole, then the children of the groups left.
//
// A generation of 4^10 children keeps a few hundred.  The 2^GB_CUT_LOG2
// children that differ in their low digit bits only read, of every table, an
// aligned run of entries; with each run replaced by its hull (k_cut_tabs) the
// child's own operations give an enclosure of what every child of the group
// computes: additions, products and the other IEEE operations with directed
// rounding are inclusion isotone, endpoint by endpoint (the widened library
// values of exp, sin and cos are not, so an outer expression that applies them
// to a sum takes no groups, and the test below skips coordinates that the
// outer expression reads itself).  No child of a group is looked at when
//   - the bound of F's lower end is above the incumbent: the cut-off removes
//     every child; or
//   - some partial's enclosure has a fixed sign and no child touches the bound
//     the sign points to (every child is ruled out by the first-order test),
//     and no sample of any child can lower the incumbent.  To know early what
//     the incumbent comes to, the group with the smallest bound of its samples
//     is sampled first (by the last block of the group pass); the others are
//     compared with the incumbent as it stands when their turn comes, and of
//     those still walked the samples alone are taken.
// The others are walked one child per thread.  Of a child that the cut-off
// removes no sample is needed: its lower bound is above the incumbent, and each
// sample's upper end is above the value of f at that point, which is above the
// lower bound.  So the flags, the bounds of the survivors and the incumbent
// are those of evaluating every child at every point.
//
// Bound: the FP64 pipe while every child was walked.  Measured on GB300 with
// 4^10 children a generation, whole solves: chain n = 100 (128 generations)
// 26.4 -> 19.4 ms, a child kernel of 110 us -> 20 after 30 for the groups;
// paper mode, Levy n = 30 (27 generations) 34.3 -> 8.25 ms (18.6
// before a group is sampled first, its samples taken five at a time and the
// test's fixed adjoints used first).  From a fan-out of
// 2^10 on: the hull tables and the groups take two launches (8.0 and 22.2 us
// for the chain) and a smaller fan-out is one latency chain either way.
// Not taken: after an FP32 pass (its list says which children are left), and
// outside paper mode for outer expressions that are not a plain sum of sums.
#pragma once
#include "gb_child.cuh"

namespace gb {

// True when some coordinate's partial rules out every child of the group that
// starts at child c (sums whose outer adjoint is the same for every box: the
// partial is their sum of it times the tabulated D; td: the parent's hulls of D).
__device__ __forceinline__ bool group_ruled_out(const GbProg& P, const GbPool& pool, const GbParents& par,
                                                const GbSplit& sp, const GbSplitPos& SP, const ChildCtx& c,
                                                const double2* td, int& ops) {
    if (!P.sum_adj) return false;
    const unsigned last = min(c.r | ((1u << GB_CUT_LOG2) - 1u), (1u << (c.info.y * sp.mshift)) - 1u);
    const int c0 = c.info.z * P.B;
    const int j0 = P.mono_all ? SP.ja : c0, j1 = P.mono_all ? SP.jb : min(P.n, c0 + P.B);
    for (int j = j0; j < j1; j++) {
        iv64 g{0.0, 0.0};
        bool ok = true;
        for (int v = 0; v < P.n_var_leaves; v++) ok = ok && P.var_leaves[v].coord != j;
        for (int k = 0; k < P.n_sum && ok; k++) {
            const int at = SP.jk0 + (j - SP.ja) * P.n_sum + k;
            const int2 rg = P.jk[at];
            if (rg.x == rg.y) continue;
            const GbJkD J = P.jkd[at];
            ok = J.shift >= 0;
            if (!ok) break;
            const double2 e = td[J.base + (int)((c.r >> J.shift) & J.mask)];
            const double2 a = P.sum_adj[k];
            g = iadd(g, imul(iv64{a.x, a.y}, iv64{e.x, e.y}));
            ops += 4;
        }
        const bool pos = gt_zero(g.lo), neg = lt_zero(g.hi);
        if (!ok || (!pos && !neg)) continue;
        const double edge = pos ? __ldg(P.l + j) : __ldg(P.u + j);
        const unsigned k = (unsigned)(j - c.info.x);
        if (k < (unsigned)c.info.y) {   // the faces of every piece the group takes
            const unsigned m1 = (1u << sp.mshift) - 1u;
            const unsigned d0 = (c.r >> (k * sp.mshift)) & m1, d1 = (last >> (k * sp.mshift)) & m1;
            const double* b = par.bnd + ((size_t)c.p * sp.dmax + k) * (sp.m + 1);
            for (unsigned d = d0; d <= d1; d++) ok = ok && !same_value(b[pos ? d : d + 1], edge);
        } else {
            const iv64 x = box_view64(pool, c.slot).get(j);
            ok = !same_value(pos ? x.lo : x.hi, edge);
        }
        if (ok) return true;
    }
    return false;
}

// Threads of a block that take a group each, and the roles that share its work:
// the first bounds F and then tries the first-order test while the others
// bound the samples of the groups that F does not cut off, a share of the kinds
// each.  (One thread doing all of it was one chain of 170k clocks, Levy n = 30
// at 10 samples: a solve 8.52 ms, 8.25 with the roles.)
constexpr int CUT_T = 128, CUT_ROLES = 4;
inline int cut_threads(int nk) {   // about five kinds a sample role
    const int roles = 1 + (nk - 1 + 4) / 5;
    return CUT_T * (roles < CUT_ROLES ? roles : CUT_ROLES);
}

// Groups: appends those to walk to ch.list32 (their number in st->n32, zero
// at the start of a generation), clears every flag and counts the children.
// The first child's place in ch.flo tells why a group is walked: the bound of
// its samples when the first-order test rules it out, else -inf.
// e: the child evaluator over the hull tables, er over the children's own; td,
// tdp: the partial sums' hulls.
template <typename E, typename R>
__device__ __forceinline__ void cut_groups(const GbProg& P, const GbPool& pool, const GbParents& par,
                                           const GbChildren& ch, const GbSplit& sp, int nk, const double2* td,
                                           long long tdp, GbState* st, const E& e, const R& er) {
    const double gub_prev = gb_key_value(st->gub_key);
    const long long total = st->nch >> GB_CUT_LOG2, stride = (long long)gridDim.x * CUT_T;
    const unsigned long long gmask = total > 1 ? ~0ull >> __clzll(total - 1) : 0;
    const int lane = threadIdx.x & 31, t = threadIdx.x % CUT_T, role = threadIdx.x / CUT_T;
    const int per = (nk - 1 + blockDim.x / CUT_T - 2) / (blockDim.x / CUT_T - 1);   // kinds of a sample role
    __shared__ unsigned s_pass[CUT_T / 32];
    __shared__ unsigned long long s_key[CUT_ROLES - 1][CUT_T];
    unsigned long long nvalid = 0, seed = ~0ull;
    int ops = 0;
    for (long long base = blockIdx.x * (long long)CUT_T; base < total; base += stride) {
        const long long g = base + t;
        ChildCtx c{};
        int spi = -1;
        if (g < total) {
            c = child_ctx(par, g << GB_CUT_LOG2, sp);
            spi = c.valid ? P.sp_of_cyc[c.info.x] : -1;
        }
        bool walk = false, ruled = false;
        if (role == 0) {
            if (g < total) {
                uint4* f = reinterpret_cast<uint4*>(ch.flag + (g << GB_CUT_LOG2));
                f[0] = f[1] = make_uint4(0, 0, 0, 0);
            }
            if (spi >= 0) {
                nvalid += min(1u << GB_CUT_LOG2, (1u << (c.info.y * sp.mshift)) - c.r);
                walk = !(e.lower(c, spi, ops) > gub_prev);
            }
            const unsigned b = __ballot_sync(0xffffffffu, walk);
            if (lane == 0) s_pass[t >> 5] = b;
        }
        __syncthreads();
        if (role == 0) {
            ruled = walk && group_ruled_out(P, pool, par, sp, P.sps[spi], c, td + c.p * tdp, ops);
        } else {
            const int k0 = 1 + (role - 1) * per, k1 = min(nk, k0 + per);
            unsigned long long k = ~0ull;
            // (read only where the test can rule a group out)
            if (P.sum_adj && k0 < k1 && ((s_pass[t >> 5] >> lane) & 1u)) k = e.bound(c, spi, k0, k1, ops);
            s_key[role - 1][t] = k;
        }
        __syncthreads();
        if (role == 0) {
            if (walk) {
                unsigned long long k = 0;   // below every key of a number
                if (ruled) {
                    k = ~0ull;
                    for (int i = 0; i < (int)blockDim.x / CUT_T - 1; i++) k = min(k, s_key[i][t]);
                    walk = k < st->gub_key;
                    if (walk && nk > 2) seed = min(seed, (k & ~gmask) | (unsigned long long)g);
                }
                if (walk) ch.flo[g << GB_CUT_LOG2] = k ? gb_key_value(k) : -__longlong_as_double(0x7ff0000000000000LL);
            }
            const unsigned bal = __ballot_sync(0xffffffffu, walk);
            unsigned at = 0;
            if (lane == 0 && bal) at = (unsigned)atomicAdd((unsigned long long*)&st->n32, (unsigned long long)__popc(bal));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (walk) ch.list32[at + __popc(bal & ((1u << lane) - 1u))] = (unsigned)g;
        }
    }
    for (int o = 16; o; o >>= 1) {
        nvalid += __shfl_down_sync(0xffffffffu, nvalid, o);
        seed = min(seed, __shfl_down_sync(0xffffffffu, seed, o));
    }
    if (lane == 0 && nvalid) {
        atomicAdd((unsigned long long*)&st->evals64, nvalid);
        atomicAdd((unsigned long long*)&st->mids, nvalid * (unsigned long long)(nk - 1));
        atomicAdd((unsigned long long*)&st->children, nvalid);
    }
    if (lane == 0 && seed != ~0ull) atomicMin(&st->cut_seed, seed);
    warp_add_ops(ops, &st->ops64);
    if (nk == 2) return;   // (one sample a child: the groups' own bounds come too late to save as much)
    __shared__ bool s_last;
    if (!arrive_last(&st->cc_done, gridDim.x, &s_last)) return;
    seed = __ldcg(&st->cut_seed);
    __syncthreads();
    if (threadIdx.x == 0) {
        st->cc_done = 0;
        st->cut_seed = ~0ull;
    }
    if (seed == ~0ull) return;
    // a warp's share of the kinds, a child per lane
    const int nw = blockDim.x >> 5, w = threadIdx.x >> 5, share = (nk - 1 + nw - 1) / nw;
    const int k0 = 1 + w * share, k1 = min(nk, k0 + share);
    unsigned long long key = ~0ull;
    ops = 0;
    if (k0 < k1) {
        const ChildCtx c = child_ctx(par, (long long)((seed & gmask) << GB_CUT_LOG2) + lane, sp);
        if (c.valid) key = er.samples(c, P.sp_of_cyc[c.info.x], k0, k1, ~0ull, ops);
    }
    warp_min_gub(key, key != ~0ull, st);
    warp_add_ops(ops, &st->ops64);
}

// Children of the listed groups (CUT_GROUPS), of the FP32 pass's list
// (CUT_LIST) or all of them (CUT_ALL), one per thread.  Those of a warp that
// pass the cut-off are queued in shared memory (q: 64 entries of the warp;
// at most 31 left over + 32 new) and sampled and tested 32 at a time, every
// lane busy (few pass).
enum { CUT_ALL = 0, CUT_LIST = 1, CUT_GROUPS = 2 };
template <typename E, typename M>
__device__ __forceinline__ void cut_children(const GbProg& P, const GbParents& par, const GbChildren& ch,
                                             const GbSplit& sp, int nk, int mode, GbState* st, unsigned long long* q, const E& e,
                                             const M& mono) {
    const double gub_prev = gb_key_value(st->gub_key);
    const long long lim = mode == CUT_GROUPS ? st->n32 << GB_CUT_LOG2 : mode == CUT_LIST ? st->n32 : st->nch;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    int qn = 0;   // warp-uniform queue length
    int ops = 0;
    unsigned long long key = ~0ull, nvalid = 0;
    constexpr unsigned long long RULED_OUT = 1ull << 63;   // (a generation may hold up to 2^32 children)
    auto test = [&](unsigned long long e0) {
        const long long ci = (long long)(e0 & ~RULED_OUT);
        const ChildCtx c = child_ctx(par, ci, sp);
        const int spi = P.sp_of_cyc[c.info.x];
        key = min(key, e.samples(c, spi, 1, nk, ~0ull, ops));
        if (!(e0 & RULED_OUT)) ch.flag[ci] = mono(c, spi, ops) ? 0 : 1;
    };
    for (long long base = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); base < lim; base += stride) {
        const long long idx = base + lane;
        bool need = false, valid = false;
        long long ci = 0;
        unsigned long long ruled = 0;
        if (mode == CUT_GROUPS) {   // (the warp's children are one group)
            const long long c0 = (long long)ch.list32[base >> GB_CUT_LOG2] << GB_CUT_LOG2;
            const double b = ch.flo[c0];
            __syncwarp();
            // Other warps lower the incumbent meanwhile, so two lanes may read two
            // values: lane 0 decides for the warp (the ballots below need all lanes).
            if (__shfl_sync(0xffffffffu, lane == 0 && gb_order_key(b) >= *(volatile unsigned long long*)&st->gub_new_key, 0)) continue;
            if (b > -__longlong_as_double(0x7ff0000000000000LL)) ruled = RULED_OUT;
            ci = c0 + lane;
        } else if (idx < lim) {
            ci = mode == CUT_LIST ? (long long)ch.list32[idx] : idx;
        }
        if (idx < lim) {
            const ChildCtx c = child_ctx(par, ci, sp);
            const int spi = c.valid ? P.sp_of_cyc[c.info.x] : -1;
            if (mode != CUT_GROUPS) ch.flag[ci] = 0;
            if (spi >= 0) {
                valid = true;
                const double lo = e.lower(c, spi, ops);
                need = !(lo > gub_prev);
                if (need) ch.flo[ci] = canon_lo(lo);
            }
        }
        nvalid += __popc(__ballot_sync(0xffffffffu, valid));
        const unsigned bal = __ballot_sync(0xffffffffu, need);
        if (need) q[qn + __popc(bal & ((1u << lane) - 1u))] = (unsigned long long)ci | ruled;
        qn += __popc(bal);
        __syncwarp();
        if (qn >= 32) {
            test(q[qn - 32 + lane]);
            qn -= 32;
            __syncwarp();
        }
    }
    if (lane < qn) test(q[lane]);   // the rest of the queue
    __syncwarp();
    warp_min_gub(key, key != ~0ull, st);
    warp_add_ops(ops, &st->ops64);
    if (lane == 0 && nvalid && mode != CUT_GROUPS) {
        atomicAdd((unsigned long long*)&st->evals64, nvalid);
        atomicAdd((unsigned long long*)&st->mids, nvalid * (unsigned long long)(nk - 1));
        if (mode == CUT_ALL) atomicAdd((unsigned long long*)&st->children, nvalid);
    }
}

}  // namespace gb
