// Device helpers of the paper-mode tables (gb_kernels_paper.cu, and the
// materialisation of their survivors in gb_kernels.cu).
#pragma once
#include "gb_child.cuh"

namespace gb {

// Views of a box by kind: 0 the box itself, else its sample point (m1 = S + 1:
// diagonal point kind of S; m1 = 0: the midpoint).
struct KindView {
    View<double> v;
    int kind, m1;
    __device__ __forceinline__ iv64 get(int j) const {
        if (kind == 0) return v.get(j);
        if (m1 == 0) return MidView{v}.get(j);
        return SampleView{v, kind, m1}.get(j);
    }
};

// Value of one dirty group of reduction k for child index r, from the term
// tree's segments starting at sg (Tree::push_level forms the group's pairwise
// tree); sg advances past the group's run.
template <bool PROD>
__device__ __forceinline__ iv64 paper_group(const GbProg& P, const GbSplitPos& SP, int k, int g, unsigned r, int& sg,
                                            const double2* tv, const double2* ts, int& ops) {
    const int send = SP.seg0 + SP.nseg;
    Tree<iv64, PROD> tr;
    tr.init();
    int ns = 0;
    while (sg < send) {
        const GbSeg G = P.segs[sg];
        if (G.sum != k || G.group != g) break;
        const int at = G.base + (int)((r >> G.shift) & G.mask);
        const double2 v = G.level ? ts[at] : tv[at];
        tr.push_level(iv64{v.x, v.y}, G.level);
        ns++;
        sg++;
    }
    ops += (PROD ? 8 : 2) * (ns > 0 ? ns - 1 : 0);
    return tr.result();
}

// First segment of (reduction k, group g).
__device__ __forceinline__ int paper_seg_of(const GbProg& P, const GbSplitPos& SP, int k, int g) {
    int sg = SP.seg0;
    const int send = SP.seg0 + SP.nseg;
    while (sg < send) {
        const GbSeg G = P.segs[sg];
        if (G.sum > k || (G.sum == k && G.group >= g)) break;
        sg++;
    }
    return sg;
}

// D of (coordinate j in [SP.ja, SP.jb), sum k) for child index r: the sum from
// [0, 0] of its leaf adjoints in ascending term and leaf order (block_D's
// value), tabulated or added up here; false when no term touches j.
__device__ __forceinline__ bool paper_D(const GbProg& P, const GbPaper& T, const GbSplitPos& SP, long long p, int j,
                                        int k, unsigned r, iv64& D) {
    const int at = SP.jk0 + (j - SP.ja) * P.n_sum + k;
    const int2 rg = P.jk[at];
    if (rg.x == rg.y) return false;
    const GbJkD J = P.jkd[at];
    if (J.shift >= 0) {
        const double2 e = T.td[(size_t)p * T.drows + J.base + (int)((r >> J.shift) & J.mask)];
        D = iv64{e.x, e.y};
        return true;
    }
    const double2* tl = T.tl + (size_t)p * T.arows * T.max_leaves;
    D = iv64{0.0, 0.0};
    for (int q = rg.x; q < rg.y; q++) {
        const GbContrib C = P.contribs[q];
        const double2 e = tl[C.base + (int)((r >> C.dshift) & C.mask) * T.max_leaves];
        D = iadd(D, iv64{e.x, e.y});
    }
    return true;
}

// The same as a cache row entry (block_D's form: untouched is (+inf, -inf)).
__device__ __forceinline__ double2 paper_D_row(const GbProg& P, const GbPaper& T, const GbSplitPos& SP, long long p,
                                               int j, int k, unsigned r) {
    iv64 D;
    if (!paper_D(P, T, SP, p, j, k, r, D))
        return make_double2(__longlong_as_double(0x7ff0000000000000LL),
                            __longlong_as_double((long long)0xfff0000000000000ULL));
    return make_double2(D.lo, D.hi);
}

// The values of a child's dirty groups at every kind, one (kind, group) per
// lane in turn: put(global group, kind, value).
template <typename F>
__device__ __forceinline__ void paper_dirty_groups(const GbProg& P, const GbPool& pool, const GbPaper& T,
                                                   const ChildCtx& c, int lane, F put) {
    const int blk = c.info.z;
    const GbSplitPos SP = P.sps[P.sp_of_cyc[c.info.x]];
    int ops = 0;
    for (int k = 0; k < P.n_sum; k++) {
        const GbSum S = P.sums[k];
        const int2 dr = P.dirty[blk * P.n_sum + k];
        const int ng = dr.y - dr.x;
        for (int it = lane; it < ng * T.nk; it += 32) {
            const int kind = it / ng, g = dr.x + it - kind * ng;
            const size_t o = (size_t)c.p * T.nk + kind;
            int sg = paper_seg_of(P, SP, k, g);
            const iv64 v = S.prod ? paper_group<true>(P, SP, k, g, c.r, sg, T.tv + o * T.arows, T.ts + o * T.srows, ops)
                                  : paper_group<false>(P, SP, k, g, c.r, sg, T.tv + o * T.arows, T.ts + o * T.srows, ops);
            put(S.group0 + g, kind, v);
        }
    }
}

}  // namespace gb
