// The paper's procedure (section 4: S diagonal samples per child, first-order
// test on every coordinate) from per-parent tables.
//
// The interpreter evaluates every dirty term of every child at S + 1 points:
// 2^20 children x 11 points x ~10 terms with their sines and cosines, 38 ms a
// generation on Levy n = 30.  But a term touches w split coordinates and so
// takes at most m^w values over all children at each point, and what the
// outer expression computes from coordinates alone takes few values too.  So
// per parent and point: the term values (k_pp_rows), the term-tree segments
// over at most 10 digit bits, the coordinate partials D over at most 6
// (k_pp_seg), the group trees of the parent's cached values and the outer
// values that no reduction enters.  A child then adds a few table entries per
// reduction and point and runs the rest of the outer expression.  Products
// (IPROD) tabulate the same way; their partials depend on every factor and
// are swept per surviving child with the factors' values from the tables.
// Every value comes from the interpreter's operations in the interpreter's
// order, so the results are bit-identical.
//
// Bound: the FP64 pipe (one addition per table entry and endpoint), where
// most children are cut off in groups (gb_cut.cuh) the latency of the rest.
// Measured on GB300, whole solves with 4^10 children a generation: Levy n = 30,
// 27 generations, 1172 ms with the interpreter, 34.3 ms from the tables, 8.1
// with the groups; Griewank n = 16, 10 generations, 1509, 34.6 and 19.6 ms
// (its survivors' caches, too, come from the tables: k_materialize 73 -> 0.2 ms
// a generation; 0.87 million of its children survive, and what bounds those is
// the product's first-order test, which takes the templates' forward values and
// library factors from the term rows: 32.5 ms before).  The domain decides how
// many survive: over four of them, its bounds moved by up to 2 % of its width,
// 0.52 .. 1.34 million, 1021 .. 2154 ms and 16.0 .. 23.6.
#include <cuda_runtime.h>

#include <algorithm>

#include "gb_dec.cuh"
#include "gb_paper.cuh"

using namespace gb;

namespace {

__device__ __forceinline__ KindView kind_view(const GbPool& pool, const GbParents& par, const GbSplit& sp,
                                              const GbProg& P, long long p, unsigned r, int kind) {
    ChildCtx c;
    c.p = p;
    c.r = r;
    c.info = par.info[p];
    c.slot = par.slot[p];
    c.valid = true;
    return KindView{view64(pool, par, c, sp), kind, P.samples > 0 ? P.samples + 1 : 0};
}

// ---------------------------------------------------------------------------
// Term rows, hoisted outer values (one thread per entry; consecutive threads
// are rows of one kind, so a warp interprets one template at a time) and, in
// blocks of their own past row_blocks, the group trees (reduction k, kind).
constexpr int PP_T = 64;

template <bool PROD>
__device__ __forceinline__ void paper_tree(const GbSum& S, const CacheRef<double2>& cache, double2* a) {
    for (int g = threadIdx.x; g < S.ngroups; g += blockDim.x) a[g] = cache[S.group0 + g];
    __syncthreads();
    int off = 0;
    for (int mL = S.ngroups; mL > 1; mL = (mL + 1) / 2) {
        const int mN = (mL + 1) / 2;
        for (int q = threadIdx.x; q < mN; q += blockDim.x) {
            const double2 x = a[off + 2 * q];
            iv64 v{x.x, x.y};
            if (2 * q + 1 < mL) {
                const double2 y = a[off + 2 * q + 1];
                v = Tree<iv64, PROD>::comb(v, iv64{y.x, y.y});
            }
            a[off + mL + q] = make_double2(v.lo, v.hi);
        }
        __syncthreads();
        off += mL;
    }
}

__global__ void __launch_bounds__(PP_T) k_pp_rows(GbProg P, GbPool pool, GbParents par, GbPaper T, GbSplit sp,
                                                  int row_blocks, GbState* st) {
    if (st->halt) return;
    const long long p = blockIdx.y;
    if (p >= st->parents) return;
    const int spi = P.sp_of_cyc[par.info[p].x];
    if (spi < 0) {   // no layout (the host sends no such parent here): its children would be lost
        if (threadIdx.x == 0) atomicOr(&st->error, 8);
        return;
    }
    const unsigned slot = par.slot[p];
    int ops = 0;
    if ((int)blockIdx.x >= row_blocks) {   // group tree (k, kind)
        const int job = blockIdx.x - row_blocks, k = job % P.n_sum, kind = job / P.n_sum;
        if (kind >= T.nk) return;
        const GbSum S = P.sums[k];
        double2* out = T.nd + ((size_t)p * T.nk + kind) * T.tree_nodes + S.node0;
        const CacheRef<double2> c = kind == 0 ? cache64(pool, P, slot, 0)
                                    : P.samples > 0 ? samp64(pool, P, slot, kind) : cache64(pool, P, slot, 1);
        if (S.prod) paper_tree<true>(S, c, out);
        else paper_tree<false>(S, c, out);
        return;
    }
    const GbSplitPos SP = P.sps[spi];
    const int nterm = SP.ndterm + SP.nx;
    const int n_dirty = SP.tab_entries * T.nk, n_term = n_dirty + SP.nx, n_all = n_term + SP.hrows * T.nk;
    for (int item = blockIdx.x * PP_T + threadIdx.x; item < n_all; item += row_blocks * PP_T) {
        if (item < n_term) {
            const int kind = item < n_dirty ? item / SP.tab_entries : 0;
            const int row = item < n_dirty ? item - kind * SP.tab_entries : SP.tab_entries + (item - n_dirty);
            int lo = 0, hi = nterm - 1;   // the term owning the row (rows ascend with the terms)
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (P.dterms[SP.dterm0 + mid].row <= row) lo = mid;
                else hi = mid - 1;
            }
            const GbDTerm D = P.dterms[SP.dterm0 + lo];
            const unsigned r = (unsigned)(row - D.row) << D.dshift;
            const GbSum S = P.sums[D.sum];
            const int i = S.first + D.term * S.step;
            const KindView X = kind_view(pool, par, sp, P, p, r, kind);
            iv64 R[GB_MAX_TREGS];
            const iv64 v = term_fwd<double>(P, S, i, X, R, ops);
            T.tv[((size_t)p * T.nk + kind) * T.arows + row] = make_double2(v.lo, v.hi);
            if (kind == 0 && S.prod && T.pv) {   // what its reverse sweep reads
                const GbIns* ins = P.tins + S.ins0;
                const size_t o = ((size_t)p * T.arows + row) * T.pw;
                for (int t = 0; t < S.nins; t++) {
                    if (!(ins[t].pad & GB_RV_LIVE) && !(ins[t].pad & GB_RV_VAL)) continue;
                    T.pv[o + t] = make_double2(R[t].lo, R[t].hi);
                    iv64 f;
                    if ((ins[t].pad & GB_RV_LIVE) && rev_factor(ins[t], R, t, f)) T.pf[o + t] = make_double2(f.lo, f.hi);
                }
            }
            if (kind == 0 && !S.prod) {
                iv64 RA[GB_MAX_TREGS];
                for (int t = 0; t < S.nins; t++) RA[t] = iv64{0.0, 0.0};
                RA[S.nins - 1] = iv64{1.0, 1.0};
                const GbIns* ins = P.tins + S.ins0;
                reverse_sweep<double>(ins, S.nins, R, RA, ops);
                double2* tl = T.tl + ((size_t)p * T.arows + row) * T.max_leaves;
                int leaf = 0;
                for (int t = 0; t < S.nins; t++)
                    if (ins[t].op == D_IVAR) tl[leaf++] = make_double2(RA[t].lo, RA[t].hi);
            }
        } else {
            const int q = item - n_term, kind = q / SP.hrows, row = q - kind * SP.hrows;
            int h = 0;
            while (h + 1 < T.n_hoist && T.hoist_pos[spi * T.n_hoist + h + 1].base <= row) h++;
            const GbHoistPos H = T.hoist_pos[spi * T.n_hoist + h];
            const KindView X = kind_view(pool, par, sp, P, p, (unsigned)(row - H.base) << H.shift, kind);
            const int node = T.hoist_node[h];
            iv64 O[GB_MAX_OREGS];
            for (int t = 0; t <= (node & 0xffff); t++) {
                if (!((T.indep >> t) & 1u)) continue;
                const GbIns in = P.outer[t];
                ops += in.pad & 0xff;
                O[t] = outer_ins<double>(in, X, (const iv64*)nullptr, O);
            }
            iv64 v = O[node & 0xffff];
            if (node >> 16) v = ircp(v);
            T.hv[((size_t)p * T.nk + kind) * T.hrows + row] = make_double2(v.lo, v.hi);
        }
    }
    warp_add_ops(ops, &st->ops64);
}

// ---------------------------------------------------------------------------
// Segments (one thread per entry and kind) and partials D (kind 0).
__global__ void __launch_bounds__(128) k_pp_seg(GbProg P, GbParents par, GbPaper T, GbState* st) {
    if (st->halt) return;
    const long long p = blockIdx.y;
    if (p >= st->parents) return;
    const int spi = P.sp_of_cyc[par.info[p].x];
    if (spi < 0) return;
    const GbSplitPos SP = P.sps[spi];
    const int nj = (SP.jb - SP.ja) * P.n_sum;
    const int n_seg = SP.srows * T.nk, n_all = n_seg + (nj << GB_TAB_DBITS);
    int ops = 0;
    for (int item = blockIdx.x * blockDim.x + threadIdx.x; item < n_all; item += gridDim.x * blockDim.x) {
        if (item < n_seg) {
            const int kind = item / SP.srows, row = item - kind * SP.srows;
            int lo = SP.seg0, hi = SP.seg0 + SP.nseg - 1;   // the tabulated segment owning the row
            int si = -1;
            for (int q = lo; q <= hi; q++) {
                const GbSeg G = P.segs[q];
                if (G.level && G.base <= row && row <= G.base + (int)G.mask) {
                    si = q;
                    break;
                }
            }
            if (si < 0) continue;
            const GbSeg G = P.segs[si];
            const unsigned r = (unsigned)(row - G.base) << G.shift;
            const double2* tv = T.tv + ((size_t)p * T.nk + kind) * T.arows;
            iv64 v;
            auto walk = [&](auto& tr) {
                tr.init();
                for (int t = 0; t < 1 << G.level; t++) {
                    const GbDTerm D = P.dterms[SP.dterm0 + G.dterm + t];
                    const double2 a = tv[D.row + (int)((r >> D.dshift) & ((1u << (D.w * P.mshift)) - 1u))];
                    tr.push(iv64{a.x, a.y});
                }
                v = tr.result();
            };
            if (P.sums[G.sum].prod) {
                Tree<iv64, true> tr;
                walk(tr);
            } else {
                Tree<iv64> tr;
                walk(tr);
            }
            ops += 2 << G.level;
            T.ts[((size_t)p * T.nk + kind) * T.srows + row] = make_double2(v.lo, v.hi);
        } else {
            const int e = (item - n_seg) >> GB_TAB_DBITS, c = (item - n_seg) & ((1 << GB_TAB_DBITS) - 1);
            const GbJkD J = P.jkd[SP.jk0 + e];
            if (J.shift < 0 || c > (int)J.mask) continue;
            const int2 rg = P.jk[SP.jk0 + e];
            const unsigned r = (unsigned)c << J.shift;
            const double2* tl = T.tl + (size_t)p * T.arows * T.max_leaves;
            iv64 D{0.0, 0.0};
            for (int q = rg.x; q < rg.y; q++) {
                const GbContrib C = P.contribs[q];
                const double2 a = tl[C.base + (int)((r >> C.dshift) & C.mask) * T.max_leaves];
                D = iadd(D, iv64{a.x, a.y});
            }
            ops += 2 * (rg.y - rg.x);
            T.td[(size_t)p * T.drows + J.base + c] = make_double2(D.lo, D.hi);
        }
    }
    warp_add_ops(ops, &st->ops64);
}

// ---------------------------------------------------------------------------
// Reduction k of a child at one kind: its dirty groups from the segments, the
// group tree's path above them.
template <bool PR>
__device__ __forceinline__ iv64 paper_sum(const GbProg& P, const GbPaper& T, const GbSplitPos& SP, long long p,
                                          int k, int blk, unsigned r, int kind, int& sg, int& ops) {
    const GbSum S = P.sums[k];
    const int2 dr = P.dirty[blk * P.n_sum + k];
    const size_t o = (size_t)p * T.nk + kind;
    const double2* tv = T.tv + o * T.arows;
    const double2* ts = T.ts + o * T.srows;
    const double2* nd = T.nd + o * T.tree_nodes + S.node0;
    auto node = [&](int i) { const double2 v = nd[i]; return iv64{v.x, v.y}; };
    iv64 cur[GB_TAB_MAX_DIRTY];
    if (PR && S.prod) {
        for (int g = dr.x; g < dr.y; g++) cur[g - dr.x] = paper_group<true>(P, SP, k, g, r, sg, tv, ts, ops);
        return tab_path<true>(S, dr, cur, node, ops);
    }
    for (int g = dr.x; g < dr.y; g++) cur[g - dr.x] = paper_group<false>(P, SP, k, g, r, sg, tv, ts, ops);
    return tab_path(S, dr, cur, node, ops);
}

// The child's outer value at one kind from its reductions and the hoisted values.
__device__ __forceinline__ iv64 paper_outer(const GbProg& P, const GbPaper& T, int spi, long long p, unsigned r,
                                            int kind, const iv64* sums, iv64* O, int& ops) {
    const double2* hv = T.hv + ((size_t)p * T.nk + kind) * T.hrows;
    auto hoist = [&](int h) {
        const GbHoistPos H = T.hoist_pos[spi * T.n_hoist + h];
        const double2 v = hv[H.base + (int)((r >> H.shift) & H.mask)];
        return iv64{v.x, v.y};
    };
    for (int t = 0; t < T.n_oprog; t++) {
        const GbOIns in = T.oprog[t];
        if (in.op == D_ISUMV) {
            O[in.dst] = sums[in.a];
            continue;
        }
        const iv64 a = in.ha ? hoist(in.a) : O[in.a];
        iv64 b = a, v;
        if (in.op == D_ADD || in.op == D_SUB || in.op == D_MUL || in.op == D_DIV) b = in.hb ? hoist(in.b) : O[in.b];
        switch (in.op) {
        case D_ADD: v = iadd(a, b); ops += 2; break;
        case D_SUB: v = isub(a, b); ops += 2; break;
        case D_MUL: v = imul(a, b); ops += 8; break;
        case D_NEG: v = ineg(a); break;
        case D_SQR: v = isqr(a); ops += 2; break;
        case D_SCALE: v = iscale(a, in.c); ops += 2; break;
        default: v = slow_fwd(in.op, a, b); ops += 2; break;
        }
        O[in.dst] = v;
    }
    return O[P.outer_root];
}

// The adjoints of all m <= PP_TREE items of a pairwise product tree with adjoint
// a, from the top level down (tree_item_adjoint's products, each formed once).
// node: the items, room for the other levels after them.
constexpr int PP_TREE = 16;
__device__ __forceinline__ void tree_adjoints(iv64 a, int m, iv64* node, iv64* out, int& ops) {
    int off[6], L = 0;
    off[0] = 0;
    for (int sz = m; sz > 1; sz = (sz + 1) / 2) {
        off[L + 1] = off[L] + sz;
        for (int i = 0; i < (sz + 1) / 2; i++) {
            iv64 v = node[off[L] + 2 * i];
            if (2 * i + 1 < sz) v = imul(v, node[off[L] + 2 * i + 1]), ops += 8;
            node[off[L + 1] + i] = v;
        }
        L++;
    }
    out[0] = a;
    for (int l = L - 1; l >= 0; l--) {
        const int sz = off[l + 1] - off[l];
        for (int i = sz - 1; i >= 0; i--) {   // (a node's adjoint is read before its place is taken)
            const iv64 up = out[i >> 1];
            out[i] = (i ^ 1) < sz ? imul(up, node[off[l] + (i ^ 1)]) : up;
            ops += 8;
        }
    }
}

// block_mono's seeder: a term's adjoint in its product, and its sweep.
template <typename F, typename G> struct PaperSeed {
    F& f;
    G& g;
    __device__ __forceinline__ iv64 operator()(int k, int tt) const { return f(k, tt); }
    __device__ __forceinline__ bool sweep(int k, int tt, const GbSum& S, iv64 sd, iv64* A, int& o) const {
        return g(k, tt, S, sd, A, o);
    }
};

// First-order test of a child that passed the cut-off.  Sums: the block's
// coordinates and those within a term's reach of it from the tabulated D, the
// others (every coordinate tested) from the parent's cached D, or swept when
// the pool caches none.  Products: every block swept, a term's adjoint in its
// product from the tabulated factors and group values.
template <bool PR>
__device__ __noinline__ bool paper_mono(const GbProg& P, const GbPool& pool, const GbParents& par, const GbPaper& T,
                                        const ChildCtx& c, const GbSplit& sp, int spi, int& ops) {
    const GbSplitPos SP = P.sps[spi];
    const int blk = c.info.z;
    const View<double> X = view64(pool, par, c, sp);
    iv64 O[GB_MAX_OREGS], OA[GB_MAX_OREGS], sums[GB_MAX_ISUM];
    iv64 R[GB_MAX_TREGS], RA[GB_MAX_TREGS];
    if constexpr (PR) {
        int sg = SP.seg0;
        for (int k = 0; k < P.n_sum; k++) sums[k] = paper_sum<PR>(P, T, SP, c.p, k, blk, c.r, 0, sg, ops);
        outer_fwd<double>(P, X, sums, O, ops);
        const double2* tv = T.tv + (size_t)c.p * T.nk * T.arows;
        const double2* ts = T.ts + (size_t)c.p * T.nk * T.srows;
        const CacheRef<double2> cf = cache64(pool, P, c.slot, 0);
        // A group's term adjoints come from one sweep down its tree when the
        // trees are small (the coordinates ask for a group's terms in turn);
        // one term at a time, every partner product is formed again for each
        // (Griewank n = 16, 6.8e5 children kept in a generation: 20 ms of it).
        iv64 gv[PP_TREE], nodes[2 * PP_TREE], adj[PP_TREE];
        int gk = -1, ak = -1, ag = -1;   // gv holds reduction gk's group values; adj group ag of reduction ak
        auto term_row = [&](const GbPaperSum& ps, int tt) {   // the table row of a product's term for this child
            const int q = tt >= ps.t_lo && tt < ps.t_hi ? ps.d0 + (tt - ps.t_lo)
                                                        : ps.x0 + (tt < ps.t_lo ? tt : tt - (ps.t_hi - ps.t_lo));
            const GbDTerm D = P.dterms[SP.dterm0 + q];
            return D.row + (int)((c.r >> D.dshift) & ((1u << (D.w * P.mshift)) - 1u));
        };
        auto seed_of = [&](int k, int tt) -> iv64 {
            const GbSum S = P.sums[k];
            const GbPaperSum ps = T.psums[spi * P.n_sum + k];
            int lo = 0, hi = S.ngroups - 1;   // the term's group
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (P.groups[S.group0 + mid].t0 <= tt) lo = mid;
                else hi = mid - 1;
            }
            const GbGroup G = P.groups[S.group0 + lo];
            if (ak == k && ag == lo) return adj[tt - G.t0];
            const int2 dr = P.dirty[blk * P.n_sum + k];
            auto gval = [&](int g) {
                if (g >= dr.x && g < dr.y) {
                    int q = paper_seg_of(P, SP, k, g);
                    return paper_group<true>(P, SP, k, g, c.r, q, tv, ts, ops);
                }
                const double2 v = cf[S.group0 + g];
                return iv64{v.x, v.y};
            };
            auto tval = [&](int t) {   // t: index in the group
                const double2 v = tv[term_row(ps, G.t0 + t)];
                return iv64{v.x, v.y};
            };
            const iv64 one{1.0, 1.0};
            if (S.ngroups > PP_TREE || G.count > PP_TREE) {
                const iv64 a = tree_item_adjoint(one, S.ngroups, lo, gval, ops);
                return tree_item_adjoint(a, G.count, tt - G.t0, tval, ops);
            }
            if (gk != k) {
                for (int g = 0; g < S.ngroups; g++) gv[g] = gval(g);
                gk = k;
            }
            const iv64 a = tree_item_adjoint(one, S.ngroups, lo, [&](int g) { return gv[g]; }, ops);
            for (int t = 0; t < G.count; t++) nodes[t] = tval(t);
            tree_adjoints(a, G.count, nodes, adj, ops);
            ak = k;
            ag = lo;
            return adj[tt - G.t0];
        };
        // a product's term swept from its row's values and factors
        auto sweep_of = [&](int k, int tt, const GbSum& S, iv64 sd, iv64* A, int& o) {
            if (!S.prod || !T.pv) return false;
            const size_t at = ((size_t)c.p * T.arows + term_row(T.psums[spi * P.n_sum + k], tt)) * T.pw;
            for (int t = 0; t < S.nins; t++) A[t] = iv64{0.0, 0.0};
            A[S.nins - 1] = sd;
            reverse_sweep_tab(P.tins + S.ins0, S.nins, T.pv + at, T.pf + at, A, o);
            return true;
        };
        const PaperSeed<decltype(seed_of), decltype(sweep_of)> seed{seed_of, sweep_of};
        if (!P.mono_all)
            return block_mono<true, double>(P, blk, X, X, O, OA, R, RA, (double*)nullptr,
                                            (const CacheRef<double2>*)nullptr, blk, ops, seed);
        for (int b = 0; b < P.nb; b++)
            if (block_mono<true, double>(P, b, X, X, O, OA, R, RA, (double*)nullptr,
                                         (const CacheRef<double2>*)nullptr, blk, ops, seed))
                return true;
        return false;
    }
    const int c0 = blk * P.B, c1 = min(P.n, c0 + P.B);
    const int ja = P.mono_all ? SP.ja : c0, jb = P.mono_all ? SP.jb : c1;
    auto hit = [&](int j, const iv64& g) {
        if (!gt_zero(g.lo) && !lt_zero(g.hi)) return false;
        const iv64 x = X.get(j);
        return (gt_zero(g.lo) && !same_value(x.lo, __ldg(P.l + j))) || (lt_zero(g.hi) && !same_value(x.hi, __ldg(P.u + j)));
    };
    auto leaf = [&](int j) {
        bool l = false;
        for (int v = 0; v < P.n_var_leaves; v++) l |= P.var_leaves[v].coord == j;
        return l;
    };
    auto leaves = [&](int j) {
        iv64 g{0.0, 0.0};
        for (int v = 0; v < P.n_var_leaves; v++) {
            const GbVarLeaf L = P.var_leaves[v];
            if (L.coord == j) g = iadd(g, OA[L.reg]), ops += 2;
        }
        return g;
    };
    // Where the sums' outer adjoints are the same for every box, the coordinates
    // that the outer expression does not read need nothing of it and go first
    // (nearly every child is ruled out by one of them, and the outer expression
    // with its sines and its reverse sweep is most of the test).
    const bool cached = pool.gdp || pool.rgdp;
    for (int pass = P.sum_adj ? 0 : 1; pass < 2; pass++) {
        if (pass) {
            int sg = SP.seg0;
            for (int k = 0; k < P.n_sum; k++) sums[k] = paper_sum<PR>(P, T, SP, c.p, k, blk, c.r, 0, sg, ops);
            outer_fwd<double>(P, X, sums, O, ops);
            for (int t = 0; t < P.n_outer; t++) OA[t] = iv64{0.0, 0.0};
            OA[P.outer_root] = iv64{1.0, 1.0};
            reverse_sweep<double>(P.outer, P.n_outer, O, OA, ops);
        }
        auto adj = [&](int k) {
            if (pass) return OA[P.sums[k].outer_reg];
            const double2 a = P.sum_adj[k];
            return iv64{a.x, a.y};
        };
        auto mine = [&](int j) { return P.sum_adj == nullptr || leaf(j) == (pass == 1); };
        for (int j = ja; j < jb; j++) {
            if (!mine(j)) continue;
            iv64 g = pass ? leaves(j) : iv64{0.0, 0.0};
            for (int k = 0; k < P.n_sum; k++) {
                iv64 D;
                if (!paper_D(P, T, SP, c.p, j, k, c.r, D)) continue;
                g = iadd(g, imul(adj(k), D));
                ops += 4;
            }
            if (hit(j, g)) return true;
        }
        for (int j = 0; P.mono_all && cached && j < P.n; j++) {
            if (j == ja) j = jb;
            if (j >= P.n) break;
            if (!mine(j)) continue;
            const int b = j / P.B;
            const double2* row = pool.recs
                ? pool.rgdp + (size_t)pool.rid[(size_t)c.slot * pool.nb + b] * P.n_sum * pool.B + (j - b * P.B)
                : pool.gdp + (size_t)c.slot * P.n_sum * P.n + j;
            const int stride = pool.recs ? pool.B : P.n;
            iv64 g = pass ? leaves(j) : iv64{0.0, 0.0};
            for (int k = 0; k < P.n_sum; k++) {
                if (!P.sums[k].has_var) continue;
                const double2 d = row[(size_t)k * stride];
                if (!d_touched(d)) continue;
                g = iadd(g, imul(adj(k), iv64{d.x, d.y}));
                ops += 4;
            }
            if (hit(j, g)) return true;
        }
    }
    if (!P.mono_all || cached) return false;
    for (int b = 0; b < P.nb; b++) {   // no cache: sweep the blocks beyond the tabulated coordinates
        if (b * P.B >= ja && min(P.n, (b + 1) * P.B) <= jb) continue;
        if (block_mono<false, double>(P, b, X, X, O, OA, R, RA, (double*)nullptr, (const CacheRef<double2>*)nullptr, -1,
                                      ops))
            return true;
    }
    return false;
}

// The child evaluator of gb_cut.cuh over the interval walk.
template <bool PR> struct PaperEval {
    const GbProg& P;
    const GbPaper& T;
    __device__ __forceinline__ iv64 value(const ChildCtx& c, int spi, int kind, int& ops) const {
        const GbSplitPos SP = P.sps[spi];
        iv64 O[GB_MAX_OREGS], sums[GB_MAX_ISUM];
        int sg = SP.seg0;
        for (int k = 0; k < P.n_sum; k++) sums[k] = paper_sum<PR>(P, T, SP, c.p, k, c.info.z, c.r, kind, sg, ops);
        return paper_outer(P, T, spi, c.p, c.r, kind, sums, O, ops);
    }
    __device__ __forceinline__ double lower(const ChildCtx& c, int spi, int& ops) const {
        return value(c, spi, 0, ops).lo;
    }
    __device__ __forceinline__ unsigned long long samples(const ChildCtx& c, int spi, int k0, int k1,
                                                          unsigned long long nan, int& ops) const {
        unsigned long long key = ~0ull;
        for (int kind = k0; kind < k1; kind++) {
            const double v = value(c, spi, kind, ops).hi;
            key = min(key, nan_bits(v) ? nan : gb_order_key(v));
        }
        return key;
    }
    __device__ __forceinline__ unsigned long long bound(const ChildCtx& c, int spi, int k0, int k1, int& ops) const {
        unsigned long long key = ~0ull;   // (below each sample's upper end: its enclosure's lower end over the hulls)
        for (int kind = k0; kind < k1; kind++) {
            const double v = value(c, spi, kind, ops).lo;
            key = min(key, nan_bits(v) ? 0ull : gb_order_key(v));
        }
        return key;
    }
};

template <bool PR>
__global__ void __launch_bounds__(128) k_pp_eval(GbProg P, GbPool pool, GbParents par, GbPaper T, GbChildren ch,
                                                 GbSplit sp, int mode, GbState* st) {
    if (st->halt) return;
    __shared__ unsigned long long s_queue[4][64];
    cut_children(P, par, ch, sp, T.nk, mode, st, s_queue[threadIdx.x >> 5], PaperEval<PR>{P, T},
                 [&](const ChildCtx& c, int spi, int& ops) { return paper_mono<PR>(P, pool, par, T, c, sp, spi, ops); });
}

// The same from the endpoint programs.
__global__ void __launch_bounds__(128) k_pp_dec(GbProg P, GbPool pool, GbParents par, GbPaper T, GbDec D, GbChildren ch,
                                                GbSplit sp, int mode, GbState* st) {
    if (st->halt) return;
    __shared__ unsigned long long s_queue[4][64];
    cut_children(P, par, ch, sp, T.nk, mode, st, s_queue[threadIdx.x >> 5], DecEval<5>{P, D},
                 [&](const ChildCtx& c, int spi, int& ops) { return paper_mono<false>(P, pool, par, T, c, sp, spi, ops); });
}

// ---------------------------------------------------------------------------
// Hull tables (GbCut): a block per (field, kind, parent); a field is the
// entries of a term row, a segment, a hoisted value or (kind 0) a coordinate's
// partial sum.  A warp takes 32 of its entries; the aligned runs of at most 32
// are reduced by shuffles, as order keys (the FP64 pipe would take 16 clocks a
// comparison).  An entry that is not a number becomes the whole line (the
// children decide for themselves).  ends: the samples' tables are read by the
// endpoint programs for a lower bound of upper ends, so theirs hold the largest
// lower and the smallest upper end of a run.
__global__ void __launch_bounds__(128) k_cut_tabs(GbProg P, GbParents par, GbDec D, GbDec out, int n_hoist,
                                                  const GbHoistPos* hoist_pos, int ends, GbState* st) {
    if (st->halt) return;
    const long long p = blockIdx.z;
    const int kind = blockIdx.y;
    if (p >= st->parents) return;
    const int spi = P.sp_of_cyc[par.info[p].x];
    if (spi < 0) return;
    const GbSplitPos SP = P.sps[spi];
    int f = blockIdx.x;
    int base, shift, mask;
    const double2 *src, *dst;
    if (f < SP.nseg) {
        const GbSeg G = P.segs[SP.seg0 + f];
        base = G.base;
        shift = G.shift;
        mask = G.mask;
        src = G.level ? D.ts + p * D.tsp + kind * D.tsk : D.tv + p * D.tvp + kind * D.tvk;
        dst = G.level ? out.ts + p * out.tsp + kind * out.tsk : out.tv + p * out.tvp + kind * out.tvk;
    } else if ((f -= SP.nseg) < n_hoist) {
        const GbHoistPos H = hoist_pos[spi * n_hoist + f];
        base = H.base;
        shift = H.shift;
        mask = H.mask;
        src = D.hv + p * D.hvp + kind * D.hvk;
        dst = out.hv + p * out.hvp + kind * out.hvk;
    } else if (kind == 0 && (f -= n_hoist) < (SP.jb - SP.ja) * P.n_sum) {
        const GbJkD J = P.jkd[SP.jk0 + f];
        if (J.shift < 0) return;
        base = J.base;
        shift = J.shift;
        mask = J.mask;
        src = D.td + p * D.tdp;
        dst = out.td + p * out.tdp;
    } else {
        return;
    }
    const int free_bits = min(max(GB_CUT_LOG2 - shift, 0), __popc((unsigned)mask));
    const unsigned long long neg_inf = gb_order_key(-__longlong_as_double(0x7ff0000000000000LL)),
                             pos_inf = gb_order_key(__longlong_as_double(0x7ff0000000000000LL));
    const bool inner = ends && kind > 0;
    for (int i0 = threadIdx.x & ~31; i0 <= mask; i0 += blockDim.x) {
        const int i = i0 + (threadIdx.x & 31);
        // the run's smallest of one end in lo, its largest of the other in hi
        unsigned long long lo = pos_inf, hi = neg_inf;
        if (i <= mask) {
            const double2 v = src[base + i];
            const bool ok = magkey(v.x) <= 0x7ff0000000000000ULL && magkey(v.y) <= 0x7ff0000000000000ULL;
            lo = ok ? gb_order_key(inner ? v.y : v.x) : neg_inf;
            hi = ok ? gb_order_key(inner ? v.x : v.y) : pos_inf;
        }
        for (int o = 1; o < 1 << free_bits; o <<= 1) {
            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if (i <= mask) const_cast<double2*>(dst)[base + i] = inner ? make_double2(gb_key_value(hi), gb_key_value(lo))
                                                                  : make_double2(gb_key_value(lo), gb_key_value(hi));
    }
}

// The reverse sweep of the outer expression over its constants (the values it
// reads on the way to a sum whose adjoint is fixed are constants).
__global__ void k_outer_adj(GbProg P, double2* adj) {
    iv64 O[GB_MAX_OREGS], A[GB_MAX_OREGS];
    int ops = 0;
    for (int t = 0; t < P.n_outer; t++) {
        const GbIns in = P.outer[t];
        O[t] = A[t] = iv64{0.0, 0.0};
        if (!(in.pad & GB_RV_LIVE)) O[t] = outer_ins<double>(in, View<double>{}, (const iv64*)nullptr, O);
    }
    A[P.outer_root] = iv64{1.0, 1.0};
    reverse_sweep<double>(P.outer, P.n_outer, O, A, ops);
    for (int k = 0; k < P.n_sum; k++) adj[k] = make_double2(A[P.sums[k].outer_reg].lo, A[P.sums[k].outer_reg].hi);
}

// D: the hull tables; R: the children's own.
template <int NQ>
__global__ void __launch_bounds__(CUT_T * CUT_ROLES) k_cut_dec(GbProg P, GbPool pool, GbParents par, GbDec D, GbDec R, GbChildren ch,
                                                 GbSplit sp, GbState* st) {
    if (st->halt) return;
    cut_groups(P, pool, par, ch, sp, D.nk, D.td, D.tdp, st, DecEval<NQ>{P, D}, DecEval<NQ>{P, R});
}
template <bool PR>
__global__ void __launch_bounds__(CUT_T * CUT_ROLES) k_cut_paper(GbProg P, GbPool pool, GbParents par, GbPaper T, GbPaper R,
                                                   GbChildren ch, GbSplit sp, GbState* st) {
    if (st->halt) return;
    cut_groups(P, pool, par, ch, sp, T.nk, T.cut.td, T.drows, st, PaperEval<PR>{P, T}, PaperEval<PR>{P, R});
}

unsigned grid_for(long long items, int per_block) {
    const long long g = (items + per_block - 1) / per_block;
    return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

extern thread_local long long gb_launch_count;   // kernels launched by this thread (gb_kernels.cu)

cudaError_t gb_launch_paper_tables(const GbProg& P, const GbPool& pool, const GbParents& par, const GbPaper& T,
                                   long long K, const GbSplit& sp, GbState* st, cudaStream_t s) {
    gb_launch_count += 2;
    const unsigned sms = (unsigned)gb_sm_count();
    const long long items = (long long)(T.arows + T.hrows) * T.nk;
    const int rb = (int)std::min<long long>(grid_for(items, PP_T), sms * 16);
    k_pp_rows<<<dim3(rb + P.n_sum * T.nk, (unsigned)K), PP_T, 0, s>>>(P, pool, par, T, sp, rb, st);
    const long long segs = (long long)T.srows * T.nk + ((long long)(P.B + 2 * GB_MAX_WIN) * P.n_sum << GB_TAB_DBITS);
    k_pp_seg<<<dim3(std::min<unsigned>(grid_for(segs, 128), sms * 16), (unsigned)K), 128, 0, s>>>(P, par, T, st);
    return cudaGetLastError();
}

cudaError_t gb_launch_paper_eval(const GbProg& P, const GbPool& pool, const GbParents& par, const GbPaper& T,
                                 const GbChildren& ch, long long Cmax, const GbSplit& sp, GbState* st,
                                 cudaStream_t s) {
    GbDec D{T.tv, T.ts, T.nd, T.hv, (long long)T.nk * T.arows, (long long)T.nk * T.srows,
            (long long)T.nk * T.tree_nodes, (long long)T.nk * T.hrows, T.arows, T.srows, T.tree_nodes, T.hrows,
            T.nk, T.td, T.drows};
    const int mode = T.cut.tv ? CUT_GROUPS : CUT_ALL;
    cudaError_t e;
    if (mode == CUT_GROUPS) {
        GbDec C = D;
        C.tv = T.cut.tv;
        C.ts = T.cut.ts;
        C.hv = T.cut.hv;
        C.td = T.cut.td;
        if ((e = gb_launch_cut_tabs(P, par, D, C, T.n_hoist, T.hoist_pos, Cmax >> sp.flog2, T.dec != 0, st, s)) != cudaSuccess) return e;
        if (T.dec) {
            if ((e = gb_launch_cut_dec(P, pool, par, C, D, ch, Cmax, sp, st, s)) != cudaSuccess) return e;
        } else {
            GbPaper H = T;
            H.tv = T.cut.tv;
            H.ts = T.cut.ts;
            H.hv = T.cut.hv;
            gb_launch_count++;
            const unsigned g = std::min<unsigned>(grid_for(Cmax >> GB_CUT_LOG2, 128), (unsigned)gb_sm_count() * 16);
            if (P.any_prod) k_cut_paper<true><<<g, cut_threads(T.nk), 0, s>>>(P, pool, par, H, T, ch, sp, st);
            else k_cut_paper<false><<<g, cut_threads(T.nk), 0, s>>>(P, pool, par, H, T, ch, sp, st);
        }
    }
    gb_launch_count++;
    const unsigned g = std::min<unsigned>(grid_for(Cmax, 128), (unsigned)gb_sm_count() * (mode == CUT_GROUPS ? 8 : 32));
    if (T.dec) k_pp_dec<<<g, 128, 0, s>>>(P, pool, par, T, D, ch, sp, mode, st);
    else if (P.any_prod) k_pp_eval<true><<<g, 128, 0, s>>>(P, pool, par, T, ch, sp, mode, st);
    else k_pp_eval<false><<<g, 128, 0, s>>>(P, pool, par, T, ch, sp, mode, st);
    return cudaGetLastError();
}

cudaError_t gb_launch_cut_tabs(const GbProg& P, const GbParents& par, const GbDec& D, const GbDec& out, int n_hoist,
                               const GbHoistPos* hoist_pos, long long K, bool ends, GbState* st, cudaStream_t s) {
    gb_launch_count++;
    const int fields = std::max(1, P.max_nseg + n_hoist + (P.B + 2 * GB_MAX_WIN) * P.n_sum);
    k_cut_tabs<<<dim3((unsigned)fields, (unsigned)D.nk, (unsigned)K), 128, 0, s>>>(P, par, D, out, n_hoist, hoist_pos,
                                                                                 ends ? 1 : 0, st);
    return cudaGetLastError();
}

cudaError_t gb_launch_outer_adj(const GbProg& P, double2* adj, cudaStream_t s) {
    gb_launch_count++;
    k_outer_adj<<<1, 1, 0, s>>>(P, adj);
    return cudaGetLastError();
}

cudaError_t gb_launch_cut_dec(const GbProg& P, const GbPool& pool, const GbParents& par, const GbDec& C, const GbDec& D,
                              const GbChildren& ch, long long Cmax, const GbSplit& sp, GbState* st, cudaStream_t s) {
    gb_launch_count++;
    const unsigned g = std::min<unsigned>(grid_for(Cmax >> GB_CUT_LOG2, 128), (unsigned)gb_sm_count() * 16);
    if (D.nk > 2) k_cut_dec<5><<<g, cut_threads(D.nk), 0, s>>>(P, pool, par, C, D, ch, sp, st);
    else k_cut_dec<1><<<g, cut_threads(D.nk), 0, s>>>(P, pool, par, C, D, ch, sp, st);
    return cudaGetLastError();
}
