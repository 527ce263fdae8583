// From-scratch evaluation of given boxes (gb_eval_boxes): W threads per box.
//
// A box's terms are independent, so its threads take one term each, a tile of
// whole groups at a time: the term values go to shared memory, every group of
// the tile is reduced there by its in-place pairwise tree (all groups and the
// F and midpoint trees level by level together), then the groups' values by
// the tree over the groups, then one thread evaluates the outer expression.
// The block's partials follow the same way: one thread per term sweeps its
// template, one thread per coordinate adds the leaf adjoints in ascending
// term and leaf order.  Same operations in the same order as one thread
// walking the box (k_eval_boxes), so the same bits.
//
// What bounds it: many boxes, the FP64 pipe (the midpoint samples' library
// calls); few boxes, the dependent chain of one term.  One thread per box
// left both idle; measured on GB300, one call: 301 boxes of the mixed family,
// n = 10,001, FP32: 87.6 ms with one thread per box, 0.71 ms here; 8192 boxes
// of the chain, n = 100, FP64: 0.95 and 0.24 ms; one box, n = 2: 59 and 45 us.
// One thread a box (k_eval_boxes) is left for products, objectives without a
// sum of two terms, groups of more than 512 terms and group sums beyond the
// shared memory (about 5,900 groups: chain of n = 29,500 with blocks of 10).
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "gb_child.cuh"
#include "gb_launch.h"

using namespace gb;

namespace {

// The box in precision T (FP32: each bound rounded outward as it is loaded)
// or, point != 0, its FP64 midpoint sample.
template <typename T> struct RowView;
template <> struct RowView<double> {
    const double* lo;
    const double* hi;
    int point;
    __device__ __forceinline__ iv64 get(int j) const {
        iv64 x{lo[j], hi[j]};
        if (point) {
            const double m = __dadd_rn(__dmul_rn(0.5, x.lo), __dmul_rn(0.5, x.hi));
            x = iv64{m, m};
        }
        return x;
    }
};
template <> struct RowView<float> {
    const double* lo;
    const double* hi;
    int point;   // (unused)
    __device__ __forceinline__ iv32 get(int j) const {
        return iv32{__double2float_rd(lo[j]), __double2float_ru(hi[j])};
    }
};

// Threads per box W, terms per tile TT, block coordinates per gradient pass CH.
template <int W_, int TT_, int CH_> struct BoxCfg {
    static constexpr int W = W_, TT = TT_, CH = CH_, THREADS = W_ < 128 ? 128 : W_, BPB = THREADS / W_;
};

// Shared memory of one box (bytes), the layout k_box carves it in.
template <typename C, typename I> __host__ __device__ inline size_t box_smem(const GbProg& P) {
    const size_t f = sizeof(I) == 16 ? 0 : (size_t)C::TT * sizeof(I);   // FP64: F and midpoint share one array
    return (sizeof(I) == 16 ? 2 : 1) * (size_t)C::TT * 16 + f + (size_t)P.n_groups * (16 + sizeof(I)) +
           (size_t)P.n_sum * C::CH * (sizeof(I) + 1) + (size_t)(C::CH + GB_MAX_WIN) * P.box_leaves * sizeof(I) +
           (size_t)GB_MAX_OREGS * sizeof(I) + (size_t)C::TT * 4 + 64;
}
template <typename C, typename I> inline size_t box_smem_block(const GbProg& P) {
    return (size_t)P.n_tins * sizeof(GbIns) + (size_t)GB_MAX_ISUM * GB_MAX_TREGS * 4 +
           C::BPB * ((box_smem<C, I>(P) + 15) / 16 * 16);
}

template <typename I> __device__ __forceinline__ I zero_iv() { I z; z.lo = 0; z.hi = 0; return z; }

template <typename C, typename T>
__global__ void __launch_bounds__(C::THREADS) k_box(GbProg P, const GbBoxTile* __restrict__ tiles, int ntiles,
                                                    const double* __restrict__ lo, const double* __restrict__ hi,
                                                    long long nbox, int blk, double* Fo, double* Fmo, double* Go,
                                                    int* mono) {
    typedef typename Prec<T>::I I;
    constexpr int W = C::W, TT = C::TT, CH = C::CH;
    constexpr bool F64 = sizeof(T) == 8;
    extern __shared__ __align__(16) unsigned char smem[];
    auto sync = [] {
        if constexpr (W <= 32) __syncwarp();
        else __syncthreads();
    };
    const int lane = threadIdx.x % W, bx = threadIdx.x / W;
    const long long b0 = (long long)blockIdx.x * C::BPB + bx;
    const bool live = b0 < nbox;
    const long long b = live ? b0 : nbox - 1;   // (a spare slot repeats the last box, unwritten)
    // block: the template instructions and each sum's IVAR offsets
    GbIns* s_ins = (GbIns*)smem;
    int* s_leaf = (int*)(s_ins + P.n_tins);
    {
        const int4* src = (const int4*)P.tins;
        int4* dst = (int4*)s_ins;
        for (int i = threadIdx.x; i < P.n_tins * (int)(sizeof(GbIns) / 16); i += blockDim.x) dst[i] = src[i];
        __syncthreads();
        if ((int)threadIdx.x < P.n_sum) {
            const GbSum S = P.sums[threadIdx.x];
            int l = 0;
            for (int t = 0; t < S.nins; t++)
                if (s_ins[S.ins0 + t].op == D_IVAR) s_leaf[threadIdx.x * GB_MAX_TREGS + l++] = s_ins[S.ins0 + t].aux;
        }
    }
    unsigned char* q = (unsigned char*)(s_leaf + GB_MAX_ISUM * GB_MAX_TREGS) + bx * ((box_smem<C, I>(P) + 15) / 16 * 16);
    auto take = [&](size_t bytes) {
        unsigned char* r = q;
        q += bytes;
        return r;
    };
    iv64* v64 = (iv64*)take((F64 ? 2 : 1) * (size_t)TT * 16);   // FP64: [F | midpoint]; FP32: [midpoint]
    iv64* gmid = (iv64*)take((size_t)P.n_groups * 16);
    I* oa = (I*)take((size_t)GB_MAX_OREGS * sizeof(I));
    I* gF = (I*)take((size_t)P.n_groups * sizeof(I));
    I* acc = (I*)take((size_t)P.n_sum * CH * sizeof(I));
    I* adj = (I*)take((size_t)(CH + GB_MAX_WIN) * P.box_leaves * sizeof(I));
    I* vF = F64 ? (I*)v64 : (I*)take((size_t)TT * sizeof(I));
    iv64* vM = F64 ? v64 + TT : v64;
    ushort2* place = (ushort2*)take((size_t)TT * 4);   // (index in its group, terms of the group)
    int* s_mono = (int*)take(16);
    unsigned char* touched = take((size_t)P.n_sum * CH);
    __syncthreads();

    const double* rlo = lo + (size_t)b * P.n;
    const double* rhi = hi + (size_t)b * P.n;
    const RowView<T> X{rlo, rhi, 0};
    int ops = 0;
    I R[GB_MAX_TREGS];
    // ---- term values, tile by tile, and the tree of every group ----
    for (int w = 0; w < ntiles; w++) {
        const GbBoxTile L = tiles[w];
        const GbSum S = P.sums[L.sum];
        const GbGroup* G = P.groups + S.group0 + L.g0;
        const GbIns* ins = s_ins + S.ins0;
        for (int t = lane; t < L.nt; t += W) {
            int a = 0, z = L.ng - 1;
            while (a < z) {
                const int m = (a + z + 1) >> 1;
                if (G[m].t0 <= L.t0 + t) a = m;
                else z = m - 1;
            }
            place[t] = make_ushort2((unsigned short)(L.t0 + t - G[a].t0), (unsigned short)G[a].count);
        }
        if constexpr (F64) {   // F and midpoint as one list: a lane's view decides which
            for (int it = lane; it < 2 * L.nt; it += W) {
                const int role = it >= L.nt ? 1 : 0, t = it - role * L.nt;
                v64[role * TT + t] = term_fwd<double>(P, S, S.first + (L.t0 + t) * S.step,
                                                      RowView<double>{rlo, rhi, role}, R, ops, ins);
            }
        } else {
            iv64 R64[GB_MAX_TREGS];
            for (int t = lane; t < L.nt; t += W)
                vM[t] = term_fwd<double>(P, S, S.first + (L.t0 + t) * S.step, RowView<double>{rlo, rhi, 1}, R64, ops,
                                         ins);
            for (int t = lane; t < L.nt; t += W)
                vF[t] = term_fwd<T>(P, S, S.first + (L.t0 + t) * S.step, X, R, ops, ins);
        }
        sync();
        for (int s = 1; s < L.cmax; s <<= 1) {
            for (int t = lane; t < L.nt; t += W) {
                const ushort2 p = place[t];
                if ((p.x & (2 * s - 1)) == 0 && p.x + s < p.y) {
                    vF[t] = iadd(vF[t], vF[t + s]);
                    vM[t] = iadd(vM[t], vM[t + s]);
                }
            }
            sync();
        }
        for (int g = lane; g < L.ng; g += W) {
            const int at = G[g].t0 - L.t0;
            gF[S.group0 + L.g0 + g] = vF[at];
            gmid[S.group0 + L.g0 + g] = vM[at];
        }
        sync();
    }
    // ---- the tree over the groups of every sum ----
    for (int k = 0; k < P.n_sum; k++) {
        const GbSum S = P.sums[k];
        I* f = gF + S.group0;
        iv64* m = gmid + S.group0;
        for (int s = 1; s < S.ngroups; s <<= 1) {
            for (int g = lane * 2 * s; g + s < S.ngroups; g += W * 2 * s) {
                f[g] = iadd(f[g], f[g + s]);
                m[g] = iadd(m[g], m[g + s]);
            }
            sync();
        }
    }
    // ---- outer expression: F (and its adjoints) and the midpoint sample in two threads ----
    constexpr int ML = W > 32 ? 32 : 1;
    if (lane == 0 || lane == ML) {
        const bool point = lane == ML;
        if (F64 || point) {
            iv64 sums[GB_MAX_ISUM], O[GB_MAX_OREGS];
            for (int k = 0; k < P.n_sum; k++) {
                const GbSum S = P.sums[k];
                sums[k] = S.ngroups ? (point ? gmid[S.group0] : ((const iv64*)gF)[S.group0]) : iv64{0.0, 0.0};
            }
            const iv64 F = outer_fwd<double>(P, RowView<double>{rlo, rhi, point ? 1 : 0}, sums, O, ops);
            double* out = point ? Fmo : Fo;
            if (live) {
                out[2 * b] = F.lo;
                out[2 * b + 1] = F.hi;
            }
            if (!point && blk >= 0) {
                iv64 OA[GB_MAX_OREGS];
                for (int t = 0; t < P.n_outer; t++) OA[t] = iv64{0.0, 0.0};
                OA[P.outer_root] = iv64{1.0, 1.0};
                reverse_sweep<double>(P.outer, P.n_outer, O, OA, ops);
                for (int t = 0; t < P.n_outer; t++) ((iv64*)oa)[t] = OA[t];
            }
        }
        if (!F64 && !point) {
            I sums[GB_MAX_ISUM], O[GB_MAX_OREGS];
            for (int k = 0; k < P.n_sum; k++) {
                const GbSum S = P.sums[k];
                sums[k] = S.ngroups ? gF[S.group0] : zero_iv<I>();
            }
            const I F = outer_fwd<T>(P, X, sums, O, ops);
            if (live) {
                Fo[2 * b] = F.lo;
                Fo[2 * b + 1] = F.hi;
            }
            if (blk >= 0) {
                I OA[GB_MAX_OREGS];
                for (int t = 0; t < P.n_outer; t++) OA[t] = zero_iv<I>();
                OA[P.outer_root] = mk<T>((T)1, (T)1);
                reverse_sweep<T>(P.outer, P.n_outer, O, OA, ops);
                for (int t = 0; t < P.n_outer; t++) oa[t] = OA[t];
            }
        }
        if (lane == 0) *s_mono = 0;
    }
    sync();
    if (blk < 0) return;
    // ---- partials of block blk, CH coordinates at a time ----
    const int c0 = blk * P.B, c1 = min(P.n, c0 + P.B);
    for (int ca = c0; ca < c1; ca += CH) {
        const int cn = min(CH, c1 - ca);
        for (int k = 0; k < P.n_sum; k++) {
            const GbSum S = P.sums[k];
            if (!S.has_var) {
                for (int jj = lane; jj < cn; jj += W) touched[k * CH + jj] = 0;
                continue;
            }
            const GbIns* ins = s_ins + S.ins0;
            // terms with a coordinate in [ca, ca + cn): first + t step + off_max >= ca, first + t step + off_min < ca + cn
            const int a = ca - S.off_max - S.first, z = ca + cn - 1 - S.off_min - S.first;
            const int ta = a <= 0 ? 0 : (a + S.step - 1) / S.step;
            const int tz = z < 0 ? 0 : min(S.count, z / S.step + 1);
            for (int t = ta + lane; t < tz; t += W) {
                I RA[GB_MAX_TREGS];
                term_vals<T>(P, S, S.first + t * S.step, X, R, ops, ins);
                for (int i = 0; i < S.nins; i++) RA[i] = zero_iv<I>();
                RA[S.nins - 1] = mk<T>((T)1, (T)1);
                reverse_sweep<T>(ins, S.nins, R, RA, ops);
                int l = 0;
                for (int i = 0; i < S.nins; i++)
                    if (ins[i].op == D_IVAR) adj[(t - ta) * P.box_leaves + l++] = RA[i];
            }
            sync();
            for (int jj = lane; jj < cn; jj += W) {
                const int j = ca + jj;
                const int ja = j - S.off_max - S.first, jz = j - S.off_min - S.first;
                const int a2 = ja <= 0 ? 0 : (ja + S.step - 1) / S.step;
                const int z2 = jz < 0 ? 0 : min(S.count, jz / S.step + 1);
                I w = zero_iv<I>();
                bool any = false;
                for (int t = a2; t < z2; t++)
                    for (int l = 0; l < S.nvar_leaves; l++)
                        if (S.first + t * S.step + s_leaf[k * GB_MAX_TREGS + l] == j) {
                            w = iadd(w, adj[(t - ta) * P.box_leaves + l]);
                            any = true;
                        }
                acc[k * CH + jj] = w;
                touched[k * CH + jj] = any ? 1 : 0;
            }
            sync();
        }
        bool hit = false;
        for (int jj = lane; jj < cn; jj += W) {
            const int j = ca + jj;
            I g = zero_iv<I>();
            for (int v = 0; v < P.n_var_leaves; v++) {
                const GbVarLeaf V = P.var_leaves[v];
                if (V.coord == j) g = iadd(g, oa[V.reg]);
            }
            for (int k = 0; k < P.n_sum; k++)
                if (touched[k * CH + jj]) g = iadd(g, imul(oa[P.sums[k].outer_reg], acc[k * CH + jj]));
            if (live) {
                double* o = Go + ((size_t)b * P.B + (j - c0)) * 2;
                o[0] = (double)g.lo;
                o[1] = (double)g.hi;
            }
            hit |= (gt_zero(g.lo) && !same_value(rlo[j], __ldg(P.l + j))) ||
                   (lt_zero(g.hi) && !same_value(rhi[j], __ldg(P.u + j)));
        }
        if (hit) atomicOr(s_mono, 1);
        sync();
    }
    if (lane == 0 && live) mono[b] = *s_mono;
}

// Shared memory a block may take (of the 227 KB): one block per SM (the box
// evaluation), two (the children).
constexpr size_t BOX_SMEM = 200 * 1024, CHILD_SMEM = 100 * 1024;
// Dynamic shared memory a launch gets without asking: 48 KB less the kernel's
// static arrays (k_child_box: 144 bytes).
constexpr size_t FREE_SMEM = 47 * 1024;

// Lets kernel K take `cap` bytes of dynamic shared memory.  The limit belongs
// to the function and the device, not to a launch: set to a call's own size, it
// could be lowered by another thread's call between the setting and the launch.
// So it is set to the most that the dispatch allows, once per device.
template <auto K> cudaError_t allow_smem(size_t cap) {
    static std::atomic<bool> done[64];   // by device ordinal (above: set every time)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 64 && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap);
    if (e == cudaSuccess && dev < 64) done[dev].store(true, std::memory_order_release);
    return e;
}

// Threads per box.  No sum of two terms: one (nothing runs side by side but F
// and the midpoint, and the staging costs more than that saves: up to 3000
// boxes of objectives without a sum, 73-80 us a call here, 64-68 by one thread
// a box).  Small objectives (no sum over 16 terms): the next power of two,
// several boxes per warp.  Else a warp per box once the boxes give every SM 16
// warps; with fewer boxes 128 and then 512 threads, so that a handful of boxes
// still fills the chip.  The tiles must hold every group.
struct BoxPick { int cfg, list; };
template <typename C, typename I> bool fits_smem(const GbProg& P) { return box_smem_block<C, I>(P) <= BOX_SMEM; }

typedef BoxCfg<4, 4, 4> Cfg4;
typedef BoxCfg<8, 8, 8> Cfg8;
typedef BoxCfg<16, 16, 16> Cfg16;
typedef BoxCfg<32, 128, 32> Cfg32;
typedef BoxCfg<128, 128, 64> Cfg128;
typedef BoxCfg<512, 512, 128> Cfg512;

BoxPick box_pick(const GbProg& P, long long nbox) {
    const BoxPick none{-1, 0};
    if (P.any_prod || P.max_terms <= 1 || nbox > (1LL << 30)) return none;
    const bool l0 = P.n_box_tiles[0] > 0, l1 = P.n_box_tiles[1] > 0;
    if (l0 && P.max_terms <= 4 && fits_smem<Cfg4, iv64>(P)) return BoxPick{0, 0};
    if (l0 && P.max_terms <= 8 && fits_smem<Cfg8, iv64>(P)) return BoxPick{1, 0};
    if (l0 && P.max_terms <= 16 && fits_smem<Cfg16, iv64>(P)) return BoxPick{2, 0};
    const long long sms = gb_sm_count();
    if (l0 && nbox >= sms * 16 && fits_smem<Cfg32, iv64>(P)) return BoxPick{3, 0};
    if (l0 && (nbox >= sms * 4 || P.max_terms <= 128) && fits_smem<Cfg128, iv64>(P)) return BoxPick{4, 0};
    if (l1 && fits_smem<Cfg512, iv64>(P)) return BoxPick{5, 1};
    if (l0 && fits_smem<Cfg128, iv64>(P)) return BoxPick{4, 0};
    return none;
}

// ---------------------------------------------------------------------------
// FP64 children of small programs (no term tables: fewer than 16 children a
// parent), W threads per child: the terms of the dirty groups, F and midpoint
// side by side, the clean groups from the parent's cache, then the trees, the
// outer expression and the block's partials as in k_box.  A generation of
// such a solve holds a few dozen children, so it waits for one child's chain:
// one thread per child walked midpoint, F and partials one term after the
// other (n = 2: 70 us a generation).  W <= 16, so warps never wait for one
// another, and every loop around a __syncwarp has the same trip count in all
// lanes whatever their children's blocks.  Generations above
// GB_CHILD_BOX_MAX children fill the chip one thread per child (which tests
// only the children that pass the cut-off): k_eval64.
template <typename C>
__global__ void __launch_bounds__(128) k_child_box(GbProg P, GbPool pool, GbParents par, GbChildren ch, GbSplit sp,
                                                   GbState* st, GbGenConst G) {
    constexpr int W = C::W, TT = C::TT, CH = C::CH, BPB = C::BPB;
    if (st->halt) return;
    if (st->nch > GB_CHILD_BOX_MAX) {   // k_eval64 takes them
        if (blockIdx.x == 0 && threadIdx.x == 0) st->cc_listed = 0;
        return;
    }
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x % W, bx = threadIdx.x / W;
    GbIns* s_ins = (GbIns*)smem;
    int* s_leaf = (int*)(s_ins + P.n_tins);
    {
        const int4* src = (const int4*)P.tins;
        int4* dst = (int4*)s_ins;
        for (int i = threadIdx.x; i < P.n_tins * (int)(sizeof(GbIns) / 16); i += blockDim.x) dst[i] = src[i];
        __syncthreads();
        if ((int)threadIdx.x < P.n_sum) {
            const GbSum S = P.sums[threadIdx.x];
            int l = 0;
            for (int t = 0; t < S.nins; t++)
                if (s_ins[S.ins0 + t].op == D_IVAR) s_leaf[threadIdx.x * GB_MAX_TREGS + l++] = s_ins[S.ins0 + t].aux;
        }
    }
    unsigned char* q = (unsigned char*)(s_leaf + GB_MAX_ISUM * GB_MAX_TREGS) + bx * ((box_smem<C, iv64>(P) + 15) / 16 * 16);
    auto take = [&](size_t bytes) {
        unsigned char* r = q;
        q += bytes;
        return r;
    };
    iv64* v64 = (iv64*)take(2 * (size_t)TT * 16);   // [F | midpoint]
    iv64* gmid = (iv64*)take((size_t)P.n_groups * 16);
    iv64* oa = (iv64*)take((size_t)GB_MAX_OREGS * 16);
    iv64* gF = (iv64*)take((size_t)P.n_groups * 16);
    iv64* acc = (iv64*)take((size_t)P.n_sum * CH * 16);
    iv64* adj = (iv64*)take((size_t)(CH + GB_MAX_WIN) * P.box_leaves * 16);
    ushort2* place = (ushort2*)take((size_t)TT * 4);
    int* s_mono = (int*)take(16);
    unsigned char* touched = take((size_t)P.n_sum * CH);
    __syncthreads();

    const long long nch = st->nch;
    const double gub_prev = gb_key_value(st->gub_key);
    unsigned long long key = ~0ull, nv = 0;
    int ops = 0;
    iv64 R[GB_MAX_TREGS];
    const int wfirst = (threadIdx.x & ~31) / W;   // the warp's first slot
    for (long long base = (long long)blockIdx.x * BPB; base + wfirst < nch; base += (long long)gridDim.x * BPB) {
        const long long ci0 = base + bx;
        const bool in = ci0 < nch;
        const long long ci = in ? ci0 : nch - 1;   // (a spare slot repeats the last child, unwritten)
        const ChildCtx c = child_ctx(par, ci, sp);
        const int blk = c.info.z;
        const View<double> X = view64(pool, par, c, sp);
        const CacheRef<double2> cf = cache64(pool, P, c.slot, 0), cm = cache64(pool, P, c.slot, 1);
        for (int k = 0; k < P.n_sum; k++) {
            const GbSum S = P.sums[k];
            const int2 dr = P.dirty[blk * P.n_sum + k];
            const GbGroup* GR = P.groups + S.group0;
            for (int g = lane; g < S.ngroups; g += W)
                if (g < dr.x || g >= dr.y) {
                    const double2 a = cf[S.group0 + g], b = cm[S.group0 + g];
                    gF[S.group0 + g] = iv64{a.x, a.y};
                    gmid[S.group0 + g] = iv64{b.x, b.y};
                }
            const int t0 = dr.x < dr.y ? GR[dr.x].t0 : 0;
            const int nt = dr.x < dr.y ? GR[dr.y - 1].t0 + GR[dr.y - 1].count - t0 : 0;
            for (int t = lane; t < nt; t += W) {
                int g = dr.x;
                while (g + 1 < dr.y && GR[g + 1].t0 <= t0 + t) g++;
                place[t] = make_ushort2((unsigned short)(t0 + t - GR[g].t0), (unsigned short)GR[g].count);
            }
            for (int it = lane; it < 2 * nt; it += W) {
                const int role = it >= nt ? 1 : 0, t = it - role * nt;
                v64[role * TT + t] = term_fwd<double>(P, S, S.first + (t0 + t) * S.step, PointView{X, role}, R, ops,
                                                      s_ins + S.ins0);
            }
            __syncwarp();
            for (int s = 1; s < TT; s <<= 1) {
                for (int t = lane; t < nt; t += W) {
                    const ushort2 pl = place[t];
                    if ((pl.x & (2 * s - 1)) == 0 && pl.x + s < pl.y) {
                        v64[t] = iadd(v64[t], v64[t + s]);
                        v64[TT + t] = iadd(v64[TT + t], v64[TT + t + s]);
                    }
                }
                __syncwarp();
            }
            for (int g = dr.x + lane; g < dr.y; g += W) {
                gF[S.group0 + g] = v64[GR[g].t0 - t0];
                gmid[S.group0 + g] = v64[TT + GR[g].t0 - t0];
            }
            __syncwarp();
        }
        for (int k = 0; k < P.n_sum; k++) {
            const GbSum S = P.sums[k];
            iv64* f = gF + S.group0;
            iv64* m = gmid + S.group0;
            for (int s = 1; s < S.ngroups; s <<= 1) {
                for (int g = lane * 2 * s; g + s < S.ngroups; g += W * 2 * s) {
                    f[g] = iadd(f[g], f[g + s]);
                    m[g] = iadd(m[g], m[g + s]);
                }
                __syncwarp();
            }
        }
        iv64 F{0.0, 0.0};
        if (lane < 2) {   // lane 0: F and its adjoints, lane 1: the midpoint sample
            iv64 sums[GB_MAX_ISUM], O[GB_MAX_OREGS];
            for (int k = 0; k < P.n_sum; k++) {
                const GbSum S = P.sums[k];
                sums[k] = S.ngroups ? (lane ? gmid : gF)[S.group0] : iv64{0.0, 0.0};
            }
            F = outer_fwd<double>(P, PointView{X, lane}, sums, O, ops);
            if (lane == 0) {
                iv64 OA[GB_MAX_OREGS];
                for (int t = 0; t < P.n_outer; t++) OA[t] = iv64{0.0, 0.0};
                OA[P.outer_root] = iv64{1.0, 1.0};
                reverse_sweep<double>(P.outer, P.n_outer, O, OA, ops);
                for (int t = 0; t < P.n_outer; t++) oa[t] = OA[t];
                *s_mono = 0;
            } else if (in && c.valid && F.hi == F.hi) {
                const unsigned long long k2 = gb_order_key(F.hi);
                key = k2 < key ? k2 : key;
            }
        }
        __syncwarp();
        const int c0 = blk * P.B, c1 = min(P.n, c0 + P.B);   // (at most CH coordinates)
        for (int k = 0; k < P.n_sum; k++) {
            const GbSum S = P.sums[k];
            if (!S.has_var) {
                for (int jj = lane; jj < c1 - c0; jj += W) touched[k * CH + jj] = 0;
                continue;
            }
            const GbIns* ins = s_ins + S.ins0;
            const int a = c0 - S.off_max - S.first, z = c1 - 1 - S.off_min - S.first;
            const int ta = a <= 0 ? 0 : (a + S.step - 1) / S.step;
            const int tz = z < 0 ? 0 : min(S.count, z / S.step + 1);
            for (int t = ta + lane; t < tz; t += W) {
                iv64 RA[GB_MAX_TREGS];
                term_vals<double>(P, S, S.first + t * S.step, X, R, ops, ins);
                for (int i = 0; i < S.nins; i++) RA[i] = iv64{0.0, 0.0};
                RA[S.nins - 1] = iv64{1.0, 1.0};
                reverse_sweep<double>(ins, S.nins, R, RA, ops);
                int l = 0;
                for (int i = 0; i < S.nins; i++)
                    if (ins[i].op == D_IVAR) adj[(t - ta) * P.box_leaves + l++] = RA[i];
            }
            __syncwarp();
            for (int jj = lane; jj < c1 - c0; jj += W) {
                const int j = c0 + jj;
                const int ja = j - S.off_max - S.first, jz = j - S.off_min - S.first;
                const int a2 = ja <= 0 ? 0 : (ja + S.step - 1) / S.step;
                const int z2 = jz < 0 ? 0 : min(S.count, jz / S.step + 1);
                iv64 w{0.0, 0.0};
                bool any = false;
                for (int t = a2; t < z2; t++)
                    for (int l = 0; l < S.nvar_leaves; l++)
                        if (S.first + t * S.step + s_leaf[k * GB_MAX_TREGS + l] == j) {
                            w = iadd(w, adj[(t - ta) * P.box_leaves + l]);
                            any = true;
                        }
                acc[k * CH + jj] = w;
                touched[k * CH + jj] = any ? 1 : 0;
            }
            __syncwarp();
        }
        bool hit = false;
        for (int jj = lane; jj < c1 - c0; jj += W) {
            const int j = c0 + jj;
            iv64 g{0.0, 0.0};
            for (int v = 0; v < P.n_var_leaves; v++) {
                const GbVarLeaf V = P.var_leaves[v];
                if (V.coord == j) g = iadd(g, oa[V.reg]);
            }
            for (int k = 0; k < P.n_sum; k++)
                if (touched[k * CH + jj]) g = iadd(g, imul(oa[P.sums[k].outer_reg], acc[k * CH + jj]));
            if (!gt_zero(g.lo) && !lt_zero(g.hi)) continue;
            const iv64 x = X.get(j);
            hit |= (gt_zero(g.lo) && !same_value(x.lo, __ldg(P.l + j))) ||
                   (lt_zero(g.hi) && !same_value(x.hi, __ldg(P.u + j)));
        }
        if (hit) atomicOr(s_mono, 1);
        __syncwarp();
        if (lane == 0 && in) {
            const bool keep = c.valid && !(F.lo > gub_prev) && *s_mono == 0;
            ch.flo[ci] = c.valid ? canon_lo(F.lo) : __longlong_as_double(0x7ff0000000000000LL);
            ch.flag[ci] = keep ? 1 : 0;
            if (c.valid) nv++;
        }
        __syncwarp();
    }
    warp_min_gub(key, key != ~0ull, st);
    warp_add_ops(ops, &st->ops64);
    for (int o = 16; o; o >>= 1) nv += __shfl_down_sync(0xffffffffu, nv, o);
    if ((threadIdx.x & 31) == 0 && nv) {
        atomicAdd((unsigned long long*)&st->evals64, nv);
        atomicAdd((unsigned long long*)&st->mids, nv);
        atomicAdd((unsigned long long*)&st->children, nv);
    }
    const bool list = nch <= 64LL * 128;
    if (blockIdx.x == 0 && threadIdx.x == 0) st->cc_listed = list ? 1 : 0;
    if (list) list_survivors_last(ch, nch, G, st);
}

template <typename C, typename T>
cudaError_t launch_box(const GbProg& P, int list, const double* lo, const double* hi, long long nbox, int blk,
                       double* F, double* Fmid, double* G, int* mono, cudaStream_t s) {
    const size_t smem = box_smem_block<C, typename Prec<T>::I>(P);
    if (smem > FREE_SMEM) {
        const cudaError_t e = allow_smem<k_box<C, T>>(BOX_SMEM);
        if (e != cudaSuccess) return e;
    }
    k_box<C, T><<<(unsigned)((nbox + C::BPB - 1) / C::BPB), C::THREADS, smem, s>>>(
        P, P.box_tiles[list], P.n_box_tiles[list], lo, hi, nbox, blk, F, Fmid, G, mono);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_pick(const GbProg& P, BoxPick k, const double* lo, const double* hi, long long nbox, int blk,
                        double* F, double* Fmid, double* G, int* mono, cudaStream_t s) {
    switch (k.cfg) {
    case 0: return launch_box<Cfg4, T>(P, k.list, lo, hi, nbox, blk, F, Fmid, G, mono, s);
    case 1: return launch_box<Cfg8, T>(P, k.list, lo, hi, nbox, blk, F, Fmid, G, mono, s);
    case 2: return launch_box<Cfg16, T>(P, k.list, lo, hi, nbox, blk, F, Fmid, G, mono, s);
    case 3: return launch_box<Cfg32, T>(P, k.list, lo, hi, nbox, blk, F, Fmid, G, mono, s);
    case 4: return launch_box<Cfg128, T>(P, k.list, lo, hi, nbox, blk, F, Fmid, G, mono, s);
    default: return launch_box<Cfg512, T>(P, k.list, lo, hi, nbox, blk, F, Fmid, G, mono, s);
    }
}

}  // namespace

extern thread_local long long gb_launch_count;   // kernels launched by this thread (gb_kernels.cu)

int gb_box_coop(const GbProg& P, long long nbox) { return box_pick(P, nbox).cfg >= 0 ? 1 : 0; }

// The dirty terms of a sum, the block's coordinates and the groups must fit a
// child's share of shared memory (W = 16: a warp per two children).
int gb_child_box(const GbProg& P) {
    if (P.any_prod || P.n_groups > 64) return 0;
    const int need = std::max(P.max_dirty_terms, P.B);
    if (need <= 4 && box_smem_block<Cfg4, iv64>(P) <= CHILD_SMEM) return 4;
    if (need <= 8 && box_smem_block<Cfg8, iv64>(P) <= CHILD_SMEM) return 8;
    if (need <= 16 && box_smem_block<Cfg16, iv64>(P) <= CHILD_SMEM) return 16;
    return 0;
}

namespace {
template <typename C>
cudaError_t launch_child_box(const GbProg& P, const GbPool& pool, const GbParents& par, const GbChildren& ch,
                             long long Cmax, const GbSplit& sp, GbState* st, const GbGenConst& G, cudaStream_t s) {
    const size_t smem = box_smem_block<C, iv64>(P);
    if (smem > FREE_SMEM) {
        const cudaError_t e = allow_smem<k_child_box<C>>(CHILD_SMEM);
        if (e != cudaSuccess) return e;
    }
    const unsigned g = (unsigned)std::min<long long>((Cmax + C::BPB - 1) / C::BPB, gb_sm_count() * 8);
    k_child_box<C><<<g, 128, smem, s>>>(P, pool, par, ch, sp, st, G);
    return cudaGetLastError();
}
}  // namespace

cudaError_t gb_launch_child_box(const GbProg& P, const GbPool& pool, const GbParents& par, const GbChildren& ch,
                                long long Cmax, const GbSplit& sp, GbState* st, const GbGenConst& G, cudaStream_t s) {
    switch (gb_child_box(P)) {
    case 4: return launch_child_box<Cfg4>(P, pool, par, ch, Cmax, sp, st, G, s);
    case 8: return launch_child_box<Cfg8>(P, pool, par, ch, Cmax, sp, st, G, s);
    default: return launch_child_box<Cfg16>(P, pool, par, ch, Cmax, sp, st, G, s);
    }
}

cudaError_t gb_launch_eval_boxes(const GbProg& P, const double* lo, const double* hi, float* scratch32,
                                 long long nbox, int blk, int fp32, double* F, double* Fmid, double* G, int* mono,
                                 cudaStream_t s) {
    const BoxPick k = box_pick(P, nbox);
    if (k.cfg < 0) return gb_launch_eval_boxes_thread(P, lo, hi, scratch32, nbox, blk, fp32, F, Fmid, G, mono, s);
    gb_launch_count++;
    return fp32 ? launch_pick<float>(P, k, lo, hi, nbox, blk, F, Fmid, G, mono, s)
                : launch_pick<double>(P, k, lo, hi, nbox, blk, F, Fmid, G, mono, s);
}
