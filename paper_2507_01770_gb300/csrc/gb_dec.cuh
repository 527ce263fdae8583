// Children from the endpoint programs (GbUop): one child per thread, F's lower
// end and the samples' upper ends only.
//
// The cut-off reads F's lower end, the incumbent the samples' upper ends, and
// where the outer expression adds the sums (scaled by positive constants)
// each of them depends on the same end of every table entry alone: half the
// directed additions of the interval walk, which the FP64 pipe (2 lanes a
// clock and SM) bounds.  The programs are straight-line per split position,
// so the stack of NQ kinds stays in registers.
//
// One parent a generation (one): the operations after the last digit-dependent
// one are the same monotone function for every child, so the samples keep
// their smallest value before it and apply it once per thread, and a child
// whose value before it is at or above `cut` -- a point whose own result is
// above the incumbent -- is cut off without it.
#pragma once
#include "gb_child.cuh"

namespace gb {

template <bool LO> __device__ __forceinline__ double dec_add(double a, double b) { return LO ? add_rd(a, b) : add_ru(a, b); }

// Executes uops [a, z) on the stack v (v[0] on top) of NQ kinds; slot 0 is a
// lower end if LO0, the others upper ends.  Tables point at the first kind's
// entries of this parent; off[i] is slot i's kind relative to it.
template <int NQ, bool LO0>
__device__ __forceinline__ void dec_exec(const GbUop* __restrict__ U, int a, int z, const GbDec& D, const double2* tv,
                                         const double2* ts, const double2* nd, const double2* hv, const int (&off)[NQ],
                                         unsigned r, double (&v)[GB_DEC_DEPTH][NQ], int& ops) {
    auto end = [](const double2* q, bool lo) { return lo ? q->x : q->y; };
    for (int u = a; u < z; u++) {
        const GbUop x = U[u];
        if (x.op <= U_ZERO) {
#pragma unroll
            for (int d = GB_DEC_DEPTH - 1; d > 0; d--)
#pragma unroll
                for (int i = 0; i < NQ; i++) v[d][i] = v[d - 1][i];
            const double2* t = x.op == U_ROW ? tv : x.op == U_SEG ? ts : nd;
            const long long st = x.op == U_ROW ? D.tvk : x.op == U_SEG ? D.tsk : D.ndk;
            const int at = x.base + (int)((r >> x.shift) & x.mask);
#pragma unroll
            for (int i = 0; i < NQ; i++) v[0][i] = x.op == U_ZERO ? 0.0 : end(t + off[i] * st + at, LO0 && i == 0);
        } else if (x.op == U_ADD) {
#pragma unroll
            for (int i = 0; i < NQ; i++)
                v[0][i] = LO0 && i == 0 ? add_rd(v[1][i], v[0][i]) : add_ru(v[1][i], v[0][i]);
#pragma unroll
            for (int d = 1; d < GB_DEC_DEPTH - 1; d++)
#pragma unroll
                for (int i = 0; i < NQ; i++) v[d][i] = v[d + 1][i];
            ops += NQ;
        } else {
            const bool node = x.op == U_ADDN, konst = x.op >= U_ADDC;
            const double2* t = node ? nd : hv;
            const long long st = node ? D.ndk : D.hvk;
            const int at = x.base + (int)((r >> x.shift) & x.mask);
#pragma unroll
            for (int i = 0; i < NQ; i++) {
                const bool lo = LO0 && i == 0;
                double2 c = make_double2(x.lo, x.hi);
                if (!konst) c = t[off[i] * st + at];
                if (node || x.op == U_ADDH || x.op == U_ADDC) {
                    v[0][i] = lo ? add_rd(v[0][i], c.x) : add_ru(v[0][i], c.y);
                } else if (x.op == U_SUBH || x.op == U_SUBC) {
                    v[0][i] = lo ? sub_rd(v[0][i], c.y) : sub_ru(v[0][i], c.x);
                } else {   // times a positive interval (Eq. 5: the value's sign picks the end)
                    const double m = sgn(v[0][i]) != lo ? c.x : c.y;
                    v[0][i] = lo ? mul_rd(v[0][i], m) : mul_ru(v[0][i], m);
                }
            }
            ops += NQ;
        }
    }
}

__device__ __forceinline__ bool nan_bits(double x) { return magkey(x) > 0x7ff0000000000000ULL; }

// One chunk of kinds [q0, q0 + NQ) over a thread's share of the children.
// LO0: the chunk starts with kind 0, whose children are cut off, queued and
// tested (mono(child) true: ruled out).
template <int NQ, bool LO0, typename M>
__device__ __forceinline__ void dec_chunk(const GbProg& P, const GbParents& par, const GbChildren& ch,
                                          const GbSplit& sp, const GbDec& D, int q0, bool from_list, bool one,
                                          GbState* st, unsigned* q, unsigned long long& key, unsigned long long& nvalid,
                                          int& ops, const M& mono) {
    const long long lim = from_list ? st->n32 : st->nch;
    const double gub_prev = gb_key_value(st->gub_key);
    const long long stride = (long long)gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    int off[NQ];
#pragma unroll
    for (int i = 0; i < NQ; i++) off[i] = min(q0 + i, D.nk - 1) - q0;
    unsigned long long m[NQ];   // smallest order key per slot: before the suffix if `one`, of the result otherwise
#pragma unroll
    for (int i = 0; i < NQ; i++) m[i] = ~0ull;
    auto tab = [&](const double2* t, long long pstride, long long kstride, long long p) {
        return t + p * pstride + q0 * kstride;
    };
    auto suffix = [&](const GbSplitPos& SP, long long p, double (&v)[GB_DEC_DEPTH][NQ]) {
        dec_exec<NQ, LO0>(P.uops + SP.u0, SP.nu - SP.nsuf, SP.nu, D, tab(D.tv, D.tvp, D.tvk, p), tab(D.ts, D.tsp, D.tsk, p),
                          tab(D.nd, D.ndp, D.ndk, p), tab(D.hv, D.hvp, D.hvk, p), off, 0u, v, ops);
    };
    // one parent: the cut (NaN: none) from the suffix as an affine map, kept
    // only if its own result is above the incumbent
    double cut = __longlong_as_double(0x7ff8000000000000LL);
    __shared__ double s_cut;
    if (LO0 && one && lim > 0 && threadIdx.x == 0) {
        const int spi = P.sp_of_cyc[par.info[0].x];
        if (spi >= 0) {
            const GbSplitPos SP = P.sps[spi];
            double A = 1.0, B = 0.0, S = fabs(gub_prev);
            for (int u = SP.nu - SP.nsuf; u < SP.nu; u++) {
                const GbUop x = P.uops[SP.u0 + u];
                double c = x.lo;
                if (x.op == U_ADDN) c = tab(D.nd, D.ndp, D.ndk, 0)[x.base].x;
                else if (x.op < U_ADDC) c = tab(D.hv, D.hvp, D.hvk, 0)[x.base].x;
                if (x.op == U_ADDN || x.op == U_ADDH || x.op == U_ADDC) B += c, S += fabs(c);
                else if (x.op == U_SUBH || x.op == U_SUBC) B -= c, S += fabs(c);
                else A *= c, B *= c, S *= fmax(c, 1.0);
            }
            const double t = A == 1.0 ? (gub_prev - B) + S * 1e-12 : (gub_prev - B) / A + S / A * 1e-12;
            double v[GB_DEC_DEPTH][NQ];
#pragma unroll
            for (int i = 0; i < NQ; i++) v[0][i] = t;
            suffix(SP, 0, v);
            if (v[0][0] > gub_prev) cut = t;
        }
    }
    if (LO0) {
        if (threadIdx.x == 0) s_cut = cut;
        __syncthreads();
        cut = s_cut;
    }
    const bool has_cut = !nan_bits(cut);
    const unsigned long long kcut = gb_order_key(cut);
    int qn = 0;   // warp-uniform queue length
    for (long long base = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); base < lim; base += stride) {
        const long long idx = base + lane;
        bool need = false, valid = false;
        long long ci = 0;
        if (idx < lim) {
            ci = from_list ? (long long)ch.list32[idx] : idx;
            const ChildCtx c = child_ctx(par, ci, sp);
            const int spi = c.valid ? P.sp_of_cyc[c.info.x] : -1;
            if (LO0) ch.flag[ci] = 0;
            if (spi >= 0) {
                valid = true;
                const GbSplitPos SP = P.sps[spi];
                double v[GB_DEC_DEPTH][NQ];
                dec_exec<NQ, LO0>(P.uops + SP.u0, 0, one ? SP.nu - SP.nsuf : SP.nu, D, tab(D.tv, D.tvp, D.tvk, c.p),
                                  tab(D.ts, D.tsp, D.tsk, c.p), tab(D.nd, D.ndp, D.ndk, c.p),
                                  tab(D.hv, D.hvp, D.hvk, c.p), off, c.r, v, ops);
#pragma unroll
                for (int i = LO0 ? 1 : 0; i < NQ; i++) {
                    const unsigned long long k = nan_bits(v[0][i]) ? ~0ull : gb_order_key(v[0][i]);
                    m[i] = k < m[i] ? k : m[i];
                }
                if (LO0 && !(has_cut && !nan_bits(v[0][0]) && gb_order_key(v[0][0]) >= kcut)) {
                    if (one) suffix(SP, c.p, v);
                    need = !(v[0][0] > gub_prev);
                    ch.flo[ci] = canon_lo(v[0][0]);
                }
            }
        }
        if (!LO0) continue;
        nvalid += __popc(__ballot_sync(0xffffffffu, valid));
        const unsigned bal = __ballot_sync(0xffffffffu, need);
        if (need) q[qn + __popc(bal & ((1u << lane) - 1u))] = (unsigned)ci;
        qn += __popc(bal);
        __syncwarp();
        if (qn >= 32) {
            const unsigned cq = q[qn - 32 + lane];
            ch.flag[cq] = mono(cq) ? 0 : 1;
            qn -= 32;
            __syncwarp();
        }
    }
    if (LO0) {
        if (lane < qn) {   // the rest of the queue
            const unsigned cq = q[lane];
            ch.flag[cq] = mono(cq) ? 0 : 1;
        }
        __syncwarp();
    }
    if (one) {   // the samples' smallest values through the suffix
        bool any = false;
#pragma unroll
        for (int i = LO0 ? 1 : 0; i < NQ; i++) any |= m[i] != ~0ull;
        if (any) {
            const GbSplitPos SP = P.sps[P.sp_of_cyc[par.info[0].x]];
            double v[GB_DEC_DEPTH][NQ];
#pragma unroll
            for (int i = 0; i < NQ; i++) v[0][i] = m[i] != ~0ull ? gb_key_value(m[i]) : 0.0;
            suffix(SP, 0, v);
#pragma unroll
            for (int i = LO0 ? 1 : 0; i < NQ; i++)
                m[i] = m[i] != ~0ull && !nan_bits(v[0][i]) ? gb_order_key(v[0][i]) : ~0ull;
        }
    }
#pragma unroll
    for (int i = LO0 ? 1 : 0; i < NQ; i++) key = m[i] < key ? m[i] : key;
}

// Every chunk, then the counters.
template <int NQ, typename M>
__device__ __forceinline__ void dec_children(const GbProg& P, const GbParents& par, const GbChildren& ch,
                                             const GbSplit& sp, const GbDec& D, bool from_list, bool one, GbState* st,
                                             unsigned* q, const M& mono) {
    unsigned long long key = ~0ull, nvalid = 0;
    int ops = 0;
    dec_chunk<NQ, true>(P, par, ch, sp, D, 0, from_list, one, st, q, key, nvalid, ops, mono);
    for (int q0 = NQ; q0 < D.nk; q0 += NQ)
        dec_chunk<NQ, false>(P, par, ch, sp, D, q0, from_list, one, st, q, key, nvalid, ops, mono);
    warp_min_gub(key, key != ~0ull, st);
    warp_add_ops(ops, &st->ops64);
    if ((threadIdx.x & 31) == 0 && nvalid) {
        atomicAdd((unsigned long long*)&st->evals64, nvalid);
        atomicAdd((unsigned long long*)&st->mids, nvalid * (unsigned long long)(D.nk - 1));
        if (!from_list) atomicAdd((unsigned long long*)&st->children, nvalid);
    }
}

}  // namespace gb
