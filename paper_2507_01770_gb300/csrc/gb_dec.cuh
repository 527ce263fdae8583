// Children from the endpoint programs (GbUop): F's lower end and the samples'
// upper ends only.
//
// The cut-off reads F's lower end, the incumbent the samples' upper ends, and
// where the outer expression adds the sums (scaled by positive constants)
// each of them depends on the same end of every table entry alone: half the
// directed additions of the interval walk, which the FP64 pipe (2 lanes a
// clock and SM) bounds.  The programs are straight-line per split position,
// so the stack of NQ kinds stays in registers.
#pragma once
#include "gb_cut.cuh"

namespace gb {

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

// The child evaluator of gb_cut.cuh over the endpoint programs, the samples
// NQ at a time.
template <int NQ> struct DecEval {
    const GbProg& P;
    const GbDec& D;
    template <int N, bool LO>
    __device__ __forceinline__ void exec(const GbSplitPos& SP, const ChildCtx& c, int q0, const int (&off)[N],
                                         double (&v)[GB_DEC_DEPTH][N], int& ops) const {
        dec_exec<N, LO>(P.uops + SP.u0, 0, SP.nu, D, D.tv + c.p * D.tvp + q0 * D.tvk, D.ts + c.p * D.tsp + q0 * D.tsk,
                        D.nd + c.p * D.ndp + q0 * D.ndk, D.hv + c.p * D.hvp + q0 * D.hvk, off, c.r, v, ops);
    }
    __device__ __forceinline__ double lower(const ChildCtx& c, int spi, int& ops) const {
        const int off[1] = {0};
        double v[GB_DEC_DEPTH][1];
        exec<1, true>(P.sps[spi], c, 0, off, v, ops);
        return v[0][0];
    }
    // smallest order key of the samples' upper ends, kinds [k0, k1); a value that is not a number counts as `nan`
    __device__ __forceinline__ unsigned long long samples(const ChildCtx& c, int spi, int k0, int k1,
                                                          unsigned long long nan, int& ops) const {
        const GbSplitPos SP = P.sps[spi];
        unsigned long long key = ~0ull;
        for (int q0 = k0; q0 < k1; q0 += NQ) {
            int off[NQ];
#pragma unroll
            for (int i = 0; i < NQ; i++) off[i] = min(q0 + i, k1 - 1) - q0;
            double v[GB_DEC_DEPTH][NQ];
            exec<NQ, false>(SP, c, q0, off, v, ops);
#pragma unroll
            for (int i = 0; i < NQ; i++) key = min(key, nan_bits(v[0][i]) ? nan : gb_order_key(v[0][i]));
        }
        return key;
    }
    // over the hull tables: no sample (kinds [k0, k1)) of the group is below the key
    __device__ __forceinline__ unsigned long long bound(const ChildCtx& c, int spi, int k0, int k1, int& ops) const {
        return samples(c, spi, k0, k1, 0, ops);
    }
};

}  // namespace gb
