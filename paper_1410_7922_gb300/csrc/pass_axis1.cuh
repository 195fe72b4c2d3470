// pass_axis1.cuh -- EDP scan pass for one label axis (up to 256 labels) in the
// frame of pass_line2.cuh: same rows, bands, copy warps and hand-offs, one
// compute warp per row.
//
// The warp's lower 16 lanes hold the vector S_a, its upper 16 lanes S_b, E
// consecutive labels each (E = 2, 4, 8, 16), so both min searches are the same
// instructions: a lane reads its labels of C, m_a, m_b, m_c, m_d with 16-byte
// loads (m_c and m_d swapped in the upper half: S_b takes them with opposite
// signs), halves the sum of Eq. DP_2D_base, sweeps its own labels (Eq. L_dec3,
// Eq. L_dec5), takes the carries of kc lanes on each side (farther labels cost
// at least the clip value), clips (Eq. derivation1) and stores its labels to X_a
// or to the stage of the row below.  No barrier: the message into the next
// column goes through shared memory of the same warp.
//
// What bounds a pass is this column step, a chain of about 120 instructions.
// (The warp-per-row kernel of pass_r1.cuh, both vectors in every lane and its own
// copies and hand-off words, issues about 356.)
#pragma once
#include "pass_line2.cuh"

namespace edp {
namespace line2 {

// E consecutive ints at a shared address aligned to their size (16 bytes at most)
template <int E>
__device__ __forceinline__ void lds_vec(unsigned a, int (&v)[E]) {
    if constexpr (E == 2) {
        asm volatile("ld.shared.v2.s32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(a));
    } else {
#pragma unroll
        for (int i = 0; i < E; i += 4)
            asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(v[i]), "=r"(v[i + 1]), "=r"(v[i + 2]), "=r"(v[i + 3])
                         : "r"(a + 4 * i));
    }
}
template <int E>
__device__ __forceinline__ void sts_vec(unsigned a, const int (&v)[E]) {
    if constexpr (E == 2) {
        asm volatile("st.shared.v2.s32 [%0], {%1, %2};" ::"r"(a), "r"(v[0]), "r"(v[1]) : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < E; i += 4)
            asm volatile("st.shared.v4.s32 [%0], {%1, %2, %3, %4};" ::"r"(a + 4 * i), "r"(v[i]), "r"(v[i + 1]),
                         "r"(v[i + 2]), "r"(v[i + 3])
                         : "memory");
    }
}

// The column loop of a row's compute warp.  QUAD: the truncated quadratic prior
// (l1 = 2).  VC: the pixels' labels of C start 16-byte aligned (Q a multiple of 4).
template <int E, bool QUAD, bool VC, bool FIN>
__device__ __forceinline__ void axis1_row(EDP_ROW_ARGS) {
    const int W = A.W, Q = A.Q, y = w.y, lane = w.lane, g = A.g;
    const unsigned vbytes = 4u * (unsigned)A.Qm, stb = 4u * (unsigned)stage_ints(A.Qm);
    const unsigned omc = vbytes + 16, omd = 2 * vbytes + 16, omb = 3 * vbytes + 16;
    const bool vb = lane >= 16;
    const int j = lane & 15, q0 = j * E;
    const bool on = q0 < Q;                        // the lane holds labels
    const unsigned o = on ? 4u * (unsigned)q0 : 0u;
    const int nq = max(0, min(E, Q - q0));         // how many
    const bool whole = nq == E;
    const unsigned xa_sum = 2 * xa0 + vbytes, xb_sum = 2 * xb0 + vbytes;
    const unsigned tmp = xb0 + 2 * vbytes + (vb ? vbytes : 0u);  // QUAD: this vector's working copy
    const unsigned send = 8u * (unsigned)A.nbuf;
    const int kc = A.seg[0].kc;
    unsigned sta = st0, sto = 0, stn = nx, sph = 0, par = 0;
    unsigned csh = VC ? 0u : (unsigned)((((size_t)y * W + (w.incx ? 0 : W - 1)) * Q) & 3);
    const unsigned dcs = VC ? 0u : (unsigned)((w.incx ? Q : -Q) & 3);
    unsigned xma = zs, xa = xa0 + vbytes, xb = xb0;
    int lam = A.lam, cap = A.capv;
#pragma unroll 1
    for (int xs = 0; xs < W; ++xs) {
        if (__builtin_expect(A.wh != nullptr, 0)) {  // per-edge multipliers of this vector's outgoing edge
            const int x = w.incx ? xs : W - 1 - xs;
            int wt = 1;
            if (!vb && xs + 1 < W) wt = __ldg(A.wh + (size_t)y * W + (w.incx ? x : x - 1));
            if (vb && w.has_next) wt = __ldg(A.wv + (size_t)(w.incy ? y : y - 1) * W + x);
            lam = A.lam * wt;
            cap = A.capv * wt;
        }
        bool ok = mbar_try(bars + kLoadB + sto, sph);
        ok = mbar_try(bars + kReadyB + sto, sph) && ok;
        if (__builtin_expect(!__all_sync(kFull, ok), 0)) {
            ok = mbar_wait(bars + kLoadB + sto, sph, A.spin_limit, s_abort) &&
                 mbar_wait(bars + kReadyB + sto, sph, A.spin_limit, s_abort);
            if (!__all_sync(kFull, ok)) {
                if (lane == 0) timed_out(A.status, s_abort);
                break;
            }
        }
        const unsigned xmc = (w.read_c && xs + 1 < W ? sta + omc : zs) + o, xmd = (w.d_ok ? sta + omd : zs) + o;
        int cv[E], ma[E], mb[E], mp[E], mm[E];  // + C + m_a + m_b, + mp - mm
        if constexpr (VC) {
            lds_vec<E>(sta + o, cv);
        } else {
#pragma unroll
            for (int i = 0; i < E; ++i) cv[i] = lds(sta + 4 * csh + o + 4 * i);
        }
        lds_vec<E>(xma + o, ma);
        lds_vec<E>((w.r > 0 ? sta + omb : zs) + o, mb);
        lds_vec<E>(vb ? xmc : xmd, mp);
        lds_vec<E>(vb ? xmd : xmc, mm);
        int h[E];
        int lm = kBig, sv = 0x7fffffff, sq = 0x7fffffff;
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int t = cv[i] + ma[i] + mb[i];
            h[i] = floor_half(t + mp[i] - mm[i]);
            if (FIN) {
                const int so = t + mp[i] + mm[i];
                if (i < nq && so < sv) {
                    sv = so;
                    sq = q0 + i;
                }
            }
            if (i >= nq) h[i] = kBig;
            lm = min(lm, h[i]);
        }
        const int ga = __reduce_min_sync(kFull, vb ? kBig : lm), gb = __reduce_min_sync(kFull, vb ? lm : kBig);
        const int cl = (vb ? gb : ga) + cap;
        if constexpr (QUAD) {
            // taps |d| < g from the working copy (farther sources cost at least the clip)
            if (on) {
                if (whole)
                    sts_vec<E>(tmp + o, h);
                else
#pragma unroll
                    for (int i = 0; i < E; ++i)
                        if (i < nq) sts(tmp + o + 4 * i, h[i]);
            }
            __syncwarp();
            const int dmax = min(g, Q);
            for (int d = 1; d < dmax; ++d) {
                const int wd = lam * d * d;
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    const int q = q0 + i;
                    const int up = lds(tmp + 4u * (unsigned)min(q + d, Q - 1)), dn = lds(tmp + 4u * (unsigned)max(min(q, Q - 1) - d, 0));
                    if (q + d < Q) h[i] = __viaddmin_s32(up, wd, h[i]);
                    if (q - d >= 0) h[i] = __viaddmin_s32(dn, wd, h[i]);
                }
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < E; ++i) h[i] = min(h[i], cl);
        } else {
            int f[E], b[E];
            f[0] = h[0];
            b[E - 1] = h[E - 1];
#pragma unroll
            for (int i = 1; i < E; ++i) {
                f[i] = __viaddmin_s32(f[i - 1], lam, h[i]);
                b[E - 1 - i] = __viaddmin_s32(b[E - i], lam, h[E - 1 - i]);
            }
            const int F = f[E - 1], B = b[0];
            int cf = __shfl_up_sync(kFull, F, 1, 16), cb = __shfl_down_sync(kFull, B, 1, 16);
            cf = j > 0 ? cf + lam : kBig;
            cb = j < 15 ? cb + lam : kBig;
            if (__builtin_expect(kc > 1, 0)) {
#pragma unroll 1
                for (int d = 2; d <= kc; ++d) {
                    const int uf = __shfl_up_sync(kFull, F, d, 16), ub = __shfl_down_sync(kFull, B, d, 16);
                    const int gap = lam * ((d - 1) * E + 1);
                    if (j >= d) cf = min(cf, uf + gap);
                    if (j + d < 16) cb = min(cb, ub + gap);
                }
            }
#pragma unroll
            for (int i = 0; i < E; ++i) {
                f[i] = __viaddmin_s32(cf, lam * i, f[i]);
                b[i] = __viaddmin_s32(cb, lam * (E - 1 - i), b[i]);
                h[i] = __vimin3_s32(f[i], b[i], cl);
            }
        }
        if (FIN) {
            // (both halves hold the same sums)
            const int v = __reduce_min_sync(kFull, sv);
            const int q = __reduce_min_sync(kFull, sv == v ? sq : 0x7fffffff);
            if (lane == 0) A.labels[(size_t)y * W + (w.incx ? xs : W - 1 - xs)] = q;
        }
        const unsigned dst = (vb ? (w.to_mbox ? stn : xb) : xa) + o;
        if (whole) {
            sts_vec<E>(dst, h);
        } else {
#pragma unroll
            for (int i = 0; i < E; ++i)
                if (i < nq) sts(dst + 4 * i, h[i]);
        }
        if (__builtin_expect(w.recs != nullptr, 0)) {
            const int s = w.col0 + xs, tag = A.tag0 + s;
            int2 *const rec = w.recs + (size_t)(s % A.ring) * A.Qm + q0;
            if (vb) {
#pragma unroll
                for (int i = 0; i < E; ++i)
                    if (i < nq) st_rec(rec + i, h[i], tag);
            }
        }
        __syncwarp();
        // the column's inputs have been read, its outputs written
        mbar_arrive_if(lane == 0, bars + kEmptyB + sto);
        mbar_arrive_if(lane == 0, bars + kOutB + par);
        mbar_arrive_if(lane == 0 && w.to_mbox, nx_ready + sto);
        par ^= 8;
        xma = xa;
        xa = xa_sum - xa;
        xb = xb_sum - xb;
        csh = (csh + dcs) & 3;
        sto += 8;
        const bool wrap = sto == send;
        sta = wrap ? st0 : sta + stb;
        stn = wrap ? nx : stn + stb;
        sph ^= wrap ? 1u : 0u;
        sto = wrap ? 0u : sto;
    }
}

template <int E, bool QUAD, bool VC>
struct Axis1Build {
    static constexpr int threads = 640;  // four rows a block
    static constexpr int extra = QUAD ? 2 : 0;
    template <bool FIN, bool PA, bool FUSED>
    static __device__ __forceinline__ void row(EDP_ROW_ARGS) {
        axis1_row<E, QUAD, VC, FIN>(A, w, zs, st0, xa0, xb0, bars, nx, nx_ready, wmin, wkey, bad, s_abort);
    }
};

}  // namespace line2
}  // namespace edp
