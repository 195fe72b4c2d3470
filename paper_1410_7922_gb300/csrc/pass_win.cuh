// pass_win.cuh -- the scan pass of EDP on per-pixel label boxes (two label
// axes, linear prior) in the frame of pass_line2.cuh: same rows, bands, copy
// warps and hand-offs, one compute warp per row.
//
// Every pixel x keeps only the N x N labels of its box B(x) (origin lo(x), from
// a proposed centre clamped into the label space); costs, messages and sums
// are in the coordinates of the pixel's own box.  A message from x to a
// neighbour x' is the exact min-convolution between the two boxes,
//     m(v) = min_{u in B(x)} floor(S(x, u) / 2) + V(u, v),  v in B(x'),
// per label axis as in Sec. 3.2: the sweeps (Eq. L_dec3, Eq. L_dec5) along the
// source box's line give the L1 distance transform D at every source
// position; a target coordinate beyond the source range takes D at the nearest
// source end plus lambda times the distance.  The per-axis clip follows each
// axis; the joint clip (box minimum + lambda f(g), Eq. derivation1) the last.
//
// Each line of N labels is cut into S segments; lane k * N + l holds segment k
// of line l of both vectors.  The result is stored at the target's
// coordinates: position u goes to u - d, d the displacement of the target's
// box; the lanes at the line's ends fill what the source does not reach (a
// distance of g labels or more ends at the clip value).  So
// equal boxes (d = 0, the common case) cost nothing extra.  No barrier: the
// warp exchanges through shared memory between __syncwarp's.
#pragma once
#include "pass_line2.cuh"

namespace edp {
namespace line2 {

// first position of segment k: the first nf segments hold e labels, the rest e - 1
__device__ __forceinline__ int box_pos(int k, int e, int nf) { return k * (e - 1) + min(k, nf); }

// distance transform of one vector's line segment, E labels per lane, n valid
// (the others kBig), all carries (S <= 3)
template <int N, int S, int E>
__device__ __forceinline__ void box_dt(int (&h)[E], const int k, const int n, const int p, const int lam) {
    int f[E], b[E];
    f[0] = h[0];
    b[E - 1] = h[E - 1];
#pragma unroll
    for (int i = 1; i < E; ++i) {
        f[i] = __viaddmin_s32(f[i - 1], lam, h[i]);
        b[E - 1 - i] = __viaddmin_s32(b[E - i], lam, h[E - 1 - i]);
    }
    if constexpr (S > 1) {
        constexpr int nf = N - S * (E - 1);  // segments of E labels
        const int F = f[E - 1], Bv = b[0];
        int cf = kBig, cb = kBig;
#pragma unroll
        for (int d = 1; d < S; ++d) {
            const int uf = __shfl_up_sync(kFull, F, d * N), ub = __shfl_down_sync(kFull, Bv, d * N);
            if (k >= d) cf = min(cf, uf + lam * (p - box_pos(k - d, E, nf) - E + 1));
            if (k + d < S) cb = min(cb, ub + lam * (box_pos(k + d, E, nf) - p - E + 1));
        }
#pragma unroll
        for (int i = 0; i < E; ++i) {
            f[i] = __viaddmin_s32(cf, lam * i, f[i]);
            b[i] = __viaddmin_s32(cb, lam * (E - 1 - i), b[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < E; ++i) h[i] = min(f[i], b[i]);
    (void)n;
}

// One vector's line after its transform: position p + i of the source line to
// target position p + i - d through st(position, value), with clip cl; the end
// lanes fill the target positions beyond the source.
template <int N, int E, typename St>
__device__ __forceinline__ void box_store(const int (&h)[E], const bool on, const int p, const int n, const int d,
                                          const int lam, const int g, const int cl, St &&st) {
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const int t = p + i - d;
        if (on && i < n && (unsigned)t < (unsigned)N) st(t, min(h[i], cl));
    }
    if (__builtin_expect(d > 0, 0)) {  // past the source's last label
        const int last = E > 1 && n < E ? h[E > 1 ? E - 2 : 0] : h[E - 1];
        if (on && p + n == N)
            for (int t = max(N - d, 0); t < N; ++t) st(t, min(last + lam * min(t + d - (N - 1), g), cl));
    }
    if (__builtin_expect(d < 0, 0)) {  // before its first
        if (on && p == 0)
            for (int t = 0; t < min(-d, N); ++t) st(t, min(h[0] + lam * min(-t - d, g), cl));
    }
}

// The column loop of a row's compute warp.
template <int N, int S, bool FIN, bool PA>
__device__ __forceinline__ void win_row(EDP_ROW_ARGS) {
    constexpr int E = (N + S - 1) / S, nf = N - S * (E - 1), hN = (N - 1) / 2;
    const int W = A.W, Q = A.Q, y = w.y, lane = w.lane;
    const unsigned vbytes = 4u * (unsigned)A.Qm, stb = 4u * (unsigned)stage_ints(A.Qm);
    const unsigned omc = vbytes + 16, omd = 2 * vbytes + 16, omb = 3 * vbytes + 16;
    const unsigned xa_sum = 2 * xa0 + vbytes, xb_sum = 2 * xb0 + vbytes;
    const unsigned ta = xb0 + 2 * vbytes, tb = ta + vbytes;  // working vectors
    const unsigned send = 8u * (unsigned)A.nbuf;
    // lane -> segment k of line l
    const int k = lane / N, l = lane - k * N;
    const bool on = k < S;
    const int p = on ? box_pos(k, E, nf) : 0, n = on ? (k < nf ? E : E - 1) : 0;
    const int r1 = ((k + 1) % S) * N + l, r2 = ((k + 2) % S) * N + l;  // the line's other lanes
    auto line_min = [&](int m) {
        if constexpr (S > 1) {
            const int m1 = __shfl_sync(kFull, m, r1 & 31), m2 = S > 2 ? __shfl_sync(kFull, m, r2 & 31) : m;
            m = __vimin3_s32(m, m1, m2);
        }
        return m;
    };
    const unsigned o0 = on ? 4u * (unsigned)(N * l + p) : 0u;  // phase 0: labels of row l, from p
    const unsigned o1 = on ? 4u * (unsigned)(l + N * p) : 0u;  // phase 1: labels of column l, from p
    const int lam = A.lam, cap = A.capv, g = A.g;
    const int step = w.incx ? 1 : -1;
    const int x0 = w.incx ? 0 : W - 1;
    const int *cen = A.centre + 2 * ((size_t)y * W + x0);  // centres of this row, from the next column on
    const int *cen_n = A.centre + 2 * ((size_t)(w.has_next ? (w.incy ? y + 1 : y - 1) : y) * W + x0);
    auto origin = [&](int c, int Qr) { return min(max(c, hN), Qr - 1 - hN) - hN; };
    const int Q0w = A.Q0w, Q1w = A.Q1w;
    // box origins: of this pixel, the next one of the row, the same column of
    // the next row
    int lo0 = origin(__ldg(cen), Q0w), lo1 = origin(__ldg(cen + 1), Q1w);
    int c2[4] = {0, 0, __ldg(cen_n), __ldg(cen_n + 1)};
    if (W > 1) {
        c2[0] = __ldg(cen + 2 * step);
        c2[1] = __ldg(cen + 2 * step + 1);
    }
    unsigned sta = st0, sto = 0, stn = nx, sph = 0, par = 0;
    unsigned csh = (unsigned)((((size_t)y * W + x0) * Q) & 3);
    const unsigned dcs = (unsigned)((w.incx ? Q : -Q) & 3);
    unsigned xma = zs, xa = xa0 + vbytes, xb = xb0;
#pragma unroll 1
    for (int xs = 0; xs < W; ++xs) {
        const bool nxt = xs + 1 < W;
        const int la0 = nxt ? origin(c2[0], Q0w) : lo0, la1 = nxt ? origin(c2[1], Q1w) : lo1;
        const int lb0 = w.has_next ? origin(c2[2], Q0w) : lo0, lb1 = w.has_next ? origin(c2[3], Q1w) : lo1;
        // the next column's centres, a column ahead of their use
        cen += 2 * step;
        cen_n += 2 * step;
        if (xs + 2 < W) {
            c2[0] = __ldg(cen + 2 * step);
            c2[1] = __ldg(cen + 2 * step + 1);
        }
        if (nxt) {
            c2[2] = __ldg(cen_n);
            c2[3] = __ldg(cen_n + 1);
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
        const int da0 = la0 - lo0, da1 = la1 - lo1, db0 = lb0 - lo0, db1 = lb1 - lo1;
        unsigned xmc = w.read_c && nxt ? sta + omc : zs, xmd = w.d_ok ? sta + omd : zs;
        // old messages no pass has written yet come from sums that are still
        // zero: M(0) between the boxes, zero where the boxes are equal (the c
        // neighbour is the next pixel of the row, the d neighbour the same
        // column of the next row); into the unused part of the stage
        auto m0 = [&](unsigned dst, int e0, int e1) {
            for (int q = lane; q < N * N; q += 32) {
                const int q1 = q / N, q0 = q - q1 * N;
                // distances beyond g are clipped anyway (and must not overflow)
                const int u0 = min(g, max(0, max(e0 - q0, q0 - e0 - (N - 1))));
                const int u1 = min(g, max(0, max(e1 - q1, q1 - e1 - (N - 1))));
                sts(dst + 4u * (unsigned)q, PA ? min(lam * u0, cap) + min(lam * u1, cap) : min(lam * (u0 + u1), cap));
            }
            __syncwarp();
        };
        if (!w.read_c && nxt && (da0 | da1) != 0) {
            xmc = sta + omc;
            m0(xmc, da0, da1);
        }
        if (!A.read_d && w.has_next && (db0 | db1) != 0) {
            xmd = sta + omd;
            m0(xmd, db0, db1);
        }
        // ---- phase 0: halved sums of the own box, sweeps along axis 0 ----
        const unsigned xc = sta + 4 * csh + o0, xm = w.r > 0 ? sta + omb + o0 : zs + o0;
        int ha[E], hb[E];
        int ma = kBig, mb = kBig, sv = 0x7fffffff, sq = 0x7fffffff;
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int mc = lds(xmc + o0 + 4 * i), md = lds(xmd + o0 + 4 * i);
            const int t = lds(xc + 4 * i) + lds(xma + o0 + 4 * i) + lds(xm + 4 * i);
            ha[i] = floor_half(t + md - mc);
            hb[i] = floor_half(t + mc - md);
            if (FIN) {
                const int so = t + mc + md;
                if (i < n && so < sv) {
                    sv = so;
                    sq = N * l + p + i;
                }
            }
            if (i >= n) ha[i] = hb[i] = kBig;
            ma = min(ma, ha[i]);
            mb = min(mb, hb[i]);
        }
        int ca = kBig, cb = kBig;  // clips of this axis, then of the last one
        int ga = kBig, gb = kBig;
        if (PA) {
            ca = line_min(ma) + cap;
            cb = line_min(mb) + cap;
        } else {
            ga = __reduce_min_sync(kFull, ma) + cap;
            gb = __reduce_min_sync(kFull, mb) + cap;
        }
        box_dt<N, S, E>(ha, k, n, p, lam);
        box_dt<N, S, E>(hb, k, n, p, lam);
        // result to a working vector or a message: position t of this line, t times st bytes from dst
        auto to_smem = [](unsigned dst, unsigned st) {
            return [=](int t, int v) { sts(dst + st * (unsigned)t, v); };
        };
        box_store<N, E>(ha, on, p, n, da0, lam, g, ca, to_smem(ta + 4u * (unsigned)(N * l), 4u));
        box_store<N, E>(hb, on, p, n, db0, lam, g, cb, to_smem(tb + 4u * (unsigned)(N * l), 4u));
        if (FIN) {
            const int v = __reduce_min_sync(kFull, sv);
            const int q = __reduce_min_sync(kFull, sv == v ? sq : 0x7fffffff);
            if (lane == 0)
                A.labels[(size_t)y * W + (w.incx ? xs : W - 1 - xs)] = lo0 + q % N + Q0w * (lo1 + q / N);
        }
        __syncwarp();
        mbar_arrive_if(lane == 0, bars + kEmptyB + sto);  // the column's inputs have been read
        // ---- phase 1: sweeps along axis 1 of the target's axis-0 columns ----
        ma = mb = kBig;
#pragma unroll
        for (int i = 0; i < E; ++i) {
            ha[i] = lds(ta + o1 + 4 * N * (i < n ? i : 0));
            hb[i] = lds(tb + o1 + 4 * N * (i < n ? i : 0));
            if (i >= n) ha[i] = hb[i] = kBig;
            ma = min(ma, ha[i]);
            mb = min(mb, hb[i]);
        }
        if (PA) {
            ga = line_min(ma) + cap;
            gb = line_min(mb) + cap;
        }
        box_dt<N, S, E>(ha, k, n, p, lam);
        box_dt<N, S, E>(hb, k, n, p, lam);
        box_store<N, E>(ha, on, p, n, da1, lam, g, ga, to_smem(xa + 4u * (unsigned)l, 4u * N));
        box_store<N, E>(hb, on, p, n, db1, lam, g, gb, to_smem((w.to_mbox ? stn : xb) + 4u * (unsigned)l, 4u * N));
        if (__builtin_expect(w.recs != nullptr, 0)) {
            const int s = w.col0 + xs, tag = A.tag0 + s;
            int2 *const rec = w.recs + (size_t)(s % A.ring) * A.Qm + l;
            box_store<N, E>(hb, on, p, n, db1, lam, g, gb, [&](int t, int v) { st_rec(rec + N * t, v, tag); });
        }
        __syncwarp();
        mbar_arrive_if(lane == 0, bars + kOutB + par);
        mbar_arrive_if(lane == 0 && w.to_mbox, nx_ready + sto);
        lo0 = la0;
        lo1 = la1;
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

template <int N, int S>
struct WinBuild {
    static constexpr int threads = 640;  // four rows a block
    static constexpr int extra = 2;
    template <bool FIN, bool PA, bool FUSED>
    static __device__ __forceinline__ void row(EDP_ROW_ARGS) {
        win_row<N, S, FIN, PA>(A, w, zs, st0, xa0, xb0, bars, nx, nx_ready, wmin, wkey, bad, s_abort);
    }
};

}  // namespace line2
}  // namespace edp
