// scanline_axis1.cu -- scanline DP with the truncated linear prior on one label
// axis of up to 256 labels (the general kernel is in scanline.cu).
//
// Bound: a chain of W columns per row, each a few dependent shuffles; rows are
// independent and few (375 rows on 152 SMs), so the time is W times the latency of
// a column.  One warp owns a row and nothing else is on its path: no block barrier,
// E consecutive labels per lane in registers, cost columns copied to shared memory
// kAhead columns early.  Messages are (value, label) pairs in 32-bit registers:
// sources to the left have lower labels and win ties, sources to the right lose
// them, so one compare decides.  Lane steps beyond the truncation are skipped:
// a source g or more labels away never beats the clip (row minimum + lambda g,
// lowest label).
//
// Back-pointers go to global memory and come back in pieces of 4 KB, the next
// piece loading while one lane walks the present one in shared memory.
//
// 450 x 375, 64 labels: 1300 us (general kernel) -> 103 us, 0.2 us a column.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace edp {

constexpr int kAhead = 16;           // cost columns in flight per row
constexpr int kPieceBytes = 4064;    // back-pointers per piece; with 16-byte ends at most 8 x 32 x 16 bytes
constexpr int kPieceCols = 64;

template <int E, bool SUMS>
__global__ void __launch_bounds__(32) scanline_axis1_kernel(ScanArgs A, int steps) {
    // cost columns [kAhead][32 E]; the walk reuses it: 4 KB of pointers, kPieceCols labels
    constexpr int kRing = kAhead * 32 * E, kWalk = 4096 / 4 + kPieceCols;
    __shared__ __align__(16) int sm[kRing > kWalk ? kRing : kWalk];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x, y = blockIdx.x, W = A.W, Q = A.Q, lam = A.lam;
    const int p0 = lane * E, nv = min(E, max(0, Q - p0));  // labels of this lane
    const int dir = SUMS && A.reverse ? -1 : 1, xs = dir < 0 ? W - 1 : 0;
    const size_t row = (size_t)y * W * Q;
    const int *cg = A.C + row + (long long)xs * Q + p0;
    unsigned char *pg = static_cast<unsigned char *>(A.ptr) + (SUMS ? 0 : row + p0);
    int *sg = SUMS ? A.sums + row + (long long)xs * Q + p0 : nullptr;
    const bool pair = Q % 2 == 0;  // two pointers per store

    for (int i = lane; i < kRing; i += 32) sm[i] = kBig;  // lanes past Q keep kBig
    __syncwarp();
    auto request = [&](int x) {
        if (x < W) {
            int *s = sm + (x % kAhead) * 32 * E + p0;
            const int *c = cg + (long long)x * dir * Q;
#pragma unroll
            for (int i = 0; i < E; ++i)
                if (i < nv) cp_async4(s + i, c + i, true);
        }
        cp_async_commit();
    };
    for (int x = 0; x < kAhead - 1; ++x) request(x);

    int S[E];
    for (int x = 0; x < W; ++x) {
        request(x + kAhead - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
        int c[E];
        const int *s = sm + (x % kAhead) * 32 * E + p0;  // copied by this lane itself
        if constexpr (E == 2) {
            const int2 t = *reinterpret_cast<const int2 *>(s);
            c[0] = t.x, c[1] = t.y;
        } else {
#pragma unroll
            for (int i = 0; i < E; i += 4) {
                const int4 t = *reinterpret_cast<const int4 *>(s + i);
                c[i] = t.x, c[i + 1] = t.y, c[i + 2] = t.z, c[i + 3] = t.w;
            }
        }
        if (x == 0) {
#pragma unroll
            for (int i = 0; i < E; ++i) S[i] = c[i];
        } else {
            // row minimum and its lowest label
            int mv = S[0], mi = p0;
#pragma unroll
            for (int i = 1; i < E; ++i)
                if (S[i] < mv) mv = S[i], mi = p0 + i;
            const int lmin = __reduce_min_sync(full, mv);
            const unsigned lq = __reduce_min_sync(full, mv == lmin ? (unsigned)mi : ~0u);
            // sources to the left and to the right, inside the lane
            int fv[E], fi[E], bv[E], bi[E];
            fv[0] = S[0], fi[0] = p0;
#pragma unroll
            for (int i = 1; i < E; ++i) {
                const int t = fv[i - 1] + lam;
                const bool l = t <= S[i];
                fv[i] = l ? t : S[i], fi[i] = l ? fi[i - 1] : p0 + i;
            }
            bv[E - 1] = S[E - 1], bi[E - 1] = p0 + E - 1;
#pragma unroll
            for (int i = E - 2; i >= 0; --i) {
                const int t = bv[i + 1] + lam;
                const bool l = t < S[i];
                bv[i] = l ? t : S[i], bi[i] = l ? bi[i + 1] : p0 + i;
            }
            // and over lanes: the best at the last (first) label of this lane's reach
            int av = fv[E - 1], ai = fi[E - 1], dv = bv[0], di = bi[0];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                if (k >= steps) break;
                const int d = 1 << k, w = lam * E * d;
                const int tv = __shfl_up_sync(full, av, d) + w, ti = __shfl_up_sync(full, ai, d);
                const int uv = __shfl_down_sync(full, dv, d) + w, ui = __shfl_down_sync(full, di, d);
                if (lane >= d && tv <= av) av = tv, ai = ti;
                if (lane + d < 32 && uv < dv) dv = uv, di = ui;
            }
            int ev = __shfl_up_sync(full, av, 1), ei = __shfl_up_sync(full, ai, 1);
            int gv = __shfl_down_sync(full, dv, 1), gi = __shfl_down_sync(full, di, 1);
            if (lane == 0) ev = kBig;
            if (lane == 31) gv = kBig;
            const int clip = lmin + A.capv;
            unsigned char o[E];
#pragma unroll
            for (int i = 0; i < E; ++i) {
                int v = fv[i], q = fi[i];
                const int l = ev + lam * (i + 1), r = gv + lam * (E - i);
                if (l <= v) v = l, q = ei;
                if (bv[i] < v) v = bv[i], q = bi[i];
                if (r < v) v = r, q = gi;
                if (clip < v || (clip == v && (int)lq < q)) v = clip, q = (int)lq;
                o[i] = (unsigned char)q;
                S[i] = i < nv ? c[i] + v : kBig;
            }
            if constexpr (!SUMS) {
                unsigned char *p = pg + (size_t)x * Q;
                if (pair) {
#pragma unroll
                    for (int i = 0; i < E; i += 2)
                        if (i < nv) *reinterpret_cast<uchar2 *>(p + i) = make_uchar2(o[i], o[i + 1]);
                } else {
#pragma unroll
                    for (int i = 0; i < E; ++i)
                        if (i < nv) p[i] = o[i];
                }
            }
        }
        if constexpr (SUMS) {
            int *p = sg + (long long)x * dir * Q;
#pragma unroll
            for (int i = 0; i < E; ++i)
                if (i < nv) p[i] = S[i];
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if constexpr (!SUMS) {
        // ---- argmin of S(W-1), lowest label on ties ----
        int mv = S[0], mi = p0;
#pragma unroll
        for (int i = 1; i < E; ++i)
            if (S[i] < mv) mv = S[i], mi = p0 + i;
        const int kv = __reduce_min_sync(full, mv);
        int lab = (int)__reduce_min_sync(full, mv == kv ? (unsigned)mi : ~0u);
        if (lab >= Q) lab = 0;
        int *out = A.labels + (size_t)y * W;
        if (lane == 0) {
            if (A.row_energy) A.row_energy[y] = kv;
            out[W - 1] = lab;
        }
        // ---- backward recovery: pointers of columns [x0, x1), last piece first ----
        unsigned char *sp = reinterpret_cast<unsigned char *>(sm);
        int *sl = sm + 4096 / 4;
        const int K = min(kPieceCols, max(1, kPieceBytes / Q));
        const unsigned char *base = static_cast<const unsigned char *>(A.ptr);
        uint4 r[8];
        auto load = [&](int x1) {
            const int x0 = max(1, x1 - K);
            const size_t b = (row + (size_t)x0 * Q) & ~(size_t)15, e = row + (size_t)x1 * Q;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const size_t o = b + (i * 32 + lane) * 16;
                if (o < e) r[i] = *reinterpret_cast<const uint4 *>(base + o);
            }
        };
        __syncwarp();  // the pointers of all lanes are written; the cost ring is free
        if (W > 1) load(W);
        for (int x1 = W; x1 > 1;) {
            const int x0 = max(1, x1 - K), n = x1 - x0;
            const int skip = (int)((row + (size_t)x0 * Q) & 15), bytes = skip + n * Q;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if ((i * 32 + lane) * 16 < bytes) *reinterpret_cast<uint4 *>(sp + (i * 32 + lane) * 16) = r[i];
            __syncwarp();
            if (x0 > 1) load(x0);
            if (lane == 0) {
                const unsigned char *p = sp + skip + (n - 1) * Q;
                for (int x = n - 1; x >= 0; --x, p -= Q) {
                    lab = p[lab];
                    if (lab >= Q) lab = 0;  // unreachable for in-range sums; keeps reads in bounds
                    sl[x] = lab;
                }
            }
            __syncwarp();
            for (int x = lane; x < n; x += 32) out[x0 - 1 + x] = sl[x];
            __syncwarp();
            x1 = x0;
        }
    }
}

int launch_scanline_axis1(const ScanArgs &a, cudaStream_t st) {
    const int E = a.Q <= 64 ? 2 : a.Q <= 128 ? 4 : 8;
    // lane steps that reach every source nearer than g labels
    const long long lanes = a.g <= 1 ? 0 : std::min(31LL, (a.g - 1LL + E - 1) / E);
    int steps = 0;
    while ((1 << steps) < lanes) ++steps;
    auto run = [&](auto k) { k<<<a.H, 32, 0, st>>>(a, steps); };
    if (a.no_ptr) {
        if (E == 2) run(scanline_axis1_kernel<2, true>);
        else if (E == 4) run(scanline_axis1_kernel<4, true>);
        else run(scanline_axis1_kernel<8, true>);
    } else {
        if (E == 2) run(scanline_axis1_kernel<2, false>);
        else if (E == 4) run(scanline_axis1_kernel<4, false>);
        else run(scanline_axis1_kernel<8, false>);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

}  // namespace edp
