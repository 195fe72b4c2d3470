// pass_line2.cuh -- EDP scan pass for label spaces of two or three axes, each
// label line shared by several lanes of a warp.
//
// Same messages, flags and pass schedule as pass_team.cuh (M[k] at pixel x
// holds m_k(x) = M(floor(S_k(x_k) / 2)); a pass updates the sums a, b from
// m_a, m_b of this pass and m_c, m_d of earlier ones).  A pass is a wavefront,
// so what bounds it is the time of one column step of one row; this kernel
// spreads a row over as many warps as its labels fill, keeps every memory
// access of the step in shared memory, and moves all global data with bulk
// asynchronous copies issued by warps that do nothing else.
//
// Roles.  A block holds NT teams (NT consecutive rows, one band).  A team has
// T compute warps and four copy warps (one lane each):
//   stage  copies C, m_c, m_d of the columns ahead into a ring of nst stages;
//   above  (first row of a band) copies m_b of the columns the row above has
//          published into the same stages;
//   out 0, out 1  (even / odd columns) copy the finished m_a and m_b to the
//          message arrays and, for the last row of a band, publish the column.
// They meet in mbarriers: load[stage] completes when a column's copies (C, m_c,
// m_d; m_b of `above`) have landed, ready[stage] when its output buffers have
// been shipped and, below another team, that team's warps have written m_b;
// empty[stage] when every compute warp has read the inputs; outf[p] when every
// compute warp has written its outputs.
//
// A column step of the compute warps:
//   phase 0   the halved sums of Eq. DP_2D_base on lines of axis 0, both
//             vectors in the same lane (the five inputs are read once), the
//             min search along axis 0, results to X_a (next buffer) and X_b;
//   barrier;  phases 1 .. R-1: the same along axes 1, 2 in place, again both
//             vectors in the same lane (a barrier between them); the last one
//             leaves m_a in X_a and m_b in the stage of the row below (or in
//             X_b, shipped by `out`);
//   barrier.
// The min search is separable, so the order of the axes changes no value.
//
// A line of L labels is cut into S segments of e = ceil(L / S) or e - 1 labels;
// lane k * lpw + l of a warp holds segment k of the warp's line l
// (lpw = 32 / S lines per warp), so neighbouring lanes read neighbouring lines
// (odd strides: distinct banks; 65 labels in 5 segments of 13, 33 in 3 of 11 or
// 8 of 4-5 put all lanes on distinct banks, 65 in 8 segments would not: its
// segments 32 labels apart share a bank).  Lanes without a line or a segment
// repeat another one, stores included, so nothing is predicated.  Per
// segment the forward and the backward sweep (Eq. L_dec3, Eq. L_dec5) run on the
// lane's own labels; the values at the segment's ends travel by one shuffle per
// direction, kc segments far, and complete the labels they can still improve:
// a source g or more labels away costs at least the clip value applied
// afterwards (Sec. 3.1), so nothing beyond is needed.
//
// A column step is a few hundred instructions in a row, run by a few warps per
// scheduler, so what costs is not the arithmetic but every taken branch and
// every load from the parameter block (tens of cycles each).  Hence one build
// per label space of the repository's workloads (all sizes constants) and a
// few for any other (up to E labels per lane), the truncation mode and the
// last pass as separate copies of the column loop.  (A build that picked the
// cut at run time took 2.2 us a column at 33 x 33 labels.)
//
// Between bands, m_b goes through a ring of `ring` columns per band in global
// memory that stays in L2, in one of two forms:
//   records (A.rec, up to kMaxRecQ labels): the compute warps of a band's last
//           row store {value, tag} words themselves, and the `above` warp of
//           the next band polls them into its stage -- a matching tag carries
//           its value, so no fence, flag or copy completion is on the path.
//           The next column's words are requested before this one's are taken
//           (0.70 -> 0.55 us a column at 64 labels);
//   copies  (longer vectors, twice whose bytes would load L2): the `out` warp
//           copies X_b to the ring (or, in the passes that keep m_b, to the
//           message array anyway) and publishes the column when the copy has
//           completed (release at GPU scope); `above` acquires that and copies.
// A ring slot is written again once the consumer has counted its column (cons).
// The halves of a pair count in a word each, since nothing orders the stores of their
// two blocks; the larger count holds.
// (33 x 33 labels, 320x240: 3.7 ms a solve with copies.  A column step of 0.9 us in
// a row alone, 1.45 us with the rows coupled; 4 us a hand-off, and 6 to 7.7 us from
// a block's two rows to the next two.)
//
// Work items.  A launch holds one pass, or two that share the vertical
// direction (A.pair: P1 then P2, or P3 then P4) as items (half, band) claimed
// in order.  Row y of the second half needs row y of the first half complete
// (its m_a are this half's m_c) and its own half's row above, both claimed
// earlier, so a block never waits for an item that nobody runs; the second
// half starts without draining the first.
#pragma once
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace edp {
namespace line2 {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kCopyWarps = 4;     // stage, above, out 0, out 1
constexpr int kMaxT = 24;         // compute warps of a team
constexpr int kMaxRows = 8;       // teams of a block
constexpr int kMaxThreads = 896;  // of a block: 72 registers a thread
constexpr int kMaxStages = 4;
constexpr int kMaxRecQ = 512;     // labels of the record form
// control ints of one team: mbarriers [0, 28), columns issued by `stage` and
// `above` (an aborted item's, [28, 30)), abort flag [30], warp minima [32, 80), warp argmin
// values and labels [80, 128)
constexpr int kCtlInts = 128;
// the planner's bound on the prior weight (sweeps add up to 33 lambda to kBig)
constexpr int kMaxLambda = (1 << 30) / 34;

// a stage: C (and 4 ints of slack for its 16-byte alignment), m_c, m_d, m_b
__host__ __device__ inline size_t stage_ints(int Qm) { return 4 * (size_t)Qm + 4; }
// ints of one team: stages, X_a and X_b (two each), `extra` further vectors,
// control
__host__ __device__ inline size_t team_ints(int Qm, int nst, int extra) {
    return nst * stage_ints(Qm) + (4 + extra) * (size_t)Qm + kCtlInts;
}

__device__ __forceinline__ unsigned saddr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ int lds(unsigned a) {
    int v;
    asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts(unsigned a, int v) { asm volatile("st.shared.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

__device__ __forceinline__ void mbar_init(unsigned b, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(b), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(unsigned b) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(b) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(b) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(unsigned b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned b, unsigned parity) {
    unsigned r;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"(b), "r"(parity)
        : "memory");
    return r != 0;
}
// bounded wait for the completion of a phase; false when it ran out or the
// block is aborting
__device__ __forceinline__ bool mbar_wait(unsigned b, unsigned parity, long long limit, volatile int *s_abort) {
    if (mbar_try(b, parity)) return true;
    for (long long n = 0; n < limit; ++n) {
        if (mbar_try(b, parity)) return true;
        if (*s_abort) return false;
    }
    return false;
}
// bulk copies (16-byte aligned addresses and sizes)
__device__ __forceinline__ void bulk_load(unsigned dst, const int *src, unsigned bytes, unsigned mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}
__device__ __forceinline__ void bulk_store(int *dst, unsigned src, unsigned bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ unsigned ld_acq_gpu(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_rel_gpu(unsigned *p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void add_rel_gpu(unsigned *p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint2 ld_acq_gpu2(const unsigned *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return make_uint2((unsigned)v, (unsigned)(v >> 32));
}
// {value, tag} records: single 64-bit accesses (two of them in one load)
__device__ __forceinline__ void st_rec(int2 *p, int v, int tag) {
    const unsigned long long w = (unsigned long long)(unsigned)v | ((unsigned long long)(unsigned)tag << 32);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ int4 ld_rec2(const int2 *p) {
    unsigned long long a, b;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
    return make_int4((int)(unsigned)a, (int)(a >> 32), (int)(unsigned)b, (int)(b >> 32));
}
__device__ __forceinline__ void st_relaxed_gpu(unsigned *p, unsigned v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// bounded poll of a counter of another block
__device__ __forceinline__ bool wait_count(const unsigned *p, int need, long long limit, volatile int *s_abort,
                                           const int *status) {
    for (long long n = 0; n <= limit; ++n) {
        if ((int)ld_acq_gpu(p) >= need) return true;
        if (*s_abort || ((n & 63) == 63 && *(volatile const int *)status != 0)) return false;
        __nanosleep(20);
    }
    return false;
}
// barriers of the T compute warps of a team; the second also returns the OR
// of pred over them
__device__ __forceinline__ void team_sync(int tm, int T) {
    asm volatile("barrier.sync %0, %1;" ::"r"(tm + 1), "r"(32 * T) : "memory");
}
__device__ __forceinline__ bool team_sync_or(int tm, int T, bool pred) {
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.s32 p, %1, 0;\n\t"
        "barrier.red.or.pred q, %2, %3, p;\n\t"
        "selp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((int)pred), "r"(tm + 1), "r"(32 * T)
        : "memory");
    return r != 0;
}

// one lane's arrival, without a branch
__device__ __forceinline__ void mbar_arrive_if(bool p, unsigned b) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %1, 0;\n\t@q mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(b),
                 "r"((int)p)
                 : "memory");
}

// The cut of one axis: S segments per line, at most E labels each.  L, LINES,
// STRIDE: the axis' sizes where the build fixes them (L = 0: run time).
template <int S_, int E_, int L_ = 0, int LINES_ = 0, int STRIDE_ = 0>
struct Cut {
    static constexpr int S = S_, E = E_, L = L_, lpw = 32 / S_;
    static constexpr bool fixed = L_ > 0;
    static constexpr bool full = L_ == S_ * E_;      // every segment holds E labels
    static constexpr int NF = L_ - S_ * (E_ - 1);    // fixed: segments of E labels
    static_assert(!fixed || (NF >= 1 && NF <= S_), "lines cut into segments of E or E - 1 labels");
    static __device__ __forceinline__ int nlines(const TeamArgs &A, int r) { return fixed ? LINES_ : A.ax[r].nlines; }
    static __device__ __forceinline__ int stride(const TeamArgs &A, int r) { return fixed ? STRIDE_ : A.ax[r].stride; }
    static __device__ __forceinline__ int len(const TeamArgs &A, int r) { return fixed ? L_ : A.ax[r].L; }
    // first position of segment k: the last nf segments hold e labels, the others
    // e - 1 (33 labels in 8 segments start at 0, 4, .. 28: with 4 lines a warp,
    // on distinct banks; the long segment first would put two on one bank)
    static __device__ __forceinline__ int pos(const TeamArgs &A, int r, int k) {
        const int e = fixed ? E_ : A.ax[r].E, nf = fixed ? NF : A.seg[r].nf;
        return k * (e - 1) + max(0, k - (S - nf));
    }
};

// A lane's place on one axis.
struct Seg {
    int k, l;          // segment, line within the warp
    int off;           // linear index of the segment's first label
    int n;             // its labels
    int sl, sr, s2;    // lanes of the segments before, after (cyclic), two after (cyclic)
};
// the lane's place when the warp serves the lines from li0 (lines past the
// last one, and lanes past the last segment, repeat)
template <class C>
__device__ __forceinline__ Seg seg_of(const TeamArgs &A, int r, int li0, int lane) {
    Seg s;
    s.k = min(lane / C::lpw, C::S - 1);
    s.l = lane - (lane / C::lpw) * C::lpw;
    const int nl = C::nlines(A, r), st = C::stride(A, r), L = C::len(A, r);
    const int li = min(li0 + s.l, nl - 1);
    const int p = C::pos(A, r, s.k);
    s.n = C::pos(A, r, s.k + 1) - p;
    s.sl = max(s.k - 1, 0) * C::lpw + s.l;
    s.sr = (s.k + 1) % C::S * C::lpw + s.l;
    s.s2 = (s.k + 2) % C::S * C::lpw + s.l;
    // first label of line li
    int f = li;
    if (st == 1)
        f = li * L;
    else if (li >= st)
        f = (li % st) + (li / st) * st * L;
    s.off = f + p * st;
    return s;
}

// Truncated L1 distance transform and clip of one vector's segment, in place
// (positions n .. E - 1 hold kBig); cl is the clip value.  f, b: the lane's
// own sweeps.  near: carries from one segment, and only labels next to a
// boundary can improve (g <= 4).
template <class C>
__device__ __forceinline__ void seg_dt(const TeamArgs &A, const int r, int (&h)[C::E], const Seg &s, const bool near,
                                       const int lam, const int cl) {
    constexpr int E = C::E, S = C::S;
    int f[E], b[E];
    f[0] = h[0];
    b[E - 1] = h[E - 1];
#pragma unroll
    for (int i = 1; i < E; ++i) {
        f[i] = __viaddmin_s32(f[i - 1], lam, h[i]);
        b[E - 1 - i] = __viaddmin_s32(b[E - i], lam, h[E - 1 - i]);
    }
    if constexpr (S > 1) {
        // carries: cf at position 0 of the segment, cb at position E - 1
        const int F = f[E - 1], B = b[0];
        int cf = __shfl_sync(kFull, F, s.sl), cb = __shfl_sync(kFull, B, s.sr);
        if constexpr (C::full) {
            cf += lam;
            cb += lam;
        } else if constexpr (C::fixed) {
            cf += s.k > S - C::NF ? lam : 0;
            cb += s.k >= S - C::NF ? lam : 0;
        } else {
            cf += lam * (C::pos(A, r, s.k) - C::pos(A, r, s.k - 1) - E + 1);
            cb += lam * (s.n - E + 1);
        }
        cf = s.k > 0 ? cf : kBig;
        cb = s.k < S - 1 ? cb : kBig;
        // labels within 3 of the segment's ends, or all of them
        constexpr int NF = C::fixed && E > 3 ? 3 : E, NB = C::full && E > 3 ? 3 : C::fixed && E > 4 ? 4 : E;
        if (__builtin_expect(!near, 0)) {
            const int kc = A.seg[r].kc;
#pragma unroll 1
            for (int d = 2; d <= kc; ++d) {
                const int uf = __shfl_sync(kFull, F, max(s.k - d, 0) * C::lpw + s.l);
                const int ub = __shfl_sync(kFull, B, min(s.k + d, S - 1) * C::lpw + s.l);
                const int p = C::pos(A, r, s.k);
                if (s.k >= d) cf = min(cf, uf + lam * (p - C::pos(A, r, s.k - d) - E + 1));
                if (s.k + d < S) cb = min(cb, ub + lam * (C::pos(A, r, s.k + d) - p - E + 1));
            }
#pragma unroll
            for (int i = NF; i < E; ++i) f[i] = __viaddmin_s32(cf, lam * i, f[i]);
#pragma unroll
            for (int i = 0; i < E - NB; ++i) b[i] = __viaddmin_s32(cb, lam * (E - 1 - i), b[i]);
        }
#pragma unroll
        for (int i = 0; i < NF; ++i) f[i] = __viaddmin_s32(cf, lam * i, f[i]);
#pragma unroll
        for (int i = E - NB; i < E; ++i) b[i] = __viaddmin_s32(cb, lam * (E - 1 - i), b[i]);
    }
#pragma unroll
    for (int i = 0; i < E; ++i) h[i] = __vimin3_s32(f[i], b[i], cl);
}

// minimum over the line (every lane of the line gets it): windows of lanes
// that grow modulo S (the minimum is idempotent)
template <class C>
__device__ __forceinline__ int line_min(int m, const Seg &s) {
    constexpr int S = C::S;
    if constexpr (S == 2 || S == 4 || S == 8) {
#pragma unroll
        for (int d = C::lpw; d < 32; d <<= 1) m = min(m, __shfl_xor_sync(kFull, m, d));
    } else if constexpr (S == 3) {
        m = __vimin3_s32(m, __shfl_sync(kFull, m, s.sr), __shfl_sync(kFull, m, s.s2));
    } else if constexpr (S == 5) {
        m = min(m, __shfl_sync(kFull, m, s.sr));    // 2 segments
        m = min(m, __shfl_sync(kFull, m, s.s2));    // 4
        m = min(m, __shfl_sync(kFull, m, s.sr));    // all
    } else {
        static_assert(S == 1, "segments per line");
    }
    return m;
}

// The pair cost of Eq. Cost_value of one label (two-axis spaces) from the
// images, as the cost kernels store it.
struct FusedPix {
    int x, y, i0;  // pixel, I0(pixel)
};
__device__ __forceinline__ int fused_cost(const TeamArgs &A, const FusedPix &p, int q0, int q1) {
    const int xs = p.x + A.fv0 + A.ft0 * q0, ys = p.y + A.fv1 + A.ft1 * q1;
    if ((unsigned)xs >= (unsigned)A.W || (unsigned)ys >= (unsigned)A.H) return A.fcmax;
    const int d = abs((int)A.fI1[(size_t)ys * A.fpitch + xs] - p.i0);
    return min(A.fl2 == 1 ? d : d * d, A.fcmax);
}

// Phase 0: sums, halving, min search along axis 0 for both vectors.  C .. mb:
// shared addresses of the inputs' label 0, xa / xb of the outputs'.  ja, jb:
// minima of the halved sums (joint truncation); sv, sq: the marginal's lowest
// value and label (FIN).
struct In0 {
    unsigned C, mc, md, ma, mb, xa, xb;
    int lam_a, lam_b, cap_a, cap_b;
    FusedPix fp;
};
template <class C, bool FIN, bool PA, bool FUSED>
__device__ __forceinline__ void phase0(const TeamArgs &A, const In0 &c, const Seg &s, const bool near, const int fq0,
                                       const int fq1, int &ja, int &jb, int &sv, int &sq) {
    constexpr int E = C::E;
    const unsigned o = 4u * (unsigned)s.off;
    int ha[E], hb[E];
    int ma = kBig, mb = kBig;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const unsigned oi = o + 4 * i;
        int cv;
        if constexpr (FUSED)
            cv = fused_cost(A, c.fp, fq0 + i, fq1);
        else
            cv = lds(c.C + oi);
        const int mc = lds(c.mc + oi), md = lds(c.md + oi);
        const int t = cv + lds(c.ma + oi) + lds(c.mb + oi);
        ha[i] = floor_half(t + md - mc);
        hb[i] = floor_half(t + mc - md);
        const bool maybe = C::full ? false : C::fixed ? i == E - 1 : true;  // past the segment on some lanes
        if (FIN) {
            const int so = t + mc + md;
            if ((!maybe || i < s.n) && so < sv) {
                sv = so;
                sq = s.off + i;
            }
        }
        if (maybe && i >= s.n) ha[i] = hb[i] = kBig;
        ma = min(ma, ha[i]);
        mb = min(mb, hb[i]);
    }
    int ca = kBig, cb = kBig;
    if (PA) {
        ca = line_min<C>(ma, s) + c.cap_a;
        cb = line_min<C>(mb, s) + c.cap_b;
    } else {
        ja = min(ja, ma);
        jb = min(jb, mb);
    }
    seg_dt<C>(A, 0, ha, s, near, c.lam_a, ca);
    seg_dt<C>(A, 0, hb, s, near, c.lam_b, cb);
#pragma unroll
    for (int i = 0; i < E; ++i) {
        if (C::full || (C::fixed && i < E - 1) || i < s.n) {
            sts(c.xa + o + 4 * i, ha[i]);
            sts(c.xb + o + 4 * i, hb[i]);
        }
    }
}

// Where a band's last row leaves m_b as records (p null: it does not).
struct Rec {
    int2 *p;  // the column's slot (label 0)
    int tag;
};

// One line segment of both vectors in a later phase (axis r; two independent
// chains per lane): min search along the axis of the values in X_a and X_b,
// m_a's back to X_a, m_b's to nb; ca, cb: the clip values, or with PA what is
// added to the line's minima.
template <class C, bool PA>
__device__ __forceinline__ void phase_r(const TeamArgs &A, const int r, const Seg &s, const bool near, const In0 &c,
                                        const unsigned nb, const int ca, const int cb, const Rec &rec) {
    constexpr int E = C::E;
    int ha[E], hb[E];
    int ma = kBig, mb = kBig;
    const unsigned st4 = 4u * (unsigned)C::stride(A, r), o = 4u * (unsigned)s.off;
#pragma unroll
    for (int i = 0; i < E; ++i) {
        const bool maybe = C::full ? false : C::fixed ? i == E - 1 : true;
        const unsigned oi = o + (maybe && i >= s.n ? 0u : i * st4);
        ha[i] = lds(c.xa + oi);
        hb[i] = lds(c.xb + oi);
        if (maybe && i >= s.n) ha[i] = hb[i] = kBig;
        ma = min(ma, ha[i]);
        mb = min(mb, hb[i]);
    }
    seg_dt<C>(A, r, ha, s, near, c.lam_a, PA ? line_min<C>(ma, s) + ca : ca);
    seg_dt<C>(A, r, hb, s, near, c.lam_b, PA ? line_min<C>(mb, s) + cb : cb);
#pragma unroll
    for (int i = 0; i < E; ++i) {
        if (C::full || (C::fixed && i < E - 1) || i < s.n) {
            sts(c.xa + o + i * st4, ha[i]);
            sts(nb + o + i * st4, hb[i]);
        }
    }
    if (__builtin_expect(rec.p != nullptr, 0)) {
        int2 *const q = rec.p + s.off;
#pragma unroll
        for (int i = 0; i < E; ++i)
            if (C::full || (C::fixed && i < E - 1) || i < s.n) st_rec(q + i * C::stride(A, r), hb[i], rec.tag);
    }
}

static __device__ __noinline__ void timed_out(int *status, volatile int *s_abort) {
    atomicCAS(status, 0, EDP_ERR_TIMEOUT_CODE);
    *s_abort = 1;
}

// byte offsets of a team's mbarriers
constexpr unsigned kLoadB = 0, kReadyB = 8 * kMaxStages, kEmptyB = 16 * kMaxStages, kOutB = 24 * kMaxStages;
constexpr int kBars = (kOutB + 16) / 8;
static_assert(kBars * 8 <= 112, "mbarriers of a team");

struct Row {
    int r, y, tm, wt, lane;
    bool incx, incy, has_next, to_mbox, read_c, d_ok;
    int2 *recs;  // the band's record ring, where its last row uses one (else null)
    int col0;    // columns of the launch before this half (tags, ring slots)
};

// arguments of a row's column loop: shared addresses of the zero vector, the
// stages, X_a, X_b, the barriers, and of the team below the m_b of its first
// stage and its ready barriers; the joint minima and argmin slots; the team's
// abort flag
#define EDP_ROW_ARGS                                                                                                   \
    const TeamArgs &A, const Row &w, const unsigned zs, const unsigned st0, const unsigned xa0, const unsigned xb0,    \
        const unsigned bars, const unsigned nx, const unsigned nx_ready, int *wmin, int *wkey, int *bad,               \
        volatile int *s_abort
template <class B, bool FIN, bool PA, bool FUSED>
__device__ __forceinline__ void line2_row(EDP_ROW_ARGS);

// A build: the cuts of the axes (C2::S = 0: two axes).
struct NoCut {
    static constexpr int S = 0, E = 1, lpw = 32, L = 1;
    static constexpr bool fixed = true;
    static __device__ __forceinline__ int nlines(const TeamArgs &, int) { return 1; }
};
template <class C0_, class C1_, class C2_, int THREADS = kMaxThreads>
struct Build {
    using C0 = C0_;
    using C1 = C1_;
    using C2 = C2_;
    static constexpr int R = C2_::S > 0 ? 3 : 2;
    static constexpr int threads = THREADS;  // bound of a block (registers)
    static constexpr int extra = 0;          // working vectors of a team beside X_a, X_b
    // labels (0: run time)
    static constexpr int Q = C0_::fixed ? C0_::L * C1_::L * C2_::L : 0;
    template <bool FIN, bool PA, bool FUSED>
    static __device__ __forceinline__ void row(EDP_ROW_ARGS) {
        line2_row<Build, FIN, PA, FUSED>(A, w, zs, st0, xa0, xb0, bars, nx, nx_ready, wmin, wkey, bad, s_abort);
    }
};
// the cuts of a fixed two- or three-axis space
template <int Q0, int Q1, int S0, int E0, int S1, int E1, int THREADS = kMaxThreads>
using Fixed2 = Build<Cut<S0, E0, Q0, Q1, 1>, Cut<S1, E1, Q1, Q0, Q0>, NoCut, THREADS>;
template <int Q0, int Q1, int Q2, int S0, int E0, int S1, int E1, int S2, int E2, int THREADS = kMaxThreads>
using Fixed3 = Build<Cut<S0, E0, Q0, Q1 * Q2, 1>, Cut<S1, E1, Q1, Q0 * Q2, Q0>, Cut<S2, E2, Q2, Q0 * Q1, Q0 * Q1>,
                     THREADS>;

// The column loop of one compute warp.
template <class B, bool FIN, bool PA, bool FUSED>
__device__ __forceinline__ void line2_row(EDP_ROW_ARGS) {
    using C0 = typename B::C0;
    using C1 = typename B::C1;
    using C2 = typename B::C2;
    constexpr int R = B::R;
    using CL = std::conditional_t<R == 3, C2, C1>;
    const int W = A.W, T = A.T, tm = w.tm, wt = w.wt, lane = w.lane, y = w.y;
    const int Q = B::Q ? B::Q : A.Q, Qm = B::Q ? (B::Q + 3) / 4 * 4 : A.Qm;
    const unsigned vbytes = 4u * (unsigned)Qm, stb = 4u * (unsigned)stage_ints(Qm);
    const unsigned omc = vbytes + 16, omd = 2 * vbytes + 16, omb = 3 * vbytes + 16;
    const int n0 = (C0::nlines(A, 0) + C0::lpw - 1) / C0::lpw;  // warp rounds of the phases, per vector
    const int n1 = (C1::nlines(A, 1) + C1::lpw - 1) / C1::lpw, nl = R == 3 ? (CL::nlines(A, 2) + CL::lpw - 1) / CL::lpw : n1;
    const Seg s0 = seg_of<C0>(A, 0, wt * C0::lpw, lane);
    const Seg s1 = seg_of<C1>(A, 1, wt * C1::lpw, lane);
    Seg s2 = s1;
    if constexpr (R == 3) s2 = seg_of<CL>(A, 2, wt * CL::lpw, lane);
    const unsigned send = 8u * (unsigned)A.nbuf;
    const unsigned xa_sum = 2 * xa0 + vbytes, xb_sum = 2 * xb0 + vbytes;  // of the two buffers
    unsigned sta = st0, sto = 0, stn = nx;  // stage of the column, its barriers, m_b in the stage of the row below
    unsigned sph = 0, par = 0;
    // the pixel's labels start this many ints into the 16-byte chunks copied
    unsigned csh = FUSED ? 0u : (unsigned)((((size_t)y * W + (w.incx ? 0 : W - 1)) * Q) & 3);
    const unsigned dcs = FUSED ? 0u : (unsigned)((w.incx ? Q : -Q) & 3);
    In0 c;
    c.lam_a = c.lam_b = A.lam;
    c.cap_a = c.cap_b = A.capv;
    c.ma = zs;
    c.xa = xa0 + vbytes;
    c.xb = xb0;
#pragma unroll 1
    for (int xs = 0; xs < W; ++xs) {
        if (__builtin_expect(A.wh != nullptr, 0)) {  // per-edge multipliers of the two outgoing edges
            const int x = w.incx ? xs : W - 1 - xs;
            const int wa = xs + 1 < W ? __ldg(A.wh + (size_t)y * W + (w.incx ? x : x - 1)) : 1;
            const int wb = w.has_next ? __ldg(A.wv + (size_t)(w.incy ? y : y - 1) * W + x) : 1;
            c.lam_a = A.lam * wa;
            c.cap_a = A.capv * wa;
            c.lam_b = A.lam * wb;
            c.cap_b = A.capv * wb;
        }
        c.C = sta + 4 * csh;
        c.mc = w.read_c && xs + 1 < W ? sta + omc : zs;
        c.md = w.d_ok ? sta + omd : zs;
        c.mb = w.r > 0 ? sta + omb : zs;
        if (FUSED) {
            c.fp.x = w.incx ? xs : W - 1 - xs;
            c.fp.y = y;
            c.fp.i0 = A.fI0[(size_t)y * A.fpitch + c.fp.x];
        }
        bool ok = mbar_try(bars + kLoadB + sto, sph);
        ok = mbar_try(bars + kReadyB + sto, sph) && ok;
        if (__builtin_expect(!__all_sync(kFull, ok), 0)) {
            ok = mbar_wait(bars + kLoadB + sto, sph, A.spin_limit, s_abort) &&
                 mbar_wait(bars + kReadyB + sto, sph, A.spin_limit, s_abort);
            if (!__all_sync(kFull, ok) && lane == 0) {
                *bad = 1;
                timed_out(A.status, s_abort);
            }
            __syncwarp();
        }
        int ja = kBig, jb = kBig, sv = 0x7fffffff, sq = 0x7fffffff;
        auto first = [&](const Seg &s, const int t) {
            phase0<C0, FIN, PA, FUSED>(A, c, s, A.seg[0].near != 0, FUSED ? C0::pos(A, 0, s.k) : 0,
                                       FUSED ? min(t * C0::lpw + s.l, C0::nlines(A, 0) - 1) : 0, ja, jb, sv, sq);
        };
        if (wt < n0) {
            first(s0, wt);
#pragma unroll 1
            for (int t = wt + T; __builtin_expect(t < n0, 0); t += T) first(seg_of<C0>(A, 0, t * C0::lpw, lane), t);
        }
        if (FIN) {
            const int v = __reduce_min_sync(kFull, sv);
            const int q = __reduce_min_sync(kFull, sv == v ? sq : 0x7fffffff);
            if (lane == 0) {
                wkey[wt] = v;
                wkey[kMaxT + wt] = q;
            }
        }
        if (!PA) {
            ja = __reduce_min_sync(kFull, ja);
            jb = __reduce_min_sync(kFull, jb);
            if (lane == 0) {
                wmin[wt] = ja;
                wmin[kMaxT + wt] = jb;
            }
        }
        __syncwarp();
        mbar_arrive_if(lane == 0, bars + kEmptyB + sto);  // this warp has read the column's inputs
        team_sync(tm, T);
        const int stop = lds(saddr(bad));  // written before this barrier only
        if (FIN && wt == T - 1) {
            const int v = lane < T ? wkey[lane] : 0x7fffffff, q = lane < T ? wkey[kMaxT + lane] : 0x7fffffff;
            const int vm = __reduce_min_sync(kFull, v);
            const int qm = __reduce_min_sync(kFull, v == vm ? q : 0x7fffffff);
            if (lane == 0) A.labels[(size_t)y * W + (w.incx ? xs : W - 1 - xs)] = qm;
        }
        // a line group of a later phase
        auto later = [&](auto cut, const int r, const Seg &s, const unsigned nb, const int ca, const int cb, const Rec &rec) {
            phase_r<decltype(cut), PA>(A, r, s, A.seg[r].near != 0, c, nb, ca, cb, rec);
        };
        int ca = PA ? c.cap_a : kBig, cb = PA ? c.cap_b : kBig;
        if constexpr (R == 3) {
            if (wt < n1) {
                const Rec none{nullptr, 0};
                later(C1(), 1, s1, c.xb, ca, cb, none);
#pragma unroll 1
                for (int t = wt + T; __builtin_expect(t < n1, 0); t += T)
                    later(C1(), 1, seg_of<C1>(A, 1, t * C1::lpw, lane), c.xb, ca, cb, none);
            }
            team_sync(tm, T);
        }
        if (!PA) {
            ca = __reduce_min_sync(kFull, lane < T ? wmin[lane] : kBig) + c.cap_a;
            cb = __reduce_min_sync(kFull, lane < T ? wmin[kMaxT + lane] : kBig) + c.cap_b;
        }
        const unsigned nb = w.to_mbox ? stn : c.xb;
        Rec rec{nullptr, 0};
        if (__builtin_expect(w.recs != nullptr, 0)) {
            const int s = w.col0 + xs;
            rec.p = w.recs + (size_t)(s % A.ring) * Qm;
            rec.tag = A.tag0 + s;
        }
        if (wt < nl) {
            later(CL(), R - 1, s2, nb, ca, cb, rec);
#pragma unroll 1
            for (int t = wt + T; __builtin_expect(t < nl, 0); t += T)
                later(CL(), R - 1, seg_of<CL>(A, R - 1, t * CL::lpw, lane), nb, ca, cb, rec);
        }
        if (__builtin_expect(stop != 0, 0)) break;
        __syncwarp();
        mbar_arrive_if(lane == 0, bars + kOutB + par);
        mbar_arrive_if(lane == 0 && w.to_mbox, nx_ready + sto);
        team_sync(tm, T);
        par ^= 8;
        c.ma = c.xa;
        c.xa = xa_sum - c.xa;
        c.xb = xb_sum - c.xb;
        csh = (csh + dcs) & 3;
        sto += 8;
        const bool wrap = sto == send;
        sta = wrap ? st0 : sta + stb;
        stn = wrap ? nx : stn + stb;
        sph ^= wrap ? 1u : 0u;
        sto = wrap ? 0u : sto;
    }
}

}  // namespace line2

// One work item: half h of the launch's sweep over the rows of one band.
// Every thread of the block calls it; returns false when the pass was
// aborted (a wait timed out).
template <class B, bool FUSED>
__device__ __forceinline__ bool line2_item(const TeamArgs &A, const int h, const int band, int *smem,
                                           volatile int *s_abort) {
    using namespace line2;
    const int W = A.W, H = A.H, Q = A.Q, Qm = A.Qm, T = A.T, NT = A.NT;
    const int nst = A.nbuf, ring = A.ring;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool copy = warp >= NT * T;
    const int tm = copy ? (warp - NT * T) / kCopyWarps : warp / T;
    const int wt = copy ? (warp - NT * T) % kCopyWarps : warp - tm * T;  // role / compute warp of the team
    // shared memory: a zero vector, then the teams (stages, X_a, X_b, control)
    const size_t TI = team_ints(Qm, nst, B::extra);
    int *const zero = smem;
    auto team_of = [&](int i) { return smem + Qm + (size_t)i * TI; };
    auto ctl_of = [&](int i) { return team_of(i + 1) - kCtlInts; };
    int *const tb = team_of(tm);
    int *const XA = tb + nst * stage_ints(Qm);
    int *const XB = XA + 2 * (size_t)Qm;
    int *const ctl = ctl_of(tm);
    int *const wmin = ctl + 32, *const wkey = ctl + 80;
    auto bars_of = [&](int i) { return saddr(ctl_of(i)); };
    const unsigned bars = bars_of(tm);

    for (int i = tid; i < NT * kBars; i += blockDim.x) {
        const int t = i / kBars;
        const unsigned o = 8u * (unsigned)(i - t * kBars);
        const int n = o >= kEmptyB ? T                                   // the compute warps
                      : o >= kReadyB ? 1 + (t > 0 ? T : 0)               // out, the compute warps of the team above
                                     : 1 + (t == 0 && band > 0 ? 1 : 0); // stage, above
        mbar_init(bars_of(t) + o, (unsigned)n);
    }
    for (int i = tid; i < Qm; i += blockDim.x) zero[i] = 0;
    if (tid < NT) ctl_of(tid)[30] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
    __syncthreads();
    if (A.trace && tid == 0 && h == 0) A.trace[band * 4 + 0] = global_ns();

    const int r = band * NT + tm;
    const bool row_on = r < H;
    const bool incx = ((A.pass + h) & 1) == 0, incy = A.pass < 2;
    const bool read_c = h ? A.read_c2 : A.read_c, write_a = h ? A.write_a2 : A.write_a;
    const bool write_b = h ? A.write_b2 : A.write_b, fin = h ? A.final2 : A.final_;
    const int y = incy ? r : H - 1 - r;
    const bool has_next = r + 1 < H;
    const bool to_mbox = has_next && tm + 1 < NT, to_ring = has_next && tm + 1 == NT;
    const bool from_ring = r > 0 && tm == 0;
    const bool d_ok = A.read_d && (incy ? y + 1 < H : y - 1 >= 0);
    int *const Ma = incx ? A.M[0] : A.M[1];
    const int *const Mc = incx ? A.M[1] : A.M[0];
    int *const Mb = incy ? A.M[2] : A.M[3];
    const int *const Md = incy ? A.M[3] : A.M[2];
    int *const ringv = reinterpret_cast<int *>(A.ll);  // copies: [band][ring][Qm] ints; records: int2
    const int col0 = h * W;                              // column counters run on over both halves
    const unsigned vbytes = 4u * (unsigned)Qm;
    const unsigned stb = 4u * (unsigned)stage_ints(Qm);  // bytes of a stage
    const unsigned omc = vbytes + 16, omd = 2 * vbytes + 16, omb = 3 * vbytes + 16;  // m_c, m_d, m_b in it
    const long long lim = A.spin_limit;

    if (copy && lane == 0 && wt < 2) ctl[28 + wt] = 0;
    if (copy && row_on && wt == 1 && A.rec) {
        // ---- above, records: the whole warp polls a column's words into the stage ----
        if (from_ring) {
            const int2 *const recs = A.ll + (size_t)(band - 1) * ring * Qm;
            unsigned *const cons = A.cons + (size_t)(band - 1) * kLineFlagStride + h;
            // the test hook hold_band makes one band wait for tags never written
            const int tag0 = A.tag0 + col0 + (band == A.hold_band ? 0x20000000 : 0);
            int si = 0, slot = col0 % ring;
            unsigned ph = 0;
            bool ok = true;
            // the first half of this row still counts the ring's columns until it
            // is complete (its out warps say so); the lanes agree on the outcome,
            // since they vote in every column
            if (h == 1)
                ok = __all_sync(kFull, wait_count(A.rflag + (size_t)r * kLineFlagStride + 2, 2, lim, s_abort, A.status));
            constexpr int kBatch = 4;  // 16-byte loads per lane: 256 labels
            auto load = [&](int4 (&v)[kBatch], const int2 *src, int q0) {
#pragma unroll
                for (int u = 0; u < kBatch; ++u)
                    if (q0 + 64 * u < Q) v[u] = ld_rec2(src + q0 + 64 * u);
            };
            // the words of labels q0, q0 + 64, ...: polled until they carry the tag
            auto take = [&](int4 (&v)[kBatch], const int2 *src, unsigned dst, int q0, int tag) {
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    const int q = q0 + 64 * u;
                    if (q >= Q || !ok) continue;
                    for (long long n = 0; !(v[u].y == tag && (q + 1 >= Q || v[u].w == tag)); ++n) {
                        if (n > lim || *s_abort || ((n & 63) == 63 && *(volatile int *)A.status != 0)) {
                            ok = false;
                            break;
                        }
                        v[u] = ld_rec2(src + q);
                    }
                    sts(dst + 4u * (unsigned)q, v[u].x);
                    if (q + 1 < Q) sts(dst + 4u * (unsigned)q + 4u, v[u].z);
                }
            };
            int4 cur[kBatch], nxt[kBatch];  // this column's words, and the next one's already on their way
            if (ok) load(nxt, recs + (size_t)slot * Qm, 2 * lane);
            for (int xs = 0; xs < W && ok; ++xs) {
                const int2 *const src = recs + (size_t)slot * Qm;
                if (++slot == ring) slot = 0;
#pragma unroll
                for (int u = 0; u < kBatch; ++u) cur[u] = nxt[u];
                if (xs + 1 < W) load(nxt, recs + (size_t)slot * Qm, 2 * lane);
                if (xs >= nst) ok = mbar_wait(bars + kEmptyB + 8 * si, ph ^ 1, lim, s_abort);
                ok = __all_sync(kFull, ok);
                if (!ok) break;
                const unsigned dst = saddr(tb) + (unsigned)si * stb + omb;
                const int tag = tag0 + xs;
                take(cur, src, dst, 2 * lane, tag);
                for (int q0 = 2 * lane + 64 * kBatch; q0 < Q && ok; q0 += 64 * kBatch) {
                    load(cur, src, q0);
                    take(cur, src, dst, q0, tag);
                }
                ok = __all_sync(kFull, ok);
                if (!ok) break;
                if (lane == 0) {
                    mbar_arrive(bars + kLoadB + 8 * si);
                    ctl[29] = xs + 1;
                    // every lane's loads of the slot have returned
                    st_relaxed_gpu(cons, (unsigned)(col0 + xs + 1));
                }
                if (++si == nst) {
                    si = 0;
                    ph ^= 1;
                }
            }
            if (!ok && lane == 0) timed_out(A.status, s_abort);
        }
    } else if (copy && row_on && lane == 0) {
        int si = 0;       // stage of the column
        unsigned ph = 0;  // its phase
        bool ok = true;
        auto advance = [&](int by) {
            si += by;
            while (si >= nst) {
                si -= nst;
                ph ^= 1;
            }
        };
        if (wt == 0) {
            // ---- stage: C, m_c, m_d of every column ----
            if (h == 1) {  // this row of the first half is complete (both its out warps)
                ok = wait_count(A.rflag + (size_t)r * kLineFlagStride + 2, 2, lim, s_abort, A.status);
                fence_async();
            }
            const size_t NQ = (size_t)W * H * Q;
            for (int xs = 0; xs < W && ok; ++xs, advance(1)) {
                if (xs >= nst && !(ok = mbar_wait(bars + kEmptyB + 8 * si, ph ^ 1, lim, s_abort))) break;
                const size_t pix = (size_t)y * W + (incx ? xs : W - 1 - xs);
                const bool c_ok = read_c && xs + 1 < W;
                const unsigned dst = saddr(tb) + (unsigned)si * stb, bar = bars + kLoadB + 8 * si;
                unsigned cbytes = 0;
                size_t a0 = 0;
                if (!FUSED) {
                    // whole 16-byte chunks around the pixel's labels; the array's
                    // last labels, short of a chunk, by plain loads
                    const size_t e0 = pix * Q, e1 = e0 + Q;
                    a0 = e0 & ~(size_t)3;
                    size_t a1 = (e1 + 3) & ~(size_t)3;
                    if (a1 > NQ) {
                        a1 = max(e1 & ~(size_t)3, a0);
                        for (size_t e = a1; e < e1; ++e) tb[(size_t)si * stage_ints(Qm) + (e - a0)] = A.C[e];
                    }
                    cbytes = 4u * (unsigned)(a1 - a0);
                }
                mbar_arrive_tx(bar, cbytes + (c_ok ? vbytes : 0) + (d_ok ? vbytes : 0));
                if (cbytes) bulk_load(dst, A.C + a0, cbytes, bar);
                if (c_ok) bulk_load(dst + omc, Mc + pix * Qm, vbytes, bar);
                if (d_ok) bulk_load(dst + omd, Md + pix * Qm, vbytes, bar);
                ctl[28] = xs + 1;
            }
        } else if (wt == 1) {
            // ---- above: m_b of every column the previous band published ----
            if (from_ring) {
                const unsigned *const flag = A.rflag + (size_t)(band - 1) * kLineFlagStride;
                unsigned *const cons = A.cons + (size_t)(band - 1) * kLineFlagStride + h;
                // the test hook hold_band makes one band wait for a column never published
                const int hold = band == A.hold_band ? 0x20000000 : 0;
                int seen[2] = {0, 0};  // published columns as last read, even / odd
                for (int xs = 0; xs < W && ok; ++xs, advance(1)) {
                    const int s = col0 + xs;
                    if (xs >= nst) {
                        if (!(ok = mbar_wait(bars + kEmptyB + 8 * si, ph ^ 1, lim, s_abort))) break;
                        // column s - nst has left the ring (the compute warps have
                        // read it from shared memory)
                        st_relaxed_gpu(cons, (unsigned)(s - nst + 1));
                    }
                    for (long long n = 0; (s & 1 ? seen[1] : seen[0]) < s + 1 + hold; ++n) {
                        if (n > lim || *s_abort || ((n & 63) == 63 && *(volatile int *)A.status != 0)) {
                            ok = false;
                            break;
                        }
                        const uint2 v = ld_acq_gpu2(flag);
                        seen[0] = (int)v.x;
                        seen[1] = (int)v.y;
                    }
                    if (!ok) break;
                    fence_async();
                    const int *const src = write_b ? Mb + ((size_t)y * W + (incx ? xs : W - 1 - xs)) * Qm
                                                   : ringv + ((size_t)(band - 1) * ring + s % ring) * Qm;
                    const unsigned bar = bars + kLoadB + 8 * si;
                    mbar_arrive_tx(bar, vbytes);
                    bulk_load(saddr(tb) + (unsigned)si * stb + omb, src, vbytes, bar);
                    ctl[29] = xs + 1;
                }
                for (int xs = max(0, W - nst); xs < W && ok; ++xs)
                    ok = mbar_wait(bars + kEmptyB + 8 * (xs % nst), (xs / nst) & 1, lim, s_abort);
                if (ok) st_relaxed_gpu(cons, (unsigned)(col0 + W));
            }
        } else {
            // ---- out p: the finished columns p, p + 2, ... ----
            const int p = wt - 2;
            const unsigned *const cons = A.cons + (size_t)band * kLineFlagStride;
            unsigned *const flag = A.rflag + (size_t)band * kLineFlagStride;
            const int y_next = incy ? y + 1 : y - 1;
            const unsigned nx_bars = to_mbox ? bars_of(tm + 1) : 0;
            unsigned oph = 0;
            const bool rec = A.rec != 0;
            int room = 0;  // columns of this band's ring known to be counted by the consumer
            // the output buffers of column xs are free, and its ring slot
            auto ring_free = [&](int s) {
                if (room >= s - ring + 1) return true;
                for (long long n = 0; n <= lim; ++n) {
                    const uint2 v = ld_acq_gpu2(cons);
                    room = (int)max(v.x, v.y);
                    if (room >= s - ring + 1) return true;
                    if (*s_abort || ((n & 63) == 63 && *(volatile int *)A.status != 0)) return false;
                    __nanosleep(20);
                }
                return false;
            };
            advance(p);
            if (p < W) {
                if (to_ring && rec) ok = ring_free(col0 + p);
                if (ok) mbar_arrive(bars + kReadyB + 8 * si);
            }
            for (int xs = p; xs < W && ok; xs += 2) {
                const int s = col0 + xs;
                if (!(ok = mbar_wait(bars + kOutB + 8 * p, oph, lim, s_abort))) break;
                oph ^= 1;
                // the compute warps' shared-memory writes (ordered by the barrier
                // above) before the bulk copies' reads
                fence_async();
                const int x = incx ? xs : W - 1 - xs;
                if (write_a && xs + 1 < W)
                    bulk_store(Ma + ((size_t)y * W + (incx ? x + 1 : x - 1)) * Qm, saddr(XA + (size_t)(p ^ 1) * Qm), vbytes);
                const unsigned src = to_mbox ? saddr(team_of(tm + 1)) + (unsigned)si * stb + omb
                                             : saddr(XB + (size_t)p * Qm);
                if (has_next && write_b) {
                    bulk_store(Mb + ((size_t)y_next * W + x) * Qm, src, vbytes);
                } else if (to_ring && !rec) {
                    if (!(ok = ring_free(s))) break;
                    fence_async();
                    bulk_store(ringv + ((size_t)band * ring + s % ring) * Qm, src, vbytes);
                }
                bulk_commit();
                bulk_wait_read();
                advance(2);
                if (xs + 2 < W) {
                    // the buffers of column xs + 2 are free: those of column xs have
                    // been read, and so has the stage of the row below
                    if (to_mbox && xs + 2 >= nst &&
                        !(ok = mbar_wait(nx_bars + kEmptyB + 8 * si, ph ^ 1, lim, s_abort)))
                        break;
                    if (to_ring && rec && !(ok = ring_free(s + 2))) break;
                    mbar_arrive(bars + kReadyB + 8 * si);
                }
                if (to_ring && !rec) {
                    bulk_wait_all();
                    fence_async();
                    st_rel_gpu(flag + (s & 1), (unsigned)(s + 1));
                }
            }
            bulk_wait_all();
            if (ok && A.pair && h == 0) {
                fence_async();
                add_rel_gpu(A.rflag + (size_t)r * kLineFlagStride + 2, 1u);
            }
        }
        if (!ok) timed_out(A.status, s_abort);
    } else if (!copy && row_on) {
        const Row w{r, y, tm, wt, lane, incx, incy, has_next, to_mbox, read_c, d_ok,
                    to_ring && A.rec ? A.ll + (size_t)band * ring * Qm : nullptr, col0};
        auto run = [&](auto fin_c, auto pa_c) {
            B::template row<decltype(fin_c)::value, decltype(pa_c)::value, FUSED>(
                A, w, saddr(zero), saddr(tb), saddr(XA), saddr(XB), bars, to_mbox ? saddr(team_of(tm + 1)) + omb : 0u,
                to_mbox ? bars_of(tm + 1) + kReadyB : 0u, wmin, wkey, ctl + 30, s_abort);
        };
        if (A.mode == 1)
            fin ? run(std::true_type(), std::true_type()) : run(std::false_type(), std::true_type());
        else
            fin ? run(std::true_type(), std::false_type()) : run(std::false_type(), std::false_type());
    }
    __syncthreads();
    const bool done = *s_abort == 0;
    if (!done && tid < NT) {
        // an aborted item: wait (bounded) for the copies in flight into the
        // stages; where only one of `stage` and `above` announced a column,
        // make up the other's arrival
        const int *const issued = ctl_of(tid) + 28;
        const bool two = tid == 0 && band > 0;
        const int n = max(issued[0], issued[1]);
        if (two)
            for (int xs = min(issued[0], issued[1]); xs < n; ++xs) mbar_arrive(bars_of(tid) + kLoadB + 8 * (xs % nst));
        for (int xs = max(0, n - nst); xs < n; ++xs)
            for (int k = 0; k < 1000000 && !mbar_try(bars_of(tid) + kLoadB + 8 * (xs % nst), (xs / nst) & 1); ++k) {
            }
    }
    if (A.trace && tid == 0) {
        A.trace[band * 4 + 1] = global_ns();
        A.trace[band * 4 + 2] = 0;
        A.trace[band * 4 + 3] = sm_id();
    }
    __syncthreads();
    for (int i = tid; i < NT * kBars; i += blockDim.x) mbar_inval(bars_of(i / kBars) + 8 * (i % kBars));
    __syncthreads();
    return done;
}

}  // namespace edp
