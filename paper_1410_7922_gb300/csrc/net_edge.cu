// net_edge.cu -- the proposal network's first and last layers (5 -> 32 and
// 32 -> 2 channels) on the CUDA cores: convolutions, the last layer's input
// gradient and both weight gradients.  bf16 operands, float32 products and sums.
//
// Bound: float32 FMAs and the shared-memory reads that feed them; one channel
// count is too small for a tensor-core tile.  So every operand read from shared
// memory serves many FMAs (8 to 40), channel pairs go through the two-wide
// fma.rn.f32x2, activations move as 16-byte words of 8 channels, and the layers
// read their weights from the parameters themselves (no preparation launch).
//
// With these kernels and one weight preparation for all tensor-core layers: forward,
// 1 x 480 x 640, 264 -> 156 us; a training step, 8 x 240 x 320, 1991 -> 1048 us (948
// with one wave of blocks here and a wider sum of the partial gradients).
// (Before: one FMA per shared-memory read, channels stored 2 bytes at a time, and a
// block's 1440 gradient sums added to memory for every tile of 256 pixels.)
#include <cuda_bf16.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace edp {

namespace {
constexpr int kT = 16, kTW = kT + 2;  // tile side, with halo

typedef unsigned long long f2;  // two floats
__device__ __forceinline__ f2 pack2(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ void fma2(f2 &d, f2 a, f2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
// a word of two bf16 channels
__device__ __forceinline__ f2 widen2(unsigned w) { return pack2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
__device__ __forceinline__ float round_bf(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
__device__ __forceinline__ unsigned narrow2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const unsigned *>(&h);
}
}  // namespace

// CIN (5 or 2) -> 32 channels.  MODE 0: relu(z + b) of weights w[32][CIN][9];
// MODE 2, an input gradient: z with the flipped weights w[CIN][32][9], masked by
// act > 0.  Two pixels (8 rows apart) of a 16 x 16 tile per thread, 32 outputs each.
template <int CIN, int MODE>
__global__ void __launch_bounds__(128) net_conv_narrow(const __nv_bfloat16 *in, int H, int W, const float *w, const float *bias,
                                                       __nv_bfloat16 *out, const __nv_bfloat16 *act) {
    constexpr int CP = CIN | 1;  // odd: the lanes of a warp hit distinct banks
    __shared__ __align__(16) float ws[9 * CIN * 32];
    __shared__ float tile[kTW * kTW * CP];
    const int tid = threadIdx.x, x0 = blockIdx.x * kT, y0 = blockIdx.y * kT;
    const size_t img = (size_t)blockIdx.z * H * W;
    for (int e = tid; e < 9 * CIN * 32; e += 128) {
        const int t = e % 9;
        if (MODE == 0)
            ws[(t * CIN + (e / 9) % CIN) * 32 + e / (9 * CIN)] = round_bf(w[e]);
        else
            ws[((8 - t) * CIN + e / (9 * 32)) * 32 + (e / 9) % 32] = round_bf(w[e]);
    }
    for (int e = tid; e < kTW * kTW * CIN; e += 128) {
        const int c = e % CIN, p = e / CIN, y = y0 + p / kTW - 1, x = x0 + p % kTW - 1;
        tile[p * CP + c] = y >= 0 && y < H && x >= 0 && x < W ? __bfloat162float(in[(img + (size_t)y * W + x) * CIN + c]) : 0.f;
    }
    __syncthreads();
    const int lx = tid % kT, ly = tid / kT;
    f2 acc[2][16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[0][i] = acc[1][i] = 0;
#pragma unroll 1
    for (int t = 0; t < 9; ++t) {
        const float *a = tile + ((ly + t / 3) * kTW + lx + t % 3) * CP;
#pragma unroll
        for (int ci = 0; ci < CIN; ++ci) {
            const f2 u = pack2(a[ci], a[ci]), v = pack2(a[8 * kTW * CP + ci], a[8 * kTW * CP + ci]);
            const ulonglong2 *wr = reinterpret_cast<const ulonglong2 *>(ws + (t * CIN + ci) * 32);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const ulonglong2 q = wr[i];
                fma2(acc[0][2 * i], u, q.x);
                fma2(acc[0][2 * i + 1], u, q.y);
                fma2(acc[1][2 * i], v, q.x);
                fma2(acc[1][2 * i + 1], v, q.y);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int x = x0 + lx, y = y0 + ly + 8 * k;
        if (x >= W || y >= H) continue;
        const size_t o = (img + (size_t)y * W + x) * 32;
#pragma unroll
        for (int j = 0; j < 4; ++j) {  // 8 channels, 16 bytes
            uint4 m = make_uint4(0, 0, 0, 0), r;
            if (MODE == 2) m = *reinterpret_cast<const uint4 *>(act + o + 8 * j);
            const unsigned mw[4] = {m.x, m.y, m.z, m.w};
            unsigned rw[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float2 z = unpack2(acc[k][4 * j + i]);
                if (MODE == 0) {
                    z.x = fmaxf(z.x + bias[8 * j + 2 * i], 0.f);
                    z.y = fmaxf(z.y + bias[8 * j + 2 * i + 1], 0.f);
                } else {
                    if (!(__uint_as_float(mw[i] << 16) > 0.f)) z.x = 0.f;
                    if (!(__uint_as_float(mw[i] & 0xffff0000u) > 0.f)) z.y = 0.f;
                }
                rw[i] = narrow2(z.x, z.y);
            }
            r = make_uint4(rw[0], rw[1], rw[2], rw[3]);
            *reinterpret_cast<uint4 *>(out + o + 8 * j) = r;
        }
    }
}

// 32 -> 2 channels, out = z + b (float32).  Four rows of one column of a 16 x 16
// tile per thread: a word (two channels) of six rows and three taps' weights serve
// 24 two-wide FMAs.  17 words a pixel and 308 a row: a warp's 16 columns of two
// row groups lie in 32 banks.
__global__ void __launch_bounds__(64) net_conv_out(const __nv_bfloat16 *in, int H, int W, const float *w, const float *bias,
                                                   float *out) {
    constexpr int PW = 17, RW = kTW * PW + 2;
    __shared__ __align__(16) float ws[3 * 16 * 12];  // [dx][channel pair][dy][co][2]
    __shared__ unsigned tile[kTW * RW];
    const int tid = threadIdx.x, x0 = blockIdx.x * kT, y0 = blockIdx.y * kT;
    const size_t img = (size_t)blockIdx.z * H * W;
    for (int e = tid; e < 2 * 32 * 9; e += 64) {
        const int t = e % 9, ci = (e / 9) % 32, co = e / 288;
        ws[((t % 3) * 16 + ci / 2) * 12 + (t / 3) * 4 + co * 2 + (ci & 1)] = round_bf(w[e]);
    }
    for (int e = tid; e < kTW * kTW * 4; e += 64) {
        const int j = e % 4, p = e / 4, y = y0 + p / kTW - 1, x = x0 + p % kTW - 1;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (y >= 0 && y < H && x >= 0 && x < W) v = *reinterpret_cast<const uint4 *>(in + (img + (size_t)y * W + x) * 32 + 8 * j);
        unsigned *s = tile + (p / kTW) * RW + (p % kTW) * PW + 4 * j;
        s[0] = v.x, s[1] = v.y, s[2] = v.z, s[3] = v.w;
    }
    __syncthreads();
    const int lx = tid % kT, ly = tid / kT * 4;
    f2 acc[4][2];  // sums of even and of odd channels
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k][0] = acc[k][1] = 0;
#pragma unroll 1
    for (int dx = 0; dx < 3; ++dx) {
        const unsigned *a = tile + ly * RW + (lx + dx) * PW;
#pragma unroll 4
        for (int c = 0; c < 16; ++c) {
            f2 v[6];
#pragma unroll
            for (int i = 0; i < 6; ++i) v[i] = widen2(a[i * RW + c]);
            const ulonglong2 *wr = reinterpret_cast<const ulonglong2 *>(ws + (dx * 16 + c) * 12);
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const ulonglong2 q = wr[dy];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    fma2(acc[k][0], v[k + dy], q.x);
                    fma2(acc[k][1], v[k + dy], q.y);
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int x = x0 + lx, y = y0 + ly + k;
        if (x >= W || y >= H) continue;
        const float2 s = unpack2(acc[k][0]), t = unpack2(acc[k][1]);
        float *o = out + (img + (size_t)y * W + x) * 2;
        o[0] = s.x + s.y + bias[0];
        o[1] = t.x + t.y + bias[1];
    }
}

// Weight and bias gradients of a layer with 32 channels on one side and NN on the
// other: dW[co][ci][tap] += sum g[p][co] x[p + tap][ci], db[co] += sum g[p][co].
// IN32: the 32 channels are the layer's input (32 -> 2), else its output (5 -> 32).
// Warp = tap, lane = 8 of the 32 channels x one of 8 pixel slices: a 16-byte read
// of 8 channels and NN reads serve 8 NN products.  A block keeps its sums in
// registers over all its tiles and adds them to dW once.
template <int NN, bool IN32>
__global__ void __launch_bounds__(288) net_wgrad_edge(const __nv_bfloat16 *g, const __nv_bfloat16 *x, int N, int H, int W,
                                                      float *dW, float *db) {
    constexpr int PX = kTW * kTW, PG = kT * kT, PWD = IN32 ? PX : PG, PN = IN32 ? PG : PX;
    __shared__ uint4 wide[PWD * 5];  // 4 words of 8 channels, 80 bytes a pixel: slices in distinct banks
    __shared__ f2 thin[PN * NN];     // each value twice
    const int tid = threadIdx.x, lane = tid & 31, tap = tid >> 5, dy = tap / 3, dx = tap % 3;
    const int s = lane & 7, cg = lane >> 3;
    const int tx = (W + kT - 1) / kT, ty = (H + kT - 1) / kT;
    f2 acc[NN][4], sum[4];
    float tsum[NN];
#pragma unroll
    for (int i = 0; i < 4; ++i) sum[i] = 0;
#pragma unroll
    for (int n = 0; n < NN; ++n) {
        tsum[n] = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[n][i] = 0;
    }
    const f2 one = pack2(1.f, 1.f);
    for (long long t = blockIdx.x; t < (long long)tx * ty * N; t += gridDim.x) {
        const int x0 = (int)(t % tx) * kT, y0 = (int)(t / tx % ty) * kT;
        const size_t img = (size_t)(t / tx / ty) * H * W;
        __syncthreads();
        for (int e = tid; e < PWD * 4; e += 288) {
            const int p = e / 4, yy = IN32 ? y0 + p / kTW - 1 : y0 + p / kT, xx = IN32 ? x0 + p % kTW - 1 : x0 + p % kT;
            uint4 v = make_uint4(0, 0, 0, 0);
            if (yy >= 0 && yy < H && xx >= 0 && xx < W)
                v = *reinterpret_cast<const uint4 *>((IN32 ? x : g) + (img + (size_t)yy * W + xx) * 32 + 8 * (e % 4));
            wide[p * 5 + e % 4] = v;
        }
        for (int e = tid; e < PN * NN; e += 288) {
            const int p = e / NN, yy = IN32 ? y0 + p / kT : y0 + p / kTW - 1, xx = IN32 ? x0 + p % kT : x0 + p % kTW - 1;
            float v = 0.f;
            if (yy >= 0 && yy < H && xx >= 0 && xx < W)
                v = __bfloat162float((IN32 ? g : x)[(img + (size_t)yy * W + xx) * NN + e % NN]);
            thin[e] = pack2(v, v);
        }
        __syncthreads();
#pragma unroll 2
        for (int k = 0; k < 32; ++k) {
            const int py = k >> 1, px = s + 8 * (k & 1);
            const int ph = (py + dy) * kTW + px + dx, pc = py * kT + px;
            const uint4 v = wide[(IN32 ? ph : pc) * 5 + cg];
            const f2 c[4] = {widen2(v.x), widen2(v.y), widen2(v.z), widen2(v.w)};
            const f2 *q = thin + (IN32 ? pc : ph) * NN;
#pragma unroll
            for (int n = 0; n < NN; ++n) {
                const f2 u = q[n];
#pragma unroll
                for (int i = 0; i < 4; ++i) fma2(acc[n][i], c[i], u);
                if (IN32 && tap == 4) tsum[n] += unpack2(u).x;
            }
            if (!IN32 && tap == 4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) fma2(sum[i], c[i], one);
            }
        }
    }
    auto slices = [&](float v) {
#pragma unroll
        for (int d = 1; d < 8; d <<= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
        return v;
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = cg * 8 + 2 * i;
#pragma unroll
        for (int n = 0; n < NN; ++n) {
            const float2 a = unpack2(acc[n][i]);
            const float u = slices(a.x), v = slices(a.y);
            if (s == 0) {
                atomicAdd(dW + (IN32 ? n * 32 + c : c * NN + n) * 9 + tap, u);
                atomicAdd(dW + (IN32 ? n * 32 + c + 1 : (c + 1) * NN + n) * 9 + tap, v);
            }
        }
        if (!IN32 && tap == 4) {
            const float2 a = unpack2(sum[i]);
            const float u = slices(a.x), v = slices(a.y);
            if (s == 0) {
                atomicAdd(db + c, u);
                atomicAdd(db + c + 1, v);
            }
        }
    }
    if (IN32 && tap == 4) {
#pragma unroll
        for (int n = 0; n < NN; ++n) {
            const float u = slices(tsum[n]);
            if (lane == 0) atomicAdd(db + n, u);
        }
    }
}

static dim3 tiles(int N, int H, int W) { return dim3((W + kT - 1) / kT, (H + kT - 1) / kT, N); }

int net_edge_first(const void *in, int N, int H, int W, const float *w, const float *bias, void *out, cudaStream_t st) {
    net_conv_narrow<5, 0><<<tiles(N, H, W), 128, 0, st>>>(static_cast<const __nv_bfloat16 *>(in), H, W, w, bias,
                                                         static_cast<__nv_bfloat16 *>(out), nullptr);
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
}
int net_edge_last(const void *in, int N, int H, int W, const float *w, const float *bias, float *out, cudaStream_t st) {
    net_conv_out<<<tiles(N, H, W), 64, 0, st>>>(static_cast<const __nv_bfloat16 *>(in), H, W, w, bias, out);
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
}
int net_edge_last_dgrad(const void *g, int N, int H, int W, const float *w, void *out, const void *act, cudaStream_t st) {
    net_conv_narrow<2, 2><<<tiles(N, H, W), 128, 0, st>>>(static_cast<const __nv_bfloat16 *>(g), H, W, w, nullptr,
                                                         static_cast<__nv_bfloat16 *>(out), static_cast<const __nv_bfloat16 *>(act));
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
}
int net_edge_wgrad(const void *g, const void *x, int N, int H, int W, bool first, float *dW, float *db, cudaStream_t st) {
    const dim3 t = tiles(N, H, W);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long n = (long long)t.x * t.y * t.z;
    // one wave of blocks: with a block more per SM than fit, the last ones run alone
    const void *k = first ? (const void *)net_wgrad_edge<5, false> : (const void *)net_wgrad_edge<2, true>;
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, 288, 0);
    const unsigned grid = (unsigned)std::min<long long>(n, (long long)std::max(1, occ) * std::max(1, sms));
    const auto *gp = static_cast<const __nv_bfloat16 *>(g), *xp = static_cast<const __nv_bfloat16 *>(x);
    if (first)
        net_wgrad_edge<5, false><<<grid, 288, 0, st>>>(gp, xp, N, H, W, dW, db);
    else
        net_wgrad_edge<2, true><<<grid, 288, 0, st>>>(gp, xp, N, H, W, dW, db);
    return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

}  // namespace edp
