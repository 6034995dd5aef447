// Warm-start network: 4 layers of periodic 3x3 convolutions (5 -> 32 -> 32 ->
// 32 -> 3 channels, tanh between layers), trained and evaluated on the GPU
// by the kernels below.  Activations are float32 NCHW; the convolutions read
// fp16 copies of the weights (float32 accumulation); Adam updates float32
// master weights and refreshes the fp16 copies.
//
// Inputs (5 planes): normalised tanh-start density, T, kappa, tau, R.
// Outputs (3 planes): (rho_steady - rho_tanh) / (rho_l - rho_g), 1000 u_x, 1000 u_y.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/lb.h"
#include "cnn_common.cuh"
#include "lattice.cuh"   // lbk::static_for

void lb_internal_set_error(const char* msg);

namespace {

constexpr int TILE = 16;                 // 16 x 16 output pixels per CTA
constexpr int NL = 4;
constexpr int CH[NL + 1] = {LB_WS_IN, LB_WS_HIDDEN, LB_WS_HIDDEN, LB_WS_HIDDEN, LB_WS_OUT};

lb_status fail(lb_status s, const std::string& m) {
    lb_internal_set_error(m.c_str());
    return s;
}

// Offset of layer l's weights in the packed parameter vector.
constexpr int layer_offset(int l) {
    int p = 0;
    for (int k = 0; k < l; ++k) p += CH[k + 1] * CH[k] * 9 + CH[k + 1];
    return p;
}

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Geometry of a 16 x 16 pixel tile with its one-pixel halo in shared memory:
// 18 rows of 20 floats (16-byte aligned rows), one plane per channel.
constexpr int TP = TILE + 2, ROW = 20, PLANE = TP * ROW;
constexpr int NTH = 256;                           // threads per CTA of every convolution kernel

// The tile's planes of `in` (CH channels of one sample, periodic halo): a
// thread keeps the same pixel positions for every channel, so the wraps and
// the divisions by 18 are done once, not once per element.
template <int CHN, int PL>
__device__ __forceinline__ void load_tile(float* tile, const float* in, int x0, int y0, int H, int Wd) {
    constexpr int NPOS = (TP * TP + NTH - 1) / NTH;
    const size_t plane = size_t(H) * Wd;
#pragma unroll
    for (int m = 0; m < NPOS; ++m) {
        const int pos = threadIdx.x + m * NTH;
        if (pos < TP * TP) {
            const int ty = pos / TP, tx = pos % TP;
            const float* g = in + size_t(wrap(y0 + ty - 1, H)) * Wd + wrap(x0 + tx - 1, Wd);
            float* s = tile + ty * ROW + tx;
#pragma unroll 16
            for (int c = 0; c < CHN; ++c) s[c * PL] = g[c * plane];
        }
    }
}

// A periodic 3 x 3 convolution of CI channels into CO channels of a 16 x 16
// tile: the forward pass (bias, tanh) and, with the taps mirrored, the backward
// pass towards the data (times 1 - h^2).  A thread forms PX adjacent pixels x
// OC channels, two channels per packed FMA; weights come from shared memory as
// warp-wide broadcasts of four channels.  With PX = 4, OC = 8 a thread issues 8
// shared loads (4 or 8 wavefronts of pixels, 6 of weights) for the 96 FMAs of an
// input channel's tap row, which leaves the FP32 pipe as the bound; one pixel
// per thread issued 9 + 72 loads for 288.  A warp holds 8 rows x 4 groups, a
// group per 8 lanes: the rows are 20 banks apart, so its 16-byte loads have no
// conflicts and its stores still fill whole 64-byte rows.  (4 x 16 on 128
// threads read less but left 1.7 warps per scheduler: 42 us.)
// W: the layer's fp16 weights packed [CI][9][COP] (PACK), so a CTA copies them
// as they lie.  Every output sums its products in the same order as a plain
// loop over (channel, tap).  Measured (16 samples of 64 x 64, 32 -> 32
// channels): 34 us forward and 38 us backward against 70 and 76 with one
// pixel per thread.
template <int CI, int CO, int PX, int OC, bool BACK, bool TANH>
__global__ void __launch_bounds__(NTH) conv_tile(const float* in, const __half* W, const float* bias, const float* h,
                                                 float* out, int H, int Wd) {
    lbk::chain_begin();
    constexpr int COP = (CO + 3) / 4 * 4, QW = TILE / PX, NQ = QW * TILE;
    static_assert(NQ * (COP / OC) == NTH && COP % OC == 0 && OC % 4 == 0 && (PX == 4 || PX == 1), "work split");
    extern __shared__ __align__(16) float sm[];
    float* tile = sm;                 // [CI][18][20]
    float* wsh = sm + CI * PLANE;     // [CI][9][COP]
    const int n = blockIdx.z, tid = threadIdx.x;
    const int x0 = blockIdx.x * TILE, y0 = blockIdx.y * TILE;
    load_tile<CI, PLANE>(tile, in + size_t(n) * CI * H * Wd, x0, y0, H, Wd);
    for (int i = tid; i < CI * 9 * COP / 4; i += NTH) {
        const uint2 r = reinterpret_cast<const uint2*>(W)[i];
        __half2 a, b;
        *reinterpret_cast<unsigned*>(&a) = r.x;
        *reinterpret_cast<unsigned*>(&b) = r.y;
        const float2 fa = __half22float2(a), fb = __half22float2(b);
        reinterpret_cast<float4*>(wsh)[i] = make_float4(fa.x, fa.y, fb.x, fb.y);
    }
    __syncthreads();
    const int q = tid % NQ, o0 = (tid / NQ) * OC;
    const int lane = q % 32;
    const int lx = PX == 4 ? (lane >> 3) * 4 : q % TILE, ly = PX == 4 ? (q / 32) * 8 + (lane & 7) : q / TILE;
    float2 acc[PX][OC / 2];
#pragma unroll
    for (int p = 0; p < PX; ++p)
#pragma unroll
        for (int k = 0; k < OC / 2; ++k) {
            if constexpr (BACK) acc[p][k] = make_float2(0.f, 0.f);
            else acc[p][k] = make_float2(o0 + 2 * k < CO ? bias[o0 + 2 * k] : 0.f, o0 + 2 * k + 1 < CO ? bias[o0 + 2 * k + 1] : 0.f);
        }
#pragma unroll 1
    for (int c = 0; c < CI; ++c) {
#pragma unroll
        for (int kk = 0; kk < 3; ++kk) {
            const int ky = BACK ? 2 - kk : kk;
            const float* row = tile + c * PLANE + (ly + ky) * ROW + lx;
            float v[PX + 2];
            if constexpr (PX == 4) {
                const float4 a = *reinterpret_cast<const float4*>(row);
                const float2 b = *reinterpret_cast<const float2*>(row + 4);
                v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y;
            } else {
#pragma unroll
                for (int p = 0; p < PX + 2; ++p) v[p] = row[p];
            }
#pragma unroll
            for (int ll = 0; ll < 3; ++ll) {
                const int kx = BACK ? 2 - ll : ll;
                const float4* w4 = reinterpret_cast<const float4*>(wsh + (c * 9 + ky * 3 + kx) * COP + o0);
#pragma unroll
                for (int k = 0; k < OC / 4; ++k) {
                    const float4 w = w4[k];
#pragma unroll
                    for (int p = 0; p < PX; ++p) {
                        const float2 vv = make_float2(v[p + kx], v[p + kx]);
                        acc[p][2 * k] = ffma2(make_float2(w.x, w.y), vv, acc[p][2 * k]);
                        acc[p][2 * k + 1] = ffma2(make_float2(w.z, w.w), vv, acc[p][2 * k + 1]);
                    }
                }
            }
        }
    }
    const int x = x0 + lx, y = y0 + ly;
    if (x >= Wd || y >= H) return;
    const bool whole = PX == 4 && Wd % 4 == 0;   // a group of pixels is one aligned vector, inside the image
#pragma unroll
    for (int k = 0; k < OC; ++k) {
        if (o0 + k >= CO) break;
        const size_t idx = ((size_t(n) * CO + o0 + k) * H + y) * Wd + x;
        float r[PX];
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            r[p] = k % 2 ? acc[p][k / 2].y : acc[p][k / 2].x;
            if constexpr (TANH) r[p] = tanhf(r[p]);
        }
        if constexpr (PX == 4) {
            if (whole) {
                if constexpr (BACK) {
                    const float4 hh = *reinterpret_cast<const float4*>(h + idx);
                    r[0] *= 1.f - hh.x * hh.x;
                    r[1] *= 1.f - hh.y * hh.y;
                    r[2] *= 1.f - hh.z * hh.z;
                    r[3] *= 1.f - hh.w * hh.w;
                }
                *reinterpret_cast<float4*>(out + idx) = make_float4(r[0], r[1], r[2], r[3]);
                continue;
            }
        }
#pragma unroll
        for (int p = 0; p < PX; ++p) {
            if (x + p < Wd) {
                if constexpr (BACK) r[p] *= 1.f - h[idx + p] * h[idx + p];
                out[idx + p] = r[p];
            }
        }
    }
}

// dW[o,c,k] = sum over pixels of dout[o,p] h[c,p+k]; db[o] = sum dout[o,p].
// A thread forms OT output channels x the nine taps of one input channel (RS
// threads share them, each taking every RS-th row of a tile): for four
// adjacent pixels it loads 3 x 6 values of h and 4 x OT of dout for 36 OT
// FMAs, two channels per packed FMA, where one (channel, tap) pair per thread
// took a shared load for every FMA.  dout lies [pixel][channel] in shared
// memory, so a warp reads it as broadcasts; the channel planes of h are 364
// floats apart (12 banks), which keeps the 16-byte loads of a warp's 32
// channels free of conflicts.  Each CTA sweeps its 16 x 16 tiles, folds its RS
// shares in shared memory and writes one row of partial sums to
// part[blockIdx.x][CO * CI * 9 + CO]; reduce_grads adds the rows.  (Atomic
// additions of the shares cost more than the sums: 256 CTAs x 9216 of them,
// 89 us, and 158 us on the 1440 addresses of the first layer.)  Measured (as
// above): 32 -> 32 channels 42 us against 107 us, 5 -> 32 30 against 42,
// 32 -> 3 13 against 28.  Two CTAs per SM, at 128 registers: with one, at 180, eight
// warps per SM left the shared loads' latency open, and a pass of training (four
// epochs of these 16 samples with the copies) took 1558 us against 1500.  Chained
// launches (chain.cuh) of its fifteen kernels per minibatch take it to 1372.
template <int CI, int CO, int OT, int RS>
__global__ void __launch_bounds__(NTH, 2) conv_bwd_weight(const float* h, const float* dout, float* part, int N, int H, int Wd) {
    lbk::chain_begin();
    constexpr int COP = (CO + 3) / 4 * 4, OG = COP / OT, PL = PLANE + 4, GP = COP == 32 ? COP + 4 : COP;
    static_assert(CI * OG * RS <= NTH && COP % OT == 0 && OT % 4 == 0 && NTH % COP == 0, "work split");
    extern __shared__ __align__(16) float sm[];
    float* tile = sm;                  // [CI][18][20] of h, planes PL apart
    float* gt = sm + CI * PL;          // [256][GP] of dout
    const int tid = threadIdx.x;
    const int c = tid % CI, og = (tid / CI) % OG, rs = tid / (CI * OG);
    const int tiles_x = (Wd + TILE - 1) / TILE, tiles_y = (H + TILE - 1) / TILE;
    const int ntiles = N * tiles_x * tiles_y;
    float2 acc[9][OT / 2];
#pragma unroll
    for (int k = 0; k < 9; ++k)
#pragma unroll
        for (int j = 0; j < OT / 2; ++j) acc[k][j] = make_float2(0.f, 0.f);
    float bacc = 0.f;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int n = t / (tiles_x * tiles_y), r0 = t % (tiles_x * tiles_y);
        const int x0 = (r0 % tiles_x) * TILE, y0 = (r0 / tiles_x) * TILE;
        __syncthreads();
        load_tile<CI, PL>(tile, h + size_t(n) * CI * H * Wd, x0, y0, H, Wd);
#pragma unroll
        for (int m = 0; m < TILE * TILE / NTH; ++m) {
            const int p = tid + m * NTH, x = x0 + p % TILE, y = y0 + p / TILE;
            const bool in = x < Wd && y < H;
            const float* g = dout + (size_t(n) * CO * H + y) * Wd + x;
#pragma unroll 8
            for (int o = 0; o < CO; ++o) gt[p * GP + o] = in ? g[size_t(o) * H * Wd] : 0.f;
#pragma unroll
            for (int o = CO; o < COP; ++o) gt[p * GP + o] = 0.f;
        }
        __syncthreads();
        if (rs < RS) {
#pragma unroll 1
            for (int ly = rs; ly < TILE; ly += RS) {
#pragma unroll 1
                for (int lx = 0; lx < TILE; lx += 4) {
                    float hv[3][6];
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const float* row = tile + c * PL + (ly + r) * ROW + lx;
                        const float4 a = *reinterpret_cast<const float4*>(row);
                        const float2 b = *reinterpret_cast<const float2*>(row + 4);
                        hv[r][0] = a.x; hv[r][1] = a.y; hv[r][2] = a.z; hv[r][3] = a.w; hv[r][4] = b.x; hv[r][5] = b.y;
                    }
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const float4* g4 = reinterpret_cast<const float4*>(gt + (ly * TILE + lx + p) * GP + og * OT);
#pragma unroll
                        for (int j = 0; j < OT / 4; ++j) {
                            const float4 g = g4[j];
#pragma unroll
                            for (int k = 0; k < 9; ++k) {
                                const float2 vv = make_float2(hv[k / 3][p + k % 3], hv[k / 3][p + k % 3]);
                                acc[k][2 * j] = ffma2(make_float2(g.x, g.y), vv, acc[k][2 * j]);
                                acc[k][2 * j + 1] = ffma2(make_float2(g.z, g.w), vv, acc[k][2 * j + 1]);
                            }
                        }
                    }
                }
            }
        }
        for (int p = tid / COP; p < TILE * TILE; p += NTH / COP) bacc += gt[p * GP + tid % COP];
    }
    // the shares of a row-split are added one after the other: sm[(o * CI + c) * 9 + k]
    float* mine = part + size_t(blockIdx.x) * (CO * CI * 9 + CO);
#pragma unroll 1
    for (int r = RS - 1; r >= 0; --r) {
        __syncthreads();
        if (rs == r) {
#pragma unroll
            for (int j = 0; j < OT; ++j) {
                const int o = og * OT + j;
                if (o < CO) {
#pragma unroll
                    for (int k = 0; k < 9; ++k) {
                        const int at = (o * CI + c) * 9 + k;
                        const float v = j % 2 ? acc[k][j / 2].y : acc[k][j / 2].x;
                        sm[at] = r == RS - 1 ? v : sm[at] + v;
                    }
                }
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < CO * CI * 9; i += NTH) mine[i] = sm[i];
    __syncthreads();
    sm[tid] = bacc;
    __syncthreads();
    if (tid < CO) {
        float b = 0.f;
        for (int p = tid; p < NTH; p += COP) b += sm[p];
        mine[CO * CI * 9 + tid] = b;
    }
}

// g[i] = sum over the rows of part of parameter i of the packed gradient
// vector.  Layer l's rows (rows[l] of them, each as long as the layer's
// parameters) start at part + max_rows * woff[l].  32 parameters per CTA, eight
// threads each with every eighth row.
struct GradRows {
    int rows[NL];
};
__global__ void reduce_grads(const float* part, GradRows gr, int max_rows, int n, float* g) {
    lbk::chain_begin();
    __shared__ float red[8][33];
    const int i = blockIdx.x * 32 + threadIdx.x % 32, share = threadIdx.x / 32;
    float s = 0.f;
    lbk::static_for<0, NL>([&](auto K) {
        constexpr int l = decltype(K)::value, at = layer_offset(l), len = CH[l + 1] * CH[l] * 9 + CH[l + 1];
        if (i >= at && i < at + len) {
            const float* p = part + size_t(max_rows) * at + (i - at);
#pragma unroll 8
            for (int r = share; r < gr.rows[l]; r += 8) s += p[size_t(r) * len];
        }
    });
    red[share][threadIdx.x % 32] = s;
    __syncthreads();
    if (share == 0 && i < n) {
        float t = red[0][threadIdx.x];
        for (int k = 1; k < 8; ++k) t += red[k][threadIdx.x];
        g[i] = t;
    }
}

template <int CI, int CO>
constexpr size_t smem_conv() { return size_t(CI * PLANE + CI * 9 * ((CO + 3) / 4 * 4)) * 4; }
template <int CI, int CO>
constexpr size_t smem_bwd_w() {
    constexpr int cop = (CO + 3) / 4 * 4;
    return size_t(CI * (PLANE + 4) + TILE * TILE * (cop == 32 ? cop + 4 : cop)) * 4;
}

// Offsets of a layer's packed fp16 weights: forward [C_in][9][C_out padded to a
// multiple of 4], backward [C_out][9 taps mirrored][C_in] (not for layer 0).
struct Packing {
    int woff[NL], ffwd[NL], fbwd[NL], total;
};
constexpr int pad4(int v) { return (v + 3) / 4 * 4; }
constexpr Packing make_packing() {
    Packing k{};
    int p = 0, f = 0;
    for (int l = 0; l < NL; ++l) {
        k.woff[l] = p;
        p += CH[l + 1] * CH[l] * 9 + CH[l + 1];
        k.ffwd[l] = f;
        f += CH[l] * 9 * pad4(CH[l + 1]);
        k.fbwd[l] = f;
        if (l > 0) f += CH[l + 1] * 9 * pad4(CH[l]);
    }
    k.total = f;
    return k;
}
constexpr Packing PACK = make_packing();

// Rounds parameter i (index in the packed master vector) to fp16 into its
// forward and backward places; biases stay float32.
__device__ __forceinline__ void store_packed(__half* w16, int i, float v) {
    lbk::static_for<0, NL>([&](auto K) {
        constexpr int l = decltype(K)::value, ci = CH[l], co = CH[l + 1], at = PACK.woff[l], nw = co * ci * 9;
        constexpr int ff = PACK.ffwd[l], fb = PACK.fbwd[l];
        if (i >= at && i < at + nw) {
            const int r = i - at, o = r / (ci * 9), c = r / 9 % ci, k = r % 9;
            const __half hv = __float2half_rn(v);
            w16[ff + (c * 9 + k) * pad4(co) + o] = hv;
            if (l > 0) w16[fb + (o * 9 + 8 - k) * pad4(ci) + c] = hv;
        }
    });
}

__global__ void pack_weights(const float* p, __half* w16, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) store_packed(w16, i, p[i]);
}

__global__ void adam_pack(float* w, __half* w16, const float* g, float* m, float* v, int n, float lr, float b1, float b2,
                          float eps, float c1, float c2) {
    lbk::chain_begin();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        store_packed(w16, i, adam_one(w, g, m, v, i, lr, b1, b2, eps, c1, c2));
}

// Minibatch of samples order[0..batch): their inputs and targets gathered in one
// launch (two copies per sample and minibatch cost more than the kernels of the
// thin layers).
__global__ void gather_batch(const float* x, const float* t, const int* order, size_t nx, size_t nt, float* bx, float* bt) {
    lbk::chain_begin();
    const float* sx = x + size_t(order[blockIdx.y]) * nx;
    const float* st = t + size_t(order[blockIdx.y]) * nt;
    float* dx = bx + size_t(blockIdx.y) * nx;
    float* dt = bt + size_t(blockIdx.y) * nt;
    const size_t i0 = blockIdx.x * size_t(blockDim.x) + threadIdx.x, step = size_t(gridDim.x) * blockDim.x;
    for (size_t i = i0; i < nx; i += step) dx[i] = sx[i];
    for (size_t i = i0; i < nt; i += step) dt[i] = st[i];
}

}  // namespace

struct lb_ws {
    int nparams = 0;
    int woff[NL], boff[NL];         // offsets of W_l and b_l in the packed parameter vector
    float* p = nullptr;             // float32 master parameters (packed)
    __half* p16 = nullptr;          // fp16 copies of the weights in the kernels' layouts (PACK)
    float* g = nullptr;             // gradients
    float* m = nullptr;
    float* v = nullptr;
    double* loss = nullptr;
    float* part = nullptr;          // partial gradients: 2 sms rows per layer (first loss_grad)
    GradRows rows{};                // rows written by the current backward pass
    int sms = 1;
    int adam_t = 0;
    // activations of the current batch
    float* act[NL + 1] = {};
    float* dact[NL + 1] = {};
    size_t cap = 0;                 // pixels x batch capacity of the activation buffers
    cudaStream_t st = nullptr;
};

namespace {

lb_status ensure_acts(lb_ws* w, size_t pix) {
    if (pix <= w->cap) return LB_OK;
    for (int l = 0; l <= NL; ++l) {
        cudaFree(w->act[l]);
        cudaFree(w->dact[l]);
        w->act[l] = w->dact[l] = nullptr;
    }
    for (int l = 0; l <= NL; ++l) {
        if (cudaMalloc(&w->act[l], pix * CH[l] * sizeof(float)) != cudaSuccess ||
            cudaMalloc(&w->dact[l], pix * CH[l] * sizeof(float)) != cudaSuccess)
            return fail(LB_ENOMEM, "warm-start activations");
    }
    w->cap = pix;
    return LB_OK;
}

dim3 conv_grid(int n, int H, int Wd) { return dim3((Wd + TILE - 1) / TILE, (H + TILE - 1) / TILE, n); }

// pixels x channels of a thread: 4 x 8 for 32 channels out, 1 x 4 for the few of the last layer
template <int CI, int CO, bool TANH>
constexpr auto fwd_kernel = conv_tile<CI, CO, CO == 32 ? 4 : 1, CO == 32 ? 8 : 4, false, TANH>;
template <int CI, int CO>   // CI, CO of the layer: CO channels in, CI out
constexpr auto bwd_kernel = conv_tile<CO, CI, 4, 8, true, false>;
template <int CI, int CO>
constexpr auto wgt_kernel = conv_bwd_weight<CI, CO, CO == 32 ? 8 : 4, CI == 32 && CO == 32 ? 2 : 8>;

template <int CI, int CO, bool T>
void launch_fwd(const lb_ws* w, int l, int n, int H, int Wd) {
    lbk::launch_chained(fwd_kernel<CI, CO, T>, conv_grid(n, H, Wd), NTH, smem_conv<CI, CO>(), w->st, w->act[l],
                        w->p16 + PACK.ffwd[l], w->p + w->boff[l], nullptr, w->act[l + 1], H, Wd);
}

template <int CI, int CO>
void launch_bwd(lb_ws* w, int l, int n, int H, int Wd) {
    const int ntiles = n * ((Wd + TILE - 1) / TILE) * ((H + TILE - 1) / TILE);
    w->rows.rows[l] = ntiles < 2 * w->sms ? ntiles : 2 * w->sms;
    lbk::launch_chained(wgt_kernel<CI, CO>, w->rows.rows[l], NTH, smem_bwd_w<CI, CO>(), w->st, w->act[l], w->dact[l + 1],
                        w->part + size_t(2 * w->sms) * w->woff[l], n, H, Wd);
    if constexpr (CI == LB_WS_HIDDEN)
        lbk::launch_chained(bwd_kernel<CI, CO>, conv_grid(n, H, Wd), NTH, smem_conv<CO, CI>(), w->st, w->dact[l + 1],
                            w->p16 + PACK.fbwd[l], nullptr, w->act[l], w->dact[l], H, Wd);
}

// Dynamic shared memory limits of the kernels, on the current device.
template <class K>
cudaError_t allow(K k, size_t bytes) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
}
cudaError_t allow_smem() {
    constexpr int I = LB_WS_IN, M = LB_WS_HIDDEN, O = LB_WS_OUT;
    cudaError_t e;
    if ((e = allow(fwd_kernel<I, M, true>, smem_conv<I, M>())) != cudaSuccess ||
        (e = allow(fwd_kernel<M, M, true>, smem_conv<M, M>())) != cudaSuccess ||
        (e = allow(fwd_kernel<M, O, false>, smem_conv<M, O>())) != cudaSuccess ||
        (e = allow(bwd_kernel<M, M>, smem_conv<M, M>())) != cudaSuccess ||
        (e = allow(bwd_kernel<M, O>, smem_conv<O, M>())) != cudaSuccess ||
        (e = allow(wgt_kernel<I, M>, smem_bwd_w<I, M>())) != cudaSuccess ||
        (e = allow(wgt_kernel<M, M>, smem_bwd_w<M, M>())) != cudaSuccess)
        return e;
    return allow(wgt_kernel<M, O>, smem_bwd_w<M, O>());
}

// The sample index is the grid's z dimension: at most 65535 samples per launch.
constexpr int MAX_SAMPLES = 65535;

cudaError_t forward(lb_ws* w, int n, int H, int Wd) {
    launch_fwd<LB_WS_IN, LB_WS_HIDDEN, true>(w, 0, n, H, Wd);
    launch_fwd<LB_WS_HIDDEN, LB_WS_HIDDEN, true>(w, 1, n, H, Wd);
    launch_fwd<LB_WS_HIDDEN, LB_WS_HIDDEN, true>(w, 2, n, H, Wd);
    launch_fwd<LB_WS_HIDDEN, LB_WS_OUT, false>(w, 3, n, H, Wd);
    return cudaGetLastError();
}

// A launch of the training loop that was refused; the error is reported, not left for the next call.
lb_status launch_failed(cudaError_t e) {
    cudaGetLastError();
    return fail(LB_ECUDA, std::string("training launch: ") + cudaGetErrorString(e));
}

// loss (added to *d_loss, zeroed by the caller) and gradients of the batch whose inputs sit in act[0], targets in t
lb_status loss_grad(lb_ws* w, const float* t, int n, int H, int Wd, double* d_loss) {
    if (!w->part && cudaMalloc(&w->part, size_t(2 * w->sms) * w->nparams * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        w->part = nullptr;
        return fail(LB_ENOMEM, "partial gradients");
    }
    cudaGetLastError();   // an error that an earlier call of the program left is not this one's
    cudaError_t e = forward(w, n, H, Wd);
    if (e != cudaSuccess) return fail(LB_ECUDA, std::string("warm-start forward launch: ") + cudaGetErrorString(e));
    const size_t nout = size_t(n) * LB_WS_OUT * H * Wd;
    lbk::launch_chained(mse_grad, 256, 256, 0, w->st, w->act[4], t, w->dact[4], nout, d_loss);
    launch_bwd<LB_WS_HIDDEN, LB_WS_OUT>(w, 3, n, H, Wd);
    launch_bwd<LB_WS_HIDDEN, LB_WS_HIDDEN>(w, 2, n, H, Wd);
    launch_bwd<LB_WS_HIDDEN, LB_WS_HIDDEN>(w, 1, n, H, Wd);
    launch_bwd<LB_WS_IN, LB_WS_HIDDEN>(w, 0, n, H, Wd);
    lbk::launch_chained(reduce_grads, (w->nparams + 31) / 32, 256, 0, w->st, w->part, w->rows, 2 * w->sms, w->nparams, w->g);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(LB_ECUDA, std::string("warm-start backward: ") + cudaGetErrorString(e));
    return LB_OK;
}

}  // namespace

extern "C" {

lb_status lb_ws_create(int seed, void* cuda_stream, lb_ws** out) {
    if (!out) return fail(LB_EINVAL, "null output");
    lb_ws* w = new (std::nothrow) lb_ws();
    if (!w) return fail(LB_ENOMEM, "host allocation");
    w->st = static_cast<cudaStream_t>(cuda_stream);
    int off = 0;
    for (int l = 0; l < NL; ++l) {
        w->woff[l] = off;
        off += CH[l + 1] * CH[l] * 9;
        w->boff[l] = off;
        off += CH[l + 1];
    }
    w->nparams = off;
    // W ~ U(-s, s), s = 1/sqrt(9 C_in), from a SplitMix64 stream; b = 0
    std::vector<float> h(off, 0.f);
    unsigned long long st = (unsigned long long)seed;
    for (int l = 0; l < NL; ++l) {
        const double s = 1.0 / std::sqrt(9.0 * CH[l]);
        for (int i = 0; i < CH[l + 1] * CH[l] * 9; ++i) h[w->woff[l] + i] = float((2.0 * splitmix_u01(st) - 1.0) * s);
    }
    cudaError_t e;
    if ((e = cudaMalloc(&w->p, off * sizeof(float))) != cudaSuccess || (e = cudaMalloc(&w->p16, PACK.total * sizeof(__half))) != cudaSuccess ||
        (e = cudaMalloc(&w->g, off * sizeof(float))) != cudaSuccess || (e = cudaMalloc(&w->m, off * sizeof(float))) != cudaSuccess ||
        (e = cudaMalloc(&w->v, off * sizeof(float))) != cudaSuccess || (e = cudaMalloc(&w->loss, sizeof(double))) != cudaSuccess) {
        lb_ws_destroy(w);
        return fail(LB_ENOMEM, std::string("warm-start parameters: ") + cudaGetErrorString(e));
    }
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&w->sms, cudaDevAttrMultiProcessorCount, dev);
    if ((e = allow_smem()) != cudaSuccess || (e = cudaMemsetAsync(w->p16, 0, PACK.total * sizeof(__half), w->st)) != cudaSuccess) {
        lb_ws_destroy(w);
        return fail(LB_ECUDA, std::string("warm-start kernels: ") + cudaGetErrorString(e));
    }
    lb_status s = lb_ws_set_params(w, h.data(), size_t(off));
    if (s != LB_OK) { lb_ws_destroy(w); return s; }
    *out = w;
    return LB_OK;
}

lb_status lb_ws_destroy(lb_ws* w) {
    if (!w) return LB_OK;
    cudaStreamSynchronize(w->st);
    cudaFree(w->p);
    cudaFree(w->p16);
    cudaFree(w->g);
    cudaFree(w->m);
    cudaFree(w->v);
    cudaFree(w->loss);
    cudaFree(w->part);
    for (int l = 0; l <= NL; ++l) {
        cudaFree(w->act[l]);
        cudaFree(w->dact[l]);
    }
    delete w;
    return LB_OK;
}

lb_status lb_ws_num_params(const lb_ws* w, long long* n) {
    if (!w || !n) return fail(LB_EINVAL, "null argument");
    *n = w->nparams;
    return LB_OK;
}

lb_status lb_ws_set_params(lb_ws* w, const float* params, size_t count) {
    if (!w || !params || count != size_t(w->nparams)) return fail(LB_EINVAL, "parameter count mismatch");
    cudaError_t e = cudaMemcpyAsync(w->p, params, count * sizeof(float), cudaMemcpyHostToDevice, w->st);
    if (e == cudaSuccess) {
        pack_weights<<<64, 256, 0, w->st>>>(w->p, w->p16, int(count));
        e = cudaMemsetAsync(w->m, 0, count * sizeof(float), w->st);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(w->v, 0, count * sizeof(float), w->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->st);
    w->adam_t = 0;
    return e == cudaSuccess ? LB_OK : fail(LB_ECUDA, std::string("set params: ") + cudaGetErrorString(e));
}

lb_status lb_ws_get_params(lb_ws* w, float* params, size_t count) {
    if (!w || !params || count != size_t(w->nparams)) return fail(LB_EINVAL, "parameter count mismatch");
    cudaError_t e = cudaMemcpyAsync(params, w->p, count * sizeof(float), cudaMemcpyDeviceToHost, w->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->st);
    return e == cudaSuccess ? LB_OK : fail(LB_ECUDA, std::string("get params: ") + cudaGetErrorString(e));
}

lb_status lb_ws_forward(lb_ws* w, const float* x, int n, int H, int Wd, float* y) {
    if (!w || !x || !y || n < 1 || n > MAX_SAMPLES || H < 1 || Wd < 1) return fail(LB_EINVAL, "bad arguments");
    const size_t pix = size_t(n) * H * Wd;
    lb_status s = ensure_acts(w, pix);
    if (s != LB_OK) return s;
    cudaError_t e = cudaMemcpyAsync(w->act[0], x, pix * LB_WS_IN * sizeof(float), cudaMemcpyHostToDevice, w->st);
    if (e != cudaSuccess) return fail(LB_ECUDA, "upload");
    if ((e = forward(w, n, H, Wd)) != cudaSuccess)
        return fail(LB_ECUDA, std::string("warm-start forward launch: ") + cudaGetErrorString(e));
    e = cudaMemcpyAsync(y, w->act[4], pix * LB_WS_OUT * sizeof(float), cudaMemcpyDeviceToHost, w->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->st);
    return e == cudaSuccess ? LB_OK : fail(LB_ECUDA, std::string("warm-start forward: ") + cudaGetErrorString(e));
}

lb_status lb_ws_loss_grad(lb_ws* w, const float* x, const float* t, int n, int H, int Wd, double* loss,
                          float* grads) {
    if (!w || !x || !t || n < 1 || n > MAX_SAMPLES || H < 1 || Wd < 1) return fail(LB_EINVAL, "bad arguments");
    const size_t pix = size_t(n) * H * Wd;
    lb_status s = ensure_acts(w, pix);
    if (s != LB_OK) return s;
    float* dt = nullptr;
    if (cudaMalloc(&dt, pix * LB_WS_OUT * sizeof(float)) != cudaSuccess) return fail(LB_ENOMEM, "targets");
    cudaMemcpyAsync(w->act[0], x, pix * LB_WS_IN * sizeof(float), cudaMemcpyHostToDevice, w->st);
    cudaMemcpyAsync(dt, t, pix * LB_WS_OUT * sizeof(float), cudaMemcpyHostToDevice, w->st);
    cudaMemsetAsync(w->loss, 0, sizeof(double), w->st);
    s = loss_grad(w, dt, n, H, Wd, w->loss);
    if (s == LB_OK && (loss || grads)) {
        cudaError_t e = cudaSuccess;
        if (loss) e = cudaMemcpyAsync(loss, w->loss, sizeof(double), cudaMemcpyDeviceToHost, w->st);
        if (e == cudaSuccess && grads)
            e = cudaMemcpyAsync(grads, w->g, size_t(w->nparams) * sizeof(float), cudaMemcpyDeviceToHost, w->st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(w->st);
        if (e != cudaSuccess) s = fail(LB_ECUDA, std::string("loss and gradient download: ") + cudaGetErrorString(e));
    }
    cudaFree(dt);
    return s;
}

lb_status lb_ws_train(lb_ws* w, const float* x, const float* t, int n, int H, int Wd, int epochs, int batch,
                      float lr, int seed, double* loss_history) {
    if (!w || !x || !t || n < 1 || H < 1 || Wd < 1 || epochs < 1 || batch < 1) return fail(LB_EINVAL, "bad arguments");
    batch = batch < n ? batch : n;
    if (batch > MAX_SAMPLES) return fail(LB_EINVAL, "batch larger than 65535 samples");
    const size_t img = size_t(H) * Wd;
    lb_status s = ensure_acts(w, size_t(batch) * img);
    if (s != LB_OK) return s;
    // the data set, the minibatch's targets, the epoch's sample order and the loss of each of its minibatches
    const int nb = n / batch;
    std::vector<int> order;
    std::vector<double> losses;
    try {
        order.resize(n);
        losses.resize(nb);
    } catch (...) {
        return fail(LB_ENOMEM, "training order");
    }
    float *dx = nullptr, *dt = nullptr, *bt = nullptr;
    int* d_order = nullptr;
    double* d_loss = nullptr;
    auto release = [&] {
        cudaFree(dx);
        cudaFree(dt);
        cudaFree(bt);
        cudaFree(d_order);
        cudaFree(d_loss);
    };
    if (cudaMalloc(&dx, size_t(n) * img * LB_WS_IN * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&dt, size_t(n) * img * LB_WS_OUT * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&bt, size_t(batch) * img * LB_WS_OUT * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&d_order, size_t(n) * sizeof(int)) != cudaSuccess ||
        cudaMalloc(&d_loss, size_t(nb) * sizeof(double)) != cudaSuccess) {
        release();
        return fail(LB_ENOMEM, "training data");
    }
    cudaMemcpyAsync(dx, x, size_t(n) * img * LB_WS_IN * sizeof(float), cudaMemcpyHostToDevice, w->st);
    cudaMemcpyAsync(dt, t, size_t(n) * img * LB_WS_OUT * sizeof(float), cudaMemcpyHostToDevice, w->st);
    for (int i = 0; i < n; ++i) order[i] = i;
    unsigned long long rs = (unsigned long long)seed * 0x9E3779B97F4A7C15ull + 1;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const dim3 ggrid(unsigned(std::min<size_t>((img * LB_WS_IN + 1023) / 1024, 64)), unsigned(batch));
    cudaError_t e = cudaSuccess;
    for (int ep = 0; ep < epochs && s == LB_OK; ++ep) {
        for (int i = n - 1; i > 0; --i) {   // shuffle (xorshift)
            rs ^= rs << 13; rs ^= rs >> 7; rs ^= rs << 17;
            std::swap(order[i], order[int(rs % (unsigned long long)(i + 1))]);
        }
        // one upload and one read-back per epoch: nothing waits between its minibatches
        e = cudaMemcpyAsync(d_order, order.data(), size_t(n) * sizeof(int), cudaMemcpyHostToDevice, w->st);
        if (e == cudaSuccess) e = cudaMemsetAsync(d_loss, 0, size_t(nb) * sizeof(double), w->st);
        if (e != cudaSuccess) {
            s = fail(LB_ECUDA, std::string("training: ") + cudaGetErrorString(e));
            break;
        }
        for (int k = 0; k < nb && s == LB_OK; ++k) {
            e = lbk::launch_chained(gather_batch, ggrid, 256, 0, w->st, dx, dt, d_order + size_t(k) * batch,
                                    img * LB_WS_IN, img * LB_WS_OUT, w->act[0], bt);
            s = e == cudaSuccess ? loss_grad(w, bt, batch, H, Wd, d_loss + k) : launch_failed(e);
            if (s != LB_OK) break;   // no optimiser step without a gradient
            ++w->adam_t;
            const float c1 = 1.f - std::pow(b1, float(w->adam_t)), c2 = 1.f - std::pow(b2, float(w->adam_t));
            e = lbk::launch_chained(adam_pack, 128, 256, 0, w->st, w->p, w->p16, w->g, w->m, w->v, w->nparams, lr, b1, b2,
                                    eps, c1, c2);
            if (e != cudaSuccess) s = launch_failed(e);
        }
        if (s != LB_OK) break;
        e = cudaMemcpyAsync(losses.data(), d_loss, size_t(nb) * sizeof(double), cudaMemcpyDeviceToHost, w->st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(w->st);
        if (e != cudaSuccess) {
            s = fail(LB_ECUDA, std::string("warm-start loss: ") + cudaGetErrorString(e));
            break;
        }
        double ep_loss = 0.0;
        for (double l : losses) ep_loss += l;
        if (loss_history) loss_history[ep] = nb ? ep_loss / nb : 0.0;
    }
    e = cudaStreamSynchronize(w->st);
    release();
    if (s == LB_OK && e != cudaSuccess) s = fail(LB_ECUDA, std::string("training: ") + cudaGetErrorString(e));
    return s;
}

lb_status lb_ws_predict_sym(lb_ws* w, const float* x, int H, int Wd, float* y) {
    if (!w || !x || !y || H < 1 || Wd < 1) return fail(LB_EINVAL, "bad arguments");
    // group of the periodic lattice fixing the point (W/2, H/2): reflections
    // x -> (W - x) mod W, y -> (H - y) mod H and, on square grids, the transpose.
    const int ng = (H == Wd) ? 8 : 4;
    const size_t N = size_t(H) * Wd;
    std::vector<float> xs(size_t(ng) * LB_WS_IN * N), ys(size_t(ng) * LB_WS_OUT * N);
    std::vector<int> perm(size_t(ng) * N);
    int A[8][2][2];
    for (int g = 0; g < ng; ++g) {
        const int fx = g & 1, fy = (g >> 1) & 1, tr = (g >> 2) & 1;
        // coordinate map p -> g(p): optional transpose, then the reflections
        int M[2][2] = {{1, 0}, {0, 1}};
        if (tr) { M[0][0] = 0; M[0][1] = 1; M[1][0] = 1; M[1][1] = 0; }
        for (int j = 0; j < 2; ++j) {
            if (fx) M[0][j] = -M[0][j];
            if (fy) M[1][j] = -M[1][j];
        }
        std::memcpy(A[g], M, sizeof(M));
        for (int yy = 0; yy < H; ++yy)
            for (int xx = 0; xx < Wd; ++xx) {
                int sx = tr ? yy : xx, sy = tr ? xx : yy;
                if (fx) sx = (Wd - sx) % Wd;
                if (fy) sy = (H - sy) % H;
                perm[size_t(g) * N + size_t(yy) * Wd + xx] = sy * Wd + sx;
            }
        for (int c = 0; c < LB_WS_IN; ++c)
            for (size_t p = 0; p < N; ++p)
                xs[(size_t(g) * LB_WS_IN + c) * N + p] = x[size_t(c) * N + perm[size_t(g) * N + p]];
    }
    lb_status st = lb_ws_forward(w, xs.data(), ng, H, Wd, ys.data());
    if (st != LB_OK) return st;
    std::fill(y, y + size_t(LB_WS_OUT) * N, 0.f);
    for (int g = 0; g < ng; ++g) {
        const float* yg = ys.data() + size_t(g) * LB_WS_OUT * N;
        for (size_t p = 0; p < N; ++p) {
            const size_t q = size_t(perm[size_t(g) * N + p]);
            const float ux = yg[N + p], uy = yg[2 * N + p];
            y[q] += yg[p] / ng;                                             // scalar channel
            y[N + q] += (A[g][0][0] * ux + A[g][0][1] * uy) / ng;           // u(g p) = A u_g(p)
            y[2 * N + q] += (A[g][1][0] * ux + A[g][1][1] * uy) / ng;
        }
    }
    return LB_OK;
}

lb_status lb_ws_features(int nx, int ny, const double* rho_tanh, double rho_l, double rho_g, double T, double kappa,
                         double tau, double R, float* x) {
    if (!rho_tanh || !x || nx < 1 || ny < 1 || !(rho_l > rho_g) || !(R > 0)) return fail(LB_EINVAL, "bad arguments");
    const size_t N = size_t(nx) * ny;
    const double mid = 0.5 * (rho_l + rho_g), span = rho_l - rho_g;
    const float planes[4] = {float((T - 0.53) / 0.03), float((kappa - 0.016) / 0.014), float((tau - 1.05) / 0.45),
                             float(10.0 / R)};
    for (size_t i = 0; i < N; ++i) {
        x[i] = float((rho_tanh[i] - mid) / span);
        for (int c = 0; c < 4; ++c) x[(c + 1) * N + i] = planes[c];
    }
    return LB_OK;
}

lb_status lb_ws_decode(int nx, int ny, const double* rho_tanh, double rho_l, double rho_g, const float* y, double* rho,
                       double* u) {
    if (!rho_tanh || !y || nx < 1 || ny < 1 || !(rho_l > rho_g)) return fail(LB_EINVAL, "bad arguments");
    const size_t N = size_t(nx) * ny;
    const double span = rho_l - rho_g, mid = 0.5 * (rho_l + rho_g);
    // The prediction must describe the same drop: its mass is the tanh start's.
    // The mass residual of the predicted correction is removed with weight
    // 1 - 4c^2 (c the normalised tanh density), i.e. inside the interface.
    double dm = 0.0, wsum = 0.0;
    for (size_t i = 0; i < N; ++i) {
        const double c = (rho_tanh[i] - mid) / span;
        dm += double(y[i]);
        wsum += std::max(0.0, 1.0 - 4.0 * c * c);
    }
    const double shift = wsum > 0 ? dm / wsum : 0.0;
    for (size_t i = 0; i < N; ++i) {
        const double c = (rho_tanh[i] - mid) / span;
        const double corr = double(y[i]) - shift * std::max(0.0, 1.0 - 4.0 * c * c);
        if (rho) rho[i] = rho_tanh[i] + span * corr;
        if (u) {
            u[i] = 1e-3 * double(y[N + i]);
            u[N + i] = 1e-3 * double(y[2 * N + i]);
        }
    }
    return LB_OK;
}

}  // extern "C"
