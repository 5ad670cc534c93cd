// fastmemb.cu - FastMemb in dense form on CUDA cores (FP32), one kernel per convolution.
//
// The network (Sec. 2.2, "A lightweight network architecture"): three [conv 4x4 -> max-out over
// 2 -> 2x2 stride-2 max-pool] stages, no transfer function, then conv 4x4 to two classes and a
// softmax. Dense computation (Sec. 2.2, "Accelerating dense computation") turns each stride-2
// pool into a stride-1 max-filter plus 2-factor sub-sampling; here that becomes a max-filter
// with dilation d and a conv with dilation 2d behind it (d = 1, 2, 4; the head has dilation 8).
//
// The convolution kernel (fm_conv.cuh) tiles each dilated conv by the paper's max-pooling
// fragments: a conv with dilation d restricted to one residue class (y mod d, x mod d) is a plain
// 4x4 conv on the d-strided sub-grid, so every CTA keeps the register reuse of an undilated conv.
// The previous stage's dilated max-filter is applied while staging; epilogues are max-out of
// adjacent channel pairs or the 2-class softmax p = 1 / (1 + exp(z0 - z1)).
//
// Domains for an output region rows x cols (radius 26):
//   conv1 out (rows+49)^2 .. conv2 out (rows+42) .. conv3 out (rows+28) .. head out rows
//   (each conv removes 3d, each max-filter d).
// Sub-sampled output (factor 2: the dense map at even rows and columns, the fragment tree of
// Sec. 2.2 pruned at the first pool): conv1 at full resolution on (2H2+48)^2, then a 2x2
// stride-2 max-pool (read while staging, source stride 2) and the remaining stages on the half
// grid with dilations 1, 2, 4: conv2 out H2+21, conv3 out H2+14, head out H2 = ceil(rows/2).
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "fm_conv.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace mb {


// Per-stage geometry of one FastMemb pass with NC convolutions (4 for FastMemb, 5 for
// FastMemb_3nm): extents of the conv outputs (conv1 at full resolution; the rest at full resolution
// for the dense map, on the half grid when sub-sampled), the dilation of each conv, and how each
// conv reads its input (max-filter dilation dm, stride st). Walking back from the map, conv k's
// input needs 3 d_k + dm_k more rows than its output.
constexpr int kFmMaxConvs = 5;
struct FmGeom {
    int nc;
    int64_t r[kFmMaxConvs], c[kFmMaxConvs];
    int d[kFmMaxConvs], dm[kFmMaxConvs], st[kFmMaxConvs];
};

static FmGeom fm_geom(int nc, int64_t rows, int64_t cols, int sub) {
    FmGeom g{};
    g.nc = nc;
    for (int k = 0; k < nc; ++k) {
        g.st[k] = 1;
        if (sub == 2) {
            g.d[k] = k == 0 ? 1 : 1 << (k - 1);
            g.dm[k] = k == 0 ? 0 : (k == 1 ? 1 : g.d[k - 1]);
            if (k == 1) g.st[k] = 2;
        } else {
            g.d[k] = 1 << k;
            g.dm[k] = k == 0 ? 0 : g.d[k - 1];
        }
    }
    g.r[nc - 1] = sub == 2 ? (rows + 1) / 2 : rows;
    g.c[nc - 1] = sub == 2 ? (cols + 1) / 2 : cols;
    for (int k = nc - 1; k >= 1; --k) {
        const int64_t in_r = g.r[k] + 3 * g.d[k], in_c = g.c[k] + 3 * g.d[k];  // conv k's input domain
        g.r[k - 1] = (in_r - 1) * g.st[k] + g.dm[k] + 1;
        g.c[k - 1] = (in_c - 1) * g.st[k] + g.dm[k] + 1;
    }
    if (sub == 2) {  // conv1 covers whole 2x2 pooling windows
        g.r[0] += g.r[0] & 1;
        g.c[0] += g.c[0] & 1;
    }
    return g;
}

// Input domain of conv i >= 1: the (max-filtered, strided) view of conv i-1's output: positions r
// with st r + dm inside the source.
static inline int64_t fm_in_extent(const FmGeom& g, int i, bool rows) {
    const int64_t src = rows ? g.r[i - 1] : g.c[i - 1];
    return (src - 1 - g.dm[i]) / g.st[i] + 1;
}

// Offsets of the SIMT-layout weights of conv k (Wt[ci][ky][kx][co] then b[co]; co = 64 except the
// head's 2; ci = 1 for conv1 and 32 after).
static const float* fm_simt_w(const mb_net* net, int k, int nc, const float** bias) {
    size_t off = 0;
    for (int i = 0; i < k; ++i) off += i == 0 ? 16 * 64 + 64 : 32 * 16 * 64 + 64;
    const float* w = net->d_simt + off;
    const int co = k == nc - 1 ? 2 : 64, ci = k == 0 ? 1 : 32;
    *bias = w + (size_t)ci * 16 * co;
    return w;
}

mb_status simt_fastmemb_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w, int64_t in_pitch,
                               int64_t in_slice, int64_t y0, int64_t x0, int64_t rows, int64_t cols, void* out,
                               int64_t out_pitch, int64_t out_slice, mb_out_type ot, cudaStream_t st, int sub) {
    if (z == 0 || rows == 0 || cols == 0) return MB_OK;
    MB_TRY(x3_poll_error(net));
    const int nc = fastmemb_convs(net->family);
    const int R = nc == 5 ? kFastMemb3nmRadius : kFastMembRadius;
    const FmGeom g = fm_geom(nc, rows, cols, sub);
    size_t per = 0;
    for (int k = 0; k < nc - 1; ++k) per += (size_t)(g.r[k] * g.c[k]) * 32 * sizeof(float);
    const size_t budget = (size_t)3 << 30;
    const int64_t zc = std::min<int64_t>(std::min<int64_t>(std::max<size_t>(1, budget / per), 65535), z);
    MB_TRY(net->ws.ensure(per * (size_t)zc));
    float* act[kFmMaxConvs - 1];
    act[0] = static_cast<float*>(net->ws.ptr);
    for (int k = 1; k < nc - 1; ++k) act[k] = act[k - 1] + (size_t)zc * g.r[k - 1] * g.c[k - 1] * 32;
    for (int64_t z0 = 0; z0 < z; z0 += zc) {
        const int nz = (int)std::min<int64_t>(zc, z - z0);
        FmArgs a{};
        a.in = in + z0 * in_slice;
        a.in_slice = in_slice;
        a.in_pitch = in_pitch;
        a.in_rows = (int)(g.r[0] + 3);
        a.in_cols = (int)(g.c[0] + 3);
        a.src_h = (int)h;
        a.src_w = (int)w;
        a.off_y = (int)(y0 - R);
        a.off_x = (int)(x0 - R);
        a.d = 1;
        a.out_h = (int)g.r[0];
        a.out_w = (int)g.c[0];
        a.out = act[0];
        a.out_slice = g.r[0] * g.c[0] * 32;
        a.out_pitch = g.c[0];
        a.wt = fm_simt_w(net, 0, nc, &a.bias);
        MB_TRY((launch_fm<1, 1, 64, 8, FM_IN_U8, FM_OUT_MAXOUT>(a, nz, st)));
        for (int k = 1; k < nc; ++k) {
            FmArgs b{};
            b.in = act[k - 1];
            b.in_slice = g.r[k - 1] * g.c[k - 1] * 32;
            b.in_pitch = g.c[k - 1];
            b.in_rows = (int)fm_in_extent(g, k, true);
            b.in_cols = (int)fm_in_extent(g, k, false);
            b.d = g.d[k];
            b.dm = g.dm[k];
            b.in_stride = g.st[k];
            b.out_h = (int)g.r[k];
            b.out_w = (int)g.c[k];
            b.wt = fm_simt_w(net, k, nc, &b.bias);
            if (k < nc - 1) {
                b.out = act[k];
                b.out_slice = g.r[k] * g.c[k] * 32;
                b.out_pitch = g.c[k];
                if (net->x3_ok) {
                    X3Layer a3{};
                    a3.in = act[k - 1];
                    a3.in_slice = b.in_slice;
                    a3.in_pitch = b.in_pitch;
                    a3.in_rows = b.in_rows;
                    a3.in_cols = b.in_cols;
                    a3.src_cols = g.c[k - 1];
                    a3.d = b.d;
                    a3.dm = b.dm;
                    a3.stride = b.in_stride;
                    a3.out = act[k];
                    a3.out_slice = b.out_slice;
                    a3.out_pitch = b.out_pitch;
                    a3.out_h = b.out_h;
                    a3.out_w = b.out_w;
                    a3.nz = nz;
                    MB_TRY(x3_layer(net, k - 1, a3, st));
                } else {
                    MB_TRY((launch_fm<32, 8, 64, 8, FM_IN_F32, FM_OUT_MAXOUT>(b, nz, st)));
                }
            } else {
                b.out_slice = out_slice;
                b.out_pitch = out_pitch;
                if (ot == MB_OUT_F32) {
                    b.out = static_cast<float*>(out) + z0 * out_slice;
                    MB_TRY((launch_fm<32, 8, 2, 2, FM_IN_F32, FM_OUT_SOFTMAX_F32>(b, nz, st)));
                } else {
                    b.out = static_cast<uint8_t*>(out) + z0 * out_slice;
                    MB_TRY((launch_fm<32, 8, 2, 2, FM_IN_F32, FM_OUT_SOFTMAX_U8>(b, nz, st)));
                }
            }
        }
    }
    return x3_poll_error(net);
}

// Layer 1 of the tensor-core paths: conv 4x4 1 -> 64 from the uint8 slice in FP32, max-out over
// pairs, rounding to the net's 16-bit type, the 2x2 max-filter, and (ST = 2) its stride: features in
// the layout that the next conv's bulk copies read, [slice][row][chunk of 8][column][16 B].
//
// FP32 FMA issue bounds it (2,048 FLOP per conv pixel). A warp walks down a 32-column strip on its
// own; a lane holds all 64 conv channels of its column, packed by channel pairs, so a max-out group
// is one accumulator pair and a pixel's 16-byte chunks are stored whole. The weights are kernel
// parameters, no shared-memory broadcasts beside the FMAs (those took 62 % of the shared-memory pipe
// and left the FMA pipe at 50 %: 528 us). The inputs sit in shared memory duplicated, ready for packed
// FMAs. Tap order and rounding are those of fm_conv, so the features are bitwise the same. 343 us on
// 1024 x 1024 x 8 (FMA pipe 77 % busy, 16 warps of 128 registers); two columns a lane and 8 warps of 248
// took 354 (the max-out, the filter and the stores of 2 warps a scheduler hide less behind FMAs), two
// columns and half the channels a lane 869 (weights at a run-time offset); unpacked FMAs with the
// filter left to the next layer's loads took 534.
struct FmFirstArgs {
    const uint8_t* in;
    int64_t in_slice, in_pitch;
    int src_h, src_w;    // slice size for reflect-101
    int off_y, off_x;    // conv input (r, c) reads slice (refl(r + off_y), refl(c + off_x))
    uint16_t* out;
    int64_t out_slice, out_pitch;  // elements per slice, columns per row
    int rows, cols;      // filtered outputs
    int n_strips;
    int64_t total;       // strip-rows of the launch: nz x n_strips x rows
    float2 w[16][32];    // [4 ky + kx][channel pair]
    float2 b[32];
    WeightsTag tag;      // whether they are still the net's
    const float2* dw;    // else these are read: [16][32], then b[32]
};

constexpr int kFirstPx = 1;                   // columns of a lane
constexpr int kFirstWarps = 16 / kFirstPx;
constexpr int kFirstCols = 32 * kFirstPx + 4; // 3 more inputs per row

__device__ __forceinline__ int refl_clamp(int t, int n) {
    t = t < 0 ? -t : t;
    t = t >= n ? 2 * (n - 1) - t : t;
    return min(max(t, 0), n - 1);  // columns past the last strip's domain feed nothing that is stored
}

template <bool F16>
__device__ __forceinline__ uint32_t pack16(float a, float b) {
    uint32_t u;
    if constexpr (F16) {
        const __half2 v = __floats2half2_rn(a, b);
        u = *reinterpret_cast<const uint32_t*>(&v);
    } else {
        const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
        u = *reinterpret_cast<const uint32_t*>(&v);
    }
    return u;
}

template <bool F16>
__device__ __forceinline__ uint32_t max16(uint32_t a, uint32_t b) {
    if constexpr (F16) {
        const __half2 v = __hmax2(*reinterpret_cast<const __half2*>(&a), *reinterpret_cast<const __half2*>(&b));
        return *reinterpret_cast<const uint32_t*>(&v);
    } else {
        const __nv_bfloat162 v =
            __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
        return *reinterpret_cast<const uint32_t*>(&v);
    }
}

template <bool F16, int ST>
__global__ void __launch_bounds__(32 * kFirstWarps, 1) fm_first(const __grid_constant__ FmFirstArgs a) {
    __shared__ __align__(16) float2 s_x[kFirstWarps][4][kFirstCols];  // a ring of 4 input rows per warp
    ptx::grid_dep_launch();  // the first layer's launch may set itself up on SMs that are done
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float2(*sx)[kFirstCols] = s_x[warp];
    constexpr int kStrip = ST == 1 ? 32 * kFirstPx - 1 : 16 * kFirstPx;  // filtered columns of a strip
    auto run = [&](auto taken) {
        constexpr bool kTaken = decltype(taken)::value;
        constexpr int kTapUnroll = kTaken ? 4 : 1;  // (loads from memory, hoisted over 16 taps, would spill)
        auto bias = [&](int c) { return kTaken ? a.b[c] : __ldg(a.dw + 512 + c); };
        auto weight = [&](int tap, int c) { return kTaken ? a.w[tap][c] : __ldg(a.dw + 32 * tap + c); };
        // one equal contiguous range of strip-rows per warp
        const int64_t n_warps = (int64_t)gridDim.x * kFirstWarps, me = (int64_t)blockIdx.x * kFirstWarps + warp;
        int64_t pos = a.total * me / n_warps;
        const int64_t end = a.total * (me + 1) / n_warps;
        while (pos < end) {
            const int64_t col = pos / a.rows;
            const int y0 = (int)(pos - col * a.rows);
            const int zi = (int)(col / a.n_strips), x0 = (int)(col % a.n_strips) * kStrip;  // filtered coordinates
            const int rows = (int)min((int64_t)(a.rows - y0), end - pos);
            pos += rows;
            const int n_in = (ST == 1 ? rows + 1 : 2 * rows) + 3;  // conv rows + 3
            const uint8_t* src = a.in + (int64_t)zi * a.in_slice;
            constexpr int kIn = kFirstPx + 1;
            int sc[kIn];
#pragma unroll
            for (int i = 0; i < kIn; ++i) sc[i] = refl_clamp(ST * x0 + lane + 32 * i + a.off_x, a.src_w);
            uint8_t u[kIn];
            auto fetch = [&](int r) {  // the bytes of input row r of the item
                const uint8_t* row = src + (int64_t)refl_clamp(ST * y0 + r + a.off_y, a.src_h) * a.in_pitch;
#pragma unroll
                for (int i = 0; i < kIn; ++i) u[i] = __ldg(row + sc[i]);
            };
            uint16_t* out = a.out + (int64_t)zi * a.out_slice;
            uint32_t prev[kFirstPx][16];
#pragma unroll
            for (int i = 0; i < kFirstPx; ++i)
#pragma unroll
                for (int k = 0; k < 16; ++k) prev[i][k] = 0u;
            fetch(0);
#pragma unroll 1
            for (int r = 0; r < n_in; ++r) {
                __syncwarp();  // row r - 4, whose slot is written now, has been read
#pragma unroll
                for (int i = 0; i < kIn; ++i)
                    if (lane + 32 * i < kFirstCols) {
                        const float v = unit_of_byte(u[i]);
                        sx[r & 3][lane + 32 * i] = make_float2(v, v);
                    }
                if (r + 1 < n_in) fetch(r + 1);
                __syncwarp();
                const int yc = r - 3;  // conv row of the item that input row r completes
                if (yc < 0) continue;
                float2 acc[kFirstPx][32];
#pragma unroll
                for (int c = 0; c < 32; ++c)
#pragma unroll
                    for (int i = 0; i < kFirstPx; ++i) acc[i][c] = bias(c);
#pragma unroll kTapUnroll
                for (int ky = 0; ky < 4; ++ky) {
                    const float2* row = sx[(r + 1 + ky) & 3] + lane;  // input row yc + ky
#pragma unroll kTapUnroll
                    for (int kx = 0; kx < 4; ++kx) {
                        float2 x[kFirstPx];
#pragma unroll
                        for (int i = 0; i < kFirstPx; ++i) x[i] = row[kx + 32 * i];
#pragma unroll
                        for (int c = 0; c < 32; ++c)
#pragma unroll
                            for (int i = 0; i < kFirstPx; ++i)
                                acc[i][c] = __ffma2_rn(weight(4 * ky + kx, c), x[i], acc[i][c]);
                    }
                }
                const bool emit = ST == 1 ? yc > 0 : (yc & 1) != 0;
                const int y = ST == 1 ? y0 + yc - 1 : y0 + (yc >> 1);
                uint32_t v[kFirstPx][16];
#pragma unroll
                for (int i = 0; i < kFirstPx; ++i)
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const uint32_t f = pack16<F16>(fmaxf(acc[i][2 * k].x, acc[i][2 * k].y),
                                                       fmaxf(acc[i][2 * k + 1].x, acc[i][2 * k + 1].y));
                        v[i][k] = max16<F16>(prev[i][k], f);
                        prev[i][k] = f;
                    }
                if (!emit) continue;
                // horizontal partner: the next column, in the next lane; of a column group's last it is the next
                // group's first, and the strip's last column has none
#pragma unroll
                for (int k = 0; k < 16; ++k)
#pragma unroll
                    for (int i = 0; i < kFirstPx; ++i) {
                        const uint32_t mine = i + 1 < kFirstPx && lane == 0 ? v[(i + 1) % kFirstPx][k] : v[i][k];
                        v[i][k] = max16<F16>(v[i][k], __shfl_sync(0xffffffffu, mine, (lane + 1) & 31));
                    }
#pragma unroll
                for (int i = 0; i < kFirstPx; ++i) {
                    const int c = lane + 32 * i;  // conv column of the strip
                    const int x = x0 + (ST == 1 ? c : c >> 1);
                    if ((ST == 1 ? c < kStrip : (c & 1) == 0) && x < a.cols) {
                        uint16_t* o = out + ((int64_t)y * 4 * a.out_pitch + x) * 8;
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            *reinterpret_cast<uint4*>(o + (int64_t)q * a.out_pitch * 8) =
                                make_uint4(v[i][4 * q], v[i][4 * q + 1], v[i][4 * q + 2], v[i][4 * q + 3]);
                    }
                }
            }
        }
    };
    // the launch's parameters, or (a captured call replayed after other weights were loaded) device memory
    if (*a.tag.word == a.tag.taken)
        run(std::true_type{});
    else
        run(std::false_type{});
}

template <bool F16, int ST>
static mb_status launch_first(FmFirstArgs a, int nz, cudaStream_t st) {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        MB_CUDA(cudaGetDevice(&dev));
        MB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    }
    constexpr int kStrip = ST == 1 ? 32 * kFirstPx - 1 : 16 * kFirstPx;
    a.n_strips = (a.cols + kStrip - 1) / kStrip;
    a.total = (int64_t)nz * a.n_strips * a.rows;
    // one CTA per SM, or fewer where a warp would get no row (a row costs 2 conv rows at the start of
    // a range, so short ranges cost throughput only where the launch is too small to fill the chip)
    const int64_t want = (a.total + kFirstWarps - 1) / kFirstWarps;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(sms, want));
    fm_first<F16, ST><<<grid, 32 * kFirstWarps, 0, st>>>(a);
    count_launch();
    MB_CUDA(cudaGetLastError());
    return MB_OK;
}

// Tensor-core paths (BF16 or FP16): layer 1 on CUDA cores (FP32 arithmetic, 16-bit out); the 32->64
// dilated convs and the head on the tensor cores (fastmemb_tc.cu). Every layer leaves what the next
// one reads: max-filtered 16-bit features, chunk-planar, rows wide enough for the reader's strips.
mb_status tc_fastmemb_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w, int64_t in_pitch,
                               int64_t in_slice, int64_t y0, int64_t x0, int64_t rows, int64_t cols, void* out,
                               int64_t out_pitch, int64_t out_slice, mb_out_type ot, cudaStream_t st, int sub) {
    if (z == 0 || rows == 0 || cols == 0) return MB_OK;
    MB_TRY(fm_tc_poll_error(net));
    const int nc = fastmemb_convs(net->family);
    const int R = nc == 5 ? kFastMemb3nmRadius : kFastMembRadius;
    const FmGeom g = fm_geom(nc, rows, cols, sub);
    auto up = [](int64_t n) { return (n + 127) & ~(int64_t)127; };  // 256-byte aligned sub-buffers
    // features entering conv k = 1 .. nc-1: fr x fc of them, fp columns apart, n elements per slice
    int64_t fr[kFmMaxConvs], fc[kFmMaxConvs], fp[kFmMaxConvs], n[kFmMaxConvs];
    size_t per = 0;
    for (int k = 1; k < nc; ++k) {
        const bool head = k == nc - 1;
        fr[k] = g.r[k] + 3 * g.d[k];
        fc[k] = g.c[k] + 3 * g.d[k];
        fp[k] = fm_tc_in_pitch(head, head ? g.c[k] : g.c[k + 1] + 3 * g.d[k + 1], g.d[k]);
        n[k] = up(fr[k] * 4 * fp[k] * 8);
        per += (size_t)n[k] * 2;
    }
    const size_t budget = (size_t)3 << 30;
    const int64_t zc = std::min<int64_t>(std::min<int64_t>(std::max<size_t>(1, budget / per), 65535), z);
    MB_TRY(net->ws.ensure(per * (size_t)zc));
    uint16_t* act[kFmMaxConvs];
    act[1] = static_cast<uint16_t*>(net->ws.ptr);
    for (int k = 2; k < nc; ++k) act[k] = act[k - 1] + (size_t)zc * n[k - 1];
    const size_t osz = ot == MB_OUT_F32 ? 4 : 1;
    for (int64_t z0 = 0; z0 < z; z0 += zc) {
        const int nz = (int)std::min<int64_t>(zc, z - z0);
        FmFirstArgs a{};
        a.in = in + z0 * in_slice;
        a.in_slice = in_slice;
        a.in_pitch = in_pitch;
        a.src_h = (int)h;
        a.src_w = (int)w;
        a.off_y = (int)(y0 - R);
        a.off_x = (int)(x0 - R);
        a.out = act[1];
        a.out_slice = n[1];
        a.out_pitch = fp[1];
        a.rows = (int)fr[1];
        a.cols = (int)fc[1];
        const float* db;
        a.tag = WeightsTag{net->d_tag, net->tag};
        a.dw = reinterpret_cast<const float2*>(fm_simt_w(net, 0, nc, &db));
        const float* w1 = net->host_params.data();  // W1[64][1][4][4], b1[64]
        for (int t = 0; t < 16; ++t)
            for (int c = 0; c < 32; ++c) a.w[t][c] = make_float2(w1[32 * c + t], w1[32 * c + 16 + t]);
        for (int c = 0; c < 32; ++c) a.b[c] = make_float2(w1[64 * 16 + 2 * c], w1[64 * 16 + 2 * c + 1]);
        if (net->prec == MB_PREC_FP16)
            MB_TRY((sub == 2 ? launch_first<true, 2>(a, nz, st) : launch_first<true, 1>(a, nz, st)));
        else
            MB_TRY((sub == 2 ? launch_first<false, 2>(a, nz, st) : launch_first<false, 1>(a, nz, st)));
        for (int k = 1; k < nc; ++k) {
            const bool head = k == nc - 1;
            void* o = head ? static_cast<void*>(static_cast<uint8_t*>(out) + z0 * out_slice * osz) : act[k + 1];
            MB_TRY(fm_tc_layer(net, k - 1, act[k], n[k], fp[k], o, head ? out_slice : n[k + 1],
                               head ? out_pitch : fp[k + 1], (int)(head ? g.r[k] : fr[k + 1]),
                               (int)(head ? g.c[k] : fc[k + 1]), g.d[k], nz, head && ot == MB_OUT_U8, st));
        }
    }
    return fm_tc_poll_error(net);
}

}  // namespace mb
