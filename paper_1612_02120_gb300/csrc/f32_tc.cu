// f32_tc.cu - FP32 convolutions on the 5th-generation tensor cores: the 32 -> 32 5x5 layers of the
// FP32 teacher and the 32 -> 64 4x4 dilated layers of the FP32 FastMemb nets, as drop-in replacements
// of the CUDA-core kernels (same FP32 activations in and out).
//
// Numbers. Every FP32 value is the exact sum of three BF16 values, its leading, middle and trailing 8
// significant bits (x = x1 + x2 + x3 by truncation). Of the nine products of two such sums the six
// with i + j <= 4 are multiplied (each exact in FP32), the other three are below 2^-24 of the result.
// The tensor core adds into its FP32 accumulator by truncation, which over a whole 800-term sum would
// cost 10x the error of FP32 FMAs (4.9e-6 against 5.1e-7 relative, 5x5 32 -> 32, normal operands).
// So an accumulator holds one input row's contribution only (160 terms), the small products first and
// the ten steps of x1 w1 last, and the row taps are added up in FP32 registers with rounding to
// nearest: 2.0e-7, i.e. less than the FMA chain's error (1.6e-7 with ReLU'd inputs against 3.6e-7).
// Activations must be finite: the caller checks at load time that no input can drive one beyond
// 2^100 (x3_bounded); other nets keep the CUDA-core kernels.
//
// Implicit GEMM per staged input row u and 128-pixel strip, as in fastmemb_tc.cu:
//   D[128 px][K row taps x CO] = sum over (kx, K-half) and the six products of
//                                A_i[px + d kx][16 ch] x B_j(kx)[ky CO + co][16 ch]^T
// The K row taps are stacked along N; column tap kx is a (d kx x 16)-byte shift of the operand's
// start. Staged row u's D belongs to conv rows u .. u-K+1: the epilogue adds its ky block to the
// partial sum of conv row u - ky, which moves on by one register row per staged row.
// 60 MMAs of N = 160 per row (teacher) take 4,800 cycles, 48 of N = 128 (FastMemb; the 64 conv
// channels in two halves, one per CTA, whose 98 KB of operands leave room for the rows) 3,072: the
// tensor pipe bounds them (5,300 cycles per row measured), against 51,200 / 32,768 cycles of FP32
// FMAs for the same row. Measured against the CUDA-core kernels: teacher 16 x 512 x 512, layer 2
// 4,528 -> 770 us, layer 3 with head 4,210 -> 606 us; FastMemb region 611 x 803, layer 2 737 -> 151 us,
// layer 3 713 -> 147 us. Error of the map against 64 bits 1.3e-7 -> 6.5e-8 and 8.2e-7 -> 4.5e-7.
//
// Warp roles (640 threads, 1 CTA per SM, one equal contiguous range of strip-rows per CTA):
//   warp 0        lane 0 issues the MMAs
//   warps 4-11    epilogue, two groups of 16 channels: TMEM -> partial sums, then bias and ReLU; or
//                 bias, ReLU, head, sigmoid; or bias and max-out
//   warps 12-19   producers, two groups on alternate rows: load 8 channels of a pixel, max-filter
//                 them, split them, store 3 x 16 B
// Every mbarrier wait is bounded; after a timeout the CTA records MB_ERR_TIMEOUT, stops issuing and
// frees its TMEM.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "f32_split.cuh"
#include "internal.h"

namespace mb {

namespace {

enum { X_RELU = 0, X_HEAD = 1, X_MAXOUT = 2 };

template <int K, int OUT>
struct XCfg {
    static constexpr int CO = 32;                     // conv channels of a CTA
    static constexpr int kN = K * CO;                 // N of an MMA = columns of an accumulator
    static constexpr int kBufs = 512 / kN;            // accumulators (3 / 4 staged rows)
    static constexpr int kGroups = 2 * K;             // (kx, K-half)
    static constexpr int kBlock = 2 * kN * 16;        // B block [2 chunks][kN rows][16 B]
    static constexpr int kBBytes = 3 * kGroups * kBlock;
    static constexpr int kMaxD = K == 4 ? 8 : 1;
    // pixels per staged row; 2 mod 8, which spreads the 4 chunk planes of a pixel over distinct banks
    static constexpr int kP = (128 + (K - 1) * kMaxD + 7) / 8 * 8 + 2;
    static constexpr int kPart = 4 * kP * 16;         // bytes of one BF16 part of a staged row
    static constexpr int kSlot = 3 * kPart;
    static constexpr int kRing = K == 5 ? 2 : 4;      // staged rows
    static constexpr int oB = 0;
    static constexpr int oRing = oB + kBBytes;
    static constexpr int kConsts = 68;                    // bias[32], head w[32], head b, 3 unused
    static constexpr int kPack = kBBytes + kConsts * 4;   // bytes of one half's operands
    static constexpr int oConst = oRing + kRing * kSlot;
    static constexpr int oHead = oConst + kConsts * 4;    // partial head sums, two rows in turn
    static constexpr int oBar = oHead + (OUT == X_HEAD ? 2 * 128 * 4 : 0);
    static constexpr int kBars = 2 * kRing + 2 * kBufs + 1;
    static constexpr int oMisc = oBar + kBars * 8;
    static constexpr int kSmem = oMisc + 16;
    static constexpr int kThreads = 640;
    static_assert(kSmem <= 227 * 1024, "shared memory");
    static_assert(kBufs * kN <= 512 && kBufs >= 2, "TMEM");
};

struct XParams {
    const float* in;             // [slice][row][column (pitch)][32]
    int64_t in_slice, in_pitch;  // floats, pixels
    int in_rows, in_cols;        // domain of the (max-filtered, strided) input
    int d, dm, stride;           // conv dilation; max-filter dilation (0: none) and stride on the load
    int64_t src_cols;            // source pixels per row that may be read (prefetch bound)
    void* out;                   // X_RELU, X_MAXOUT: FP32 [slice][y][x][32]; X_HEAD: FP32 or uint8 [slice][y][x]
    int64_t out_slice, out_pitch;
    int out_h, out_w, nz, n_strips;
    int64_t total_rows;          // strip-rows per half: nz x n_strips x out_h
    const uint8_t* wpack;        // per half: B blocks, then the constants
    int halves, out_u8;
    int* err;
    int fault_stall;             // test injection: producers withhold their arrivals
    uint64_t wait_ns;
};

struct XItem {
    int z, ry, x0, m0, rows;  // conv rows y = ry + d (m0 + j), j < rows
};
struct XCursor {
    int64_t g, hi;
};

// The CTAs of a half (blockIdx.x mod halves) split its strip-rows, in (slice, residue class, strip,
// row) order, into equal contiguous ranges; an item is the part of a range in one column.
__device__ __forceinline__ XCursor x_begin(const XParams& p) {
    const int64_t n = gridDim.x / p.halves, i = blockIdx.x / p.halves;
    return XCursor{p.total_rows * i / n, p.total_rows * (i + 1) / n};
}

__device__ __forceinline__ bool x_next(const XParams& p, XCursor& c, XItem& it) {
    if (c.g >= c.hi) return false;
    const int64_t per_slice = (int64_t)p.n_strips * p.out_h;
    it.z = (int)(c.g / per_slice);
    const int r = (int)(c.g - (int64_t)it.z * per_slice);
    const int base = p.out_h / p.d, rem = p.out_h % p.d;
    auto before = [&](int ry) { return p.n_strips * (ry * base + min(ry, rem)); };
    int ry = 0;
    while (ry + 1 < p.d && before(ry + 1) <= r) ++ry;
    const int hr = base + (ry < rem ? 1 : 0);
    const int off = r - before(ry);
    const int strip = off / hr;
    it.ry = ry;
    it.x0 = strip * 128;
    it.m0 = off - strip * hr;
    it.rows = (int)min((int64_t)(hr - it.m0), c.hi - c.g);
    c.g += it.rows;
    return true;
}

__device__ __forceinline__ float4 max4(float4 a, float4 b) {
    return make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z), fmaxf(a.w, b.w));
}

template <int K, int OUT>
__global__ void __launch_bounds__(640, 1) x3_conv(const __grid_constant__ XParams p) {
    using C = XCfg<K, OUT>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* row_full = reinterpret_cast<uint64_t*>(smem + C::oBar);
    uint64_t* row_empty = row_full + C::kRing;
    uint64_t* acc_full = row_empty + C::kRing;
    uint64_t* acc_free = acc_full + C::kBufs;
    uint64_t* fin = acc_free + C::kBufs;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::oMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::oMisc + 4);
    const float* cst = reinterpret_cast<const float*>(smem + C::oConst);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int half = blockIdx.x % p.halves;

    if (tid == 0) {
        for (int i = 0; i < C::kRing; ++i) {
            ptx::mbar_init(&row_full[i], 128);
            ptx::mbar_init(&row_empty[i], 1);
        }
        for (int i = 0; i < C::kBufs; ++i) {
            ptx::mbar_init(&acc_full[i], 1);
            ptx::mbar_init(&acc_free[i], 256);
        }
        ptx::mbar_init(fin, 1);
        *abort_flag = 0;
        ptx::mbar_fence_init();
    }
    {
        const uint4* src = reinterpret_cast<const uint4*>(p.wpack + (size_t)half * C::kPack);
        uint4* dst = reinterpret_cast<uint4*>(smem + C::oB);
        for (int i = tid; i < C::kBBytes / 16; i += C::kThreads) dst[i] = __ldg(src + i);
        uint4* cdst = reinterpret_cast<uint4*>(smem + C::oConst);
        if (tid < C::kConsts / 4) cdst[tid] = __ldg(src + C::kBBytes / 16 + tid);
    }
    if (warp == 0) {
        ptx::tmem_alloc(tmem_slot, 512);
        ptx::tmem_relinquish();
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    ptx::grid_dep_launch();  // after the TMEM allocation, so that the next launch's cannot come before it
    const uint32_t tbase = *tmem_slot;
    const uint32_t sbase = ptx::smem_u32(smem);
    const int d = p.d;
    ptx::grid_dep_wait();
    // registers per warpgroup: launched with 96 each (640 threads); the producers keep theirs
    static_assert(40 + 2 * 120 + 2 * 96 <= 5 * 96, "register budget exceeds the launch allocation");

    if (warp < 4) {
        ptx::setmaxnreg_dec<40>();
        if (warp == 0) {
            // ================= MMA issuer ============================================================
            const uint64_t adesc = ptx::smem_desc(sbase + C::oRing, C::kP * 16, 128);
            const uint64_t bdesc = ptx::smem_desc(sbase + C::oB, C::kN * 16, 128);
            const uint32_t a_hi = (uint32_t)(adesc >> 32), b_hi = (uint32_t)(bdesc >> 32);
            constexpr uint32_t id = ptx::idesc_f32acc(ptx::kFmtBF16, 128, C::kN);
            const uint32_t lead = lane == 0;
            uint32_t q = 0;
            bool ok = true;
            auto wait_row = [&](uint32_t r) {
                ok = ok && x_wait(&row_full[r % C::kRing], (r / C::kRing) & 1, abort_flag, p.err, p.wait_ns);
                ok = ok && x_wait(&acc_free[r % C::kBufs], ((r / C::kBufs) & 1) ^ 1, abort_flag, p.err, p.wait_ns);
            };
            auto commit_row = [&](uint32_t r) {
                ptx::mma_commit_if(lead, &row_empty[r % C::kRing]);
                ptx::mma_commit_if(lead, &acc_full[r % C::kBufs]);
            };
            XCursor cur = x_begin(p);
            XItem it;
            while (x_next(p, cur, it)) {
                const int nst = it.rows + K - 1;
                wait_row(q);
                for (int u = 0; u < nst; ++u, ++q) {
                    const uint32_t s = q % C::kRing, b = q % C::kBufs;
                    ptx::tc_fence_after();
                    const uint32_t on = ok ? lead : 0u, dcol = tbase + b * C::kN;
                    const uint32_t arow = (uint32_t)adesc + ((s * C::kSlot) >> 4);
                    // products x_i w_j in the order (3,1) (2,2) (1,3) (2,1) (1,2) (1,1)
#pragma unroll 1
                    for (int c = 0; c < 6; ++c) {
                        const uint32_t ai = (0x001012u >> (4 * c)) & 15u, bi = (0x010210u >> (4 * c)) & 15u;
                        const uint32_t a0 = arow + ai * (C::kPart >> 4);
                        const uint32_t b0 = (uint32_t)bdesc + bi * ((C::kGroups * C::kBlock) >> 4);
#pragma unroll
                        for (int g = 0; g < C::kGroups; ++g) {
                            ptx::mma_bf16_acc(on, dcol, a0 + (g & 1) * ((2 * C::kP * 16) >> 4) + (uint32_t)((g >> 1) * d),
                                              a_hi, b0 + g * (C::kBlock >> 4), b_hi, id, g > 0 ? 1u : (uint32_t)(c > 0));
                            // between the MMAs, so that the tensor pipe does not run dry: the previous
                            // row's commits, and the waits for the next row
                            if (g == 3 && c == 0 && u > 0) commit_row(q - 1);
                            if (g == 3 && c == 5 && u + 1 < nst) wait_row(q + 1);
                        }
                    }
                }
                commit_row(q - 1);
            }
            if (lane == 0) x_drain(fin, p.err, p.wait_ns);
            __syncwarp();
        }
    } else if (warp < 12) {
        ptx::setmaxnreg_inc<120>();
        // ================= epilogue ===================================================================
        const int px = tid & 127, g = (warp - 4) >> 2;  // conv channels 16 g .. 16 g + 15 of the CTA's 32
        const uint32_t lanes = (uint32_t)(32 * (warp & 3)) << 16;
        float sum[K - 1][16];  // sum[k]: conv row u - k so far
        float* head = reinterpret_cast<float*>(smem + C::oHead);
        uint32_t q = 0, turn = 0;
        XCursor cur = x_begin(p);
        XItem it;
        while (x_next(p, cur, it)) {
            const int nst = it.rows + K - 1;
            const int x = it.x0 + px;
#pragma unroll
            for (int k = 0; k < K - 1; ++k)
#pragma unroll
                for (int c = 0; c < 16; ++c) sum[k][c] = 0.f;
            for (int u = 0; u < nst; ++u, ++q) {
                const uint32_t bf = q % C::kBufs;
                x_wait(&acc_full[bf], (q / C::kBufs) & 1, abort_flag, p.err, p.wait_ns);
                ptx::tc_fence_after();
                const uint32_t ta = tbase + lanes + bf * C::kN + 16u * g;
                float done[16];
#pragma unroll
                for (int k = K - 1; k >= 0; --k) {
                    float v[16];
                    ptx::tmem_ld16(ta + (uint32_t)(C::CO * k), v);
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        if (k == K - 1)
                            done[c] = sum[k - 1][c] + v[c];
                        else
                            sum[k][c] = k > 0 ? sum[k - 1 < 0 ? 0 : k - 1][c] + v[c] : v[c];
                    }
                }
                ptx::tc_fence_before();
                ptx::mbar_arrive(&acc_free[bf]);
                if (u < K - 1) continue;
                const int y = it.ry + d * (it.m0 + u - (K - 1));
                const bool store = x < p.out_w && !*abort_flag;
#pragma unroll
                for (int c = 0; c < 16; ++c) done[c] += cst[16 * g + c];
                if constexpr (OUT == X_RELU) {
                    if (store) {
                        float4* o = reinterpret_cast<float4*>(static_cast<float*>(p.out) + (int64_t)it.z * p.out_slice +
                                                              ((int64_t)y * p.out_pitch + x) * 32 + 16 * g);
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            o[c] = make_float4(fmaxf(done[4 * c], 0.f), fmaxf(done[4 * c + 1], 0.f),
                                               fmaxf(done[4 * c + 2], 0.f), fmaxf(done[4 * c + 3], 0.f));
                    }
                } else if constexpr (OUT == X_MAXOUT) {
                    if (store) {  // 16 conv channels -> 8 features; the halves are 16 features apart
                        float4* o = reinterpret_cast<float4*>(static_cast<float*>(p.out) + (int64_t)it.z * p.out_slice +
                                                              ((int64_t)y * p.out_pitch + x) * 32 + 16 * half + 8 * g);
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            o[c] = make_float4(fmaxf(done[8 * c], done[8 * c + 1]), fmaxf(done[8 * c + 2], done[8 * c + 3]),
                                               fmaxf(done[8 * c + 4], done[8 * c + 5]),
                                               fmaxf(done[8 * c + 6], done[8 * c + 7]));
                    }
                } else {
                    float z = 0.f;
                    const float* hw = cst + 32 + 16 * g;
#pragma unroll
                    for (int c = 0; c < 16; ++c) z = fmaf(hw[c], fmaxf(done[c], 0.f), z);
                    // the two groups' sums meet in group 0; two buffers in turn, so that one rendezvous
                    // per row keeps a row's reader from the next but one's writer
                    float* h = head + turn * 128;
                    turn ^= 1;
                    if (g == 1) h[px] = z;
                    asm volatile("bar.sync 2, 256;" ::: "memory");
                    if (g == 0 && store) {
                        const float prob = 1.0f / (1.0f + expf(-((z + h[px]) + cst[64])));
                        const int64_t idx = (int64_t)it.z * p.out_slice + (int64_t)y * p.out_pitch + x;
                        if (p.out_u8)
                            static_cast<uint8_t*>(p.out)[idx] = (uint8_t)fminf(floorf(255.0f * prob + 0.5f), 255.0f);
                        else
                            static_cast<float*>(p.out)[idx] = prob;
                    }
                }
            }
        }
    } else {
        // ================= producers ==================================================================
        // Tasks e = pt + 128 i of a row: 8 channels (e & 3) of pixel e >> 2, so 4 lanes read a pixel's
        // 128 bytes.
        const int grp = (warp - 12) >> 2, pt = tid - 384 - 128 * grp;
        const int ntask = 4 * (128 + (K - 1) * d);
        constexpr int kTasks = (4 * (128 + (K - 1) * C::kMaxD) + 127) / 128;
        const int64_t dxo = (int64_t)p.dm * 8, dyo = (int64_t)p.dm * p.in_pitch * 8;  // float4
        uint32_t q = 0;
        XCursor cur = x_begin(p);
        XItem it;
        while (x_next(p, cur, it)) {
            const int nst = it.rows + K - 1;
            const float* src = p.in + (int64_t)it.z * p.in_slice;
            const int sx0 = p.stride * it.x0;
            const int pf_cols = (int)min((int64_t)(p.stride * (127 + (K - 1) * d) + p.dm + 1), p.src_cols - sx0);
            for (int u = 0; u < nst; ++u, ++q) {
                if ((int)(q & 1) != grp) continue;
                const uint32_t s = q % C::kRing;
                const int yin = it.ry + d * (it.m0 + u);
                if (pt == 0 && u + 2 < nst) {  // this group's next row into L2
                    const int yp = yin + 2 * d;
                    if (yp < p.in_rows && pf_cols > 0) {
                        const float* r0 = src + ((int64_t)(p.stride * yp) * p.in_pitch + sx0) * 32;
                        ptx::prefetch_l2_bulk(r0, (uint32_t)pf_cols * 128u);
                        if (p.dm > 0) ptx::prefetch_l2_bulk(r0 + 4 * dyo, (uint32_t)pf_cols * 128u);
                    }
                }
                // the whole row in registers before the slot wait: after it the stores alone remain
                float4 v[kTasks][2];
#pragma unroll
                for (int i = 0; i < kTasks; ++i) {
                    const int e = pt + 128 * i, xin = it.x0 + (e >> 2);
                    v[i][0] = v[i][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (e < ntask && yin < p.in_rows && xin < p.in_cols) {
                        const float4* a = reinterpret_cast<const float4*>(
                            src + ((int64_t)(p.stride * yin) * p.in_pitch + p.stride * xin) * 32 + (e & 3) * 8);
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            v[i][j] = a[j];
                            if (p.dm > 0)
                                v[i][j] = max4(max4(v[i][j], a[dxo + j]), max4(a[dyo + j], a[dyo + dxo + j]));
                        }
                    }
                }
                x_wait(&row_empty[s], ((q / C::kRing) & 1) ^ 1, abort_flag, p.err, p.wait_ns);
                uint8_t* dst = smem + C::oRing + s * C::kSlot;
#pragma unroll
                for (int i = 0; i < kTasks; ++i) {
                    const int e = pt + 128 * i;
                    if (e < ntask) {
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            uint4 w;
                            w.x = take_part(v[i][0].x, v[i][0].y);
                            w.y = take_part(v[i][0].z, v[i][0].w);
                            w.z = take_part(v[i][1].x, v[i][1].y);
                            w.w = take_part(v[i][1].z, v[i][1].w);
                            *reinterpret_cast<uint4*>(dst + k * C::kPart + ((e & 3) * C::kP + (e >> 2)) * 16) = w;
                        }
                    }
                }
                ptx::fence_proxy_async_smem();
                if (!p.fault_stall) ptx::mbar_arrive(&row_full[s]);
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == 0) ptx::tmem_dealloc(tbase, 512);
}

uint16_t part_bits(float& f) {
    uint32_t u;
    memcpy(&u, &f, 4);
    const uint32_t hi = u & 0xffff0000u;
    float h;
    memcpy(&h, &hi, 4);
    f -= h;
    return (uint16_t)(hi >> 16);
}

// One half's operands: conv channels c0 .. c0 + 31 of W[co][32][K][K], b[co]: B blocks [chunk kc][row
// 32 ky + c][8 BF16], ci = 16 h + 8 kc + e, per (part, kx, K-half h); then bias[32], head w[32] and b.
template <int K>
void x3_pack(const float* W, const float* b, int c0, const float* head, std::vector<uint8_t>& out) {
    using C = XCfg<K, X_RELU>;
    const size_t base = out.size();
    out.resize(base + C::kPack, 0);
    uint8_t* o = out.data() + base;
    for (int c = 0; c < 32; ++c)
        for (int g = 0; g < 4; ++g) {  // input channels 8 g .. 8 g + 7: one 16-byte chunk per (part, tap)
            const float* w = W + ((size_t)(c0 + c) * 32 + 8 * g) * K * K;
            uint8_t* at = o + (g / 2) * C::kBlock + (g % 2) * C::kN * 16 + c * 16;
            for (int ky = 0; ky < K; ++ky)
                for (int kx = 0; kx < K; ++kx) {
                    uint16_t v[3][8];
                    for (int e = 0; e < 8; ++e) {
                        float f = w[e * K * K + ky * K + kx];
                        for (int i = 0; i < 3; ++i) v[i][e] = part_bits(f);
                    }
                    for (int i = 0; i < 3; ++i)
                        memcpy(at + (i * C::kGroups + kx * 2) * C::kBlock + 32 * ky * 16, v[i], 16);
                }
        }
    memcpy(o + C::kBBytes, b + c0, 32 * 4);
    if (head) memcpy(o + C::kBBytes + 128, head, 33 * 4);
}

template <int K, int OUT>
mb_status launch_x3(XParams& p, cudaStream_t st) {
    using C = XCfg<K, OUT>;
    static int n_sms = 0;
    if (n_sms == 0) {
        int dev = 0;
        MB_CUDA(cudaGetDevice(&dev));
        MB_CUDA(cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev));
    }
    static std::atomic<uint64_t> smem_set{0};
    MB_TRY(set_smem_once(smem_set, x3_conv<K, OUT>, C::kSmem));
    // one range per SM, or fewer when a range would get under 2 rows (each costs K - 1 more staged rows)
    const int64_t per_half = std::max<int64_t>(1, std::min<int64_t>(n_sms / p.halves, (p.total_rows + 1) / 2));
    MB_CUDA(launch_dependent(x3_conv<K, OUT>, (unsigned)(per_half * p.halves), C::kThreads, C::kSmem, st, p));
    count_launch();
    MB_CUDA(cudaGetLastError());
    return MB_OK;
}

struct X3State {
    uint8_t* d_w[4] = {};  // the packed layers, parts of one allocation (d_w[0])
    int* h_err = nullptr;
    int* d_err = nullptr;
};

X3State* x3_of(const mb_net* net) { return reinterpret_cast<X3State*>(net->x3_state); }

}  // namespace

// Whether no input can drive an activation of the net beyond 2^100 (finite with room for the sums):
// max |feature| of a layer <= max |b| + (max over filters of the sum of |w|) x max |feature| before it.
// And whether no layer before the head lives, with its features or its weights, wholly below 2^-60: the
// trailing part of a value is 2^-24 of it, and BF16 ends at 2^-133 (a first layer times 2^-118 with the second
// over 2^-118, the same network exactly, would lose its third parts: 2^-16 instead of 2^-24).
static bool x3_bounded(const mb_net* net) {
    const float* P = net->host_params.data();
    const double least = 8.7e-19;
    double bound = 1.0;
    for (const mb_layer_desc& L : net->layers) {
        if (L.kind == MB_MAXFILTER) continue;
        const bool head = L.kind != MB_CONV;
        const int co = L.cout * std::max(1, L.maxout_groups), k = L.cin * L.ksize * L.ksize;
        double worst = 0.0, wmax = 0.0;
        for (int c = 0; c < co; ++c) {
            double s = std::fabs((double)P[(size_t)co * k + c]);
            for (int i = 0; i < k; ++i) {
                const double w = std::fabs((double)P[(size_t)c * k + i]);
                wmax = std::max(wmax, w);
                s += bound * w;
            }
            worst = std::max(worst, s);
        }
        bound = worst;
        P += (size_t)co * k + co;
        if (!(bound < 1.2e30) || (!head && (bound < least || wmax < least))) return false;
    }
    return true;
}

mb_status x3_prepare(mb_net* net) {
    const bool teacher = net->family == FAMILY_TEACHER;
    if (net->prec != MB_PREC_FP32 || !(teacher || is_fastmemb(net->family))) return MB_OK;
    X3State* S = x3_of(net);
    if (!S) {
        S = new (std::nothrow) X3State();
        if (!S) {
            set_error("host allocation failed");
            return MB_ERR_OOM;
        }
        net->x3_state = S;
    }
    // (packed whatever the bound: a call captured with other weights in a caller's graph replays these layers)
    net->x3_ok = false;
    const int n = teacher ? 2 : fastmemb_convs(net->family) - 2;
    const float* P = net->host_params.data() + (teacher ? 832 : 64 * 16 + 64);
    std::vector<uint8_t> pk;
    size_t at[5] = {};
    for (int l = 0; l < n; ++l) {
        if (teacher) {
            x3_pack<5>(P, P + 25600, 0, l == 1 ? P + 25600 + 32 : nullptr, pk);
            P += 25600 + 32;
        } else {
            x3_pack<4>(P, P + 64 * 32 * 16, 0, nullptr, pk);
            x3_pack<4>(P, P + 64 * 32 * 16, 32, nullptr, pk);
            P += 64 * 32 * 16 + 64;
        }
        at[l + 1] = pk.size();
    }
    if (!S->d_w[0]) MB_TRY(dev_alloc((void**)&S->d_w[0], pk.size()));
    for (int l = 1; l < n; ++l) S->d_w[l] = S->d_w[0] + at[l];
    MB_CUDA(cudaMemcpy(S->d_w[0], pk.data(), pk.size(), cudaMemcpyHostToDevice));
    if (!S->h_err) {
        if (fault_oom()) {
            set_error("pinned allocation failed (MB_FAULT_OOM injected)");
            return MB_ERR_OOM;
        }
        MB_CUDA(cudaHostAlloc((void**)&S->h_err, sizeof(int), cudaHostAllocMapped));
        *S->h_err = 0;
        MB_CUDA(cudaHostGetDevicePointer((void**)&S->d_err, S->h_err, 0));
    }
    net->x3_ok = x3_bounded(net);
    return MB_OK;
}

void x3_release(mb_net* net) {
    X3State* S = x3_of(net);
    if (!S) return;
    dev_free(S->d_w[0]);
    if (S->h_err) cudaFreeHost(S->h_err);
    delete S;
    net->x3_state = nullptr;
}

mb_status x3_poll_error(mb_net* net) {
    X3State* S = x3_of(net);
    if (S && S->h_err && *(volatile int*)S->h_err) {
        *(volatile int*)S->h_err = 0;
        set_error("an FP32 tensor-core launch gave up waiting (device-side wait limit)");
        return MB_ERR_TIMEOUT;
    }
    return MB_OK;
}

mb_status x3_layer(const mb_net* net, int layer, const X3Layer& a, cudaStream_t st) {
    X3State* S = x3_of(net);
    if (!S || !net->x3_ok || !S->d_w[layer]) {
        set_error("FP32 tensor-core weights not prepared");
        return MB_ERR_NOT_READY;
    }
    const bool teacher = net->family == FAMILY_TEACHER;
    if (a.d > (teacher ? XCfg<5, X_RELU>::kMaxD : XCfg<4, X_MAXOUT>::kMaxD)) {
        set_error("FP32 tensor-core layer: dilation %d too large", a.d);
        return MB_ERR_INVALID_ARG;
    }
    XParams p{};
    p.in = a.in;
    p.in_slice = a.in_slice;
    p.in_pitch = a.in_pitch;
    p.in_rows = a.in_rows;
    p.in_cols = a.in_cols;
    p.d = a.d;
    p.dm = a.dm;
    p.stride = std::max(1, a.stride);
    p.src_cols = a.src_cols;
    p.out = a.out;
    p.out_slice = a.out_slice;
    p.out_pitch = a.out_pitch;
    p.out_h = a.out_h;
    p.out_w = a.out_w;
    p.nz = a.nz;
    p.n_strips = (a.out_w + 127) / 128;
    p.total_rows = (int64_t)a.nz * p.n_strips * a.out_h;
    p.wpack = S->d_w[layer];
    p.halves = teacher ? 1 : 2;
    p.out_u8 = a.out_u8;
    p.err = S->d_err;
    const char* stall = getenv("MB_FAULT_STALL");
    p.fault_stall = (stall && stall[0] == '1') ? 1 : 0;
    p.wait_ns = p.fault_stall ? 200000000ull : kXWaitNs;
    if (!teacher) return launch_x3<4, X_MAXOUT>(p, st);
    return layer == 0 ? launch_x3<5, X_RELU>(p, st) : launch_x3<5, X_HEAD>(p, st);
}

}  // namespace mb
