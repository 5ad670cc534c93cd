// student_x3.cu - the FP32 student's convolutions on the tensor cores with FP32 accuracy, each fused with
// what follows it: conv2 + ReLU + head, with loss + dL/dy2 (st_x3<SX_FWD>) or the probability
// (st_x3<SX_INFER>), and the data gradient + ReLU mask + conv1's weight gradient (st_x3<SX_BWD>); the first
// convolution (st_conv1) and conv2's weight gradient (st_grad2) on packed FP32 FMAs.
//
// Numbers: the three-part BF16 split of f32_tc.cu (six of nine products, error below an FMA chain's).
// With 16 channels the products of equal weight sit in columns of their own: part 1 of an input row
// is multiplied by [w1 | w2 | w3] (N = 144: 3 parts x 3 row taps x 16), part 2 by [w1 | w2] into the
// second and third column groups, part 3 by w1 into the third; the epilogue adds g1 + (g2 + g3) per row
// tap and sums the row taps in FP32.
//
// Inference, FP32 student, against the CUDA-core convolutions: 64 x 64 20.6 -> 14.6 us, 1024 x 1024 133 -> 65,
// 4096 x 4096 1,907 -> 794.
//
// st_x3 reads one 64-byte pixel of h1 or dy2 per output pixel, once, and the forward writes dy2 once
// (h2 and dy1 exist in registers only): a row of 128 pixels costs ~500 cycles of MMAs and 360-710 of
// HBM time; 1,290-1,590 measured (forward 358 us, backward 364 on a batch of 32 x 512 x 512; 370 each with
// remainders in the issue loop and a third turn for one producer warp): the issuing warp's and the epilogue's chains.
// The separate kernels (conv 865 us, head and loss 218, data gradient 1,023, conv1's weight gradient
// 395 on a batch of 32 x 512 x 512) passed 3.2 GB through HBM at 0.47-0.55 of the FP32 FMA rate.
//
// Warp roles of st_x3 (512 threads, 1 CTA per SM, one equal contiguous range of strip-rows per CTA):
//   warp 0        issues the MMAs (whole warp on uniform values, lane 0 issuing)
//   warp 1        producer of the row's last two pixels
//   warps 4-11    epilogue, two groups of 8 channels, one pixel column per thread; sums over pixels
//                 (loss, head, bias and conv1 weight gradients) stay in registers until the end
//   warps 12-15   producers: load 8 channels of a pixel, split, store 3 x 16 B
// Slices and targets are read through the read-only path: no launch of the chain writes them, and its first
// launch (student_pack; st_conv1 for inference) is an ordinary one, so that what wrote them has ended.
// The grids are fixed, so the partial sums, and with them a training run, are reproducible.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "f32_split.cuh"
#include "internal.h"
#include "student_x3.h"

namespace mb {

namespace {

constexpr int kThreadsX = 512;
constexpr int kP = 130;                       // pixels per staged row (2 mod 8: chunk planes on distinct banks)
constexpr int kPart = 2 * kP * 16;            // one BF16 part of a staged row: [2 chunks][kP][16 B]
constexpr int kSlotX = 3 * kPart;
constexpr int kRingX = 6;
constexpr int kNx = 144;                      // columns per accumulator: 3 weight groups x 3 row taps x 16
constexpr int kBufsX = 3;
constexpr int oBx = 0;
constexpr int oRingX = oBx + kX3StudentPack;
constexpr int oLut = oRingX + kRingX * kSlotX;    // u / 255 (backward)
constexpr int oXch = oLut + 256 * 4;              // partial head sums: 2 rows in turn x 2 groups x 128
constexpr int oRed = oXch + 2 * 2 * 128 * 4;      // [8 warps][80] partial sums at the end
constexpr int oBarX = oRed + 8 * 80 * 4;
constexpr int kBarsX = 2 * kRingX + 2 * kBufsX + 1;
constexpr int oMiscX = oBarX + kBarsX * 8;
constexpr int kSmemX = oMiscX + 16;
static_assert(kSmemX <= 227 * 1024 && kBufsX * kNx <= 512, "resources");

// the passes of st_x3: training forward, training backward, inference
enum { SX_FWD = 0, SX_BWD = 1, SX_INFER = 2 };

struct SxParams {
    const float* in;       // h1 [B][H+2][W+2][16], or dy2 [B][H][W][16] read as zero-padded by 2
    const uint8_t* wpack;  // student_pack's B operand of this pass: per column tap kx [2 chunks][144 rows][16 B]
    const float* fw;       // forward parameters (b2, head)
    int B, H, W;
    // forward
    const float* target;
    const int* zmap;
    float* dy2;
    float inv_n;
    // inference
    void* out;             // probabilities [B][H][W], out_pitch and out_slice elements apart
    int64_t out_pitch, out_slice;
    int out_u8;
    // backward
    const uint16_t* mask;  // h1 > 0 per channel, [B][H+2][W+2]
    const uint8_t* img;    // [slices][H][W]
    float* partial;
    int64_t total_rows;
    int n_strips, out_h, out_w;
    int* err;
    int fault_stall;
    uint64_t wait_ns;
};

struct SxItem {
    int z, x0, y0, rows;
};

__device__ __forceinline__ bool sx_next(const SxParams& p, int64_t& g, int64_t hi, SxItem& it) {
    if (g >= hi) return false;
    const int64_t col = g / p.out_h;
    it.y0 = (int)(g - col * p.out_h);
    it.z = (int)(col / p.n_strips);
    it.x0 = (int)(col % p.n_strips) * 128;
    it.rows = (int)min((int64_t)(p.out_h - it.y0), hi - g);
    g += it.rows;
    return true;
}

__device__ __forceinline__ int sx_refl(int t, int n) {
    t = t < 0 ? -t : t;
    t = t >= n ? 2 * (n - 1) - t : t;
    return min(max(t, 0), n - 1);  // columns past the strip's domain feed nothing that counts
}

// Sums of N values over the 128 threads of an epilogue group, in a fixed order; valid in the group's
// first warp's lane 0 order: out[i] written by thread i of the group.
template <int N>
__device__ __forceinline__ void group_sum(const float (&v)[N], float* red, int group, int warp_in, int lane, float* out) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        float s = v[i];
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
        if (lane == 0) red[(group * 4 + warp_in) * 80 + i] = s;
    }
    asm volatile("bar.sync %0, 128;" ::"r"(3 + group) : "memory");
    const int t = warp_in * 32 + lane;
    if (t < N) {
        const float* r = red + group * 4 * 80 + t;
        out[t] = (r[0] + r[80]) + (r[160] + r[240]);
    }
}

template <int MODE>
__global__ void __launch_bounds__(kThreadsX, 1) st_x3(const __grid_constant__ SxParams p) {
    constexpr bool BWD = MODE == SX_BWD, INFER = MODE == SX_INFER;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* row_full = reinterpret_cast<uint64_t*>(smem + oBarX);
    uint64_t* row_empty = row_full + kRingX;
    uint64_t* acc_full = row_empty + kRingX;
    uint64_t* acc_free = acc_full + kBufsX;
    uint64_t* fin = acc_free + kBufsX;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + oMiscX);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + oMiscX + 4);
    float* lut = reinterpret_cast<float*>(smem + oLut);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);

    if (tid == 0) {
        for (int i = 0; i < kRingX; ++i) {
            ptx::mbar_init(&row_full[i], 5);
            ptx::mbar_init(&row_empty[i], 1);
        }
        for (int i = 0; i < kBufsX; ++i) {
            ptx::mbar_init(&acc_full[i], 1);
            ptx::mbar_init(&acc_free[i], 8);
        }
        ptx::mbar_init(fin, 1);
        *abort_flag = 0;
        ptx::mbar_fence_init();
    }
    if (tid < 256) lut[tid] = (float)tid / 255.0f;
    if (warp == 0) {
        ptx::tmem_alloc(tmem_slot, 512);
        ptx::tmem_relinquish();
    }
    if constexpr (INFER) {
        // no packing launch before it: W2t[ci][tap][co], which no launch of the chain writes, split here
        for (int i = tid; i < 2304; i += kThreadsX) {
            const int co = i % 16, tap = (i / 16) % 9, ci = i / 144, ky = tap / 3, kx = tap % 3;
            float v = p.fw[kSW2 + i];
#pragma unroll
            for (int part = 0; part < 3; ++part) {
                const uint32_t u = __float_as_uint(v) & 0xffff0000u;
                v -= __uint_as_float(u);
                *reinterpret_cast<uint16_t*>(smem + oBx + ((kx * 2 + (ci >> 3)) * kNx + 48 * part + 16 * ky + co) * 16 + 2 * (ci & 7)) =
                    (uint16_t)(u >> 16);
            }
        }
    }
    ptx::grid_dep_wait();
    if constexpr (!INFER) {
        const uint4* src = reinterpret_cast<const uint4*>(p.wpack);
        uint4* dst = reinterpret_cast<uint4*>(smem + oBx);
        for (int i = tid; i < kX3StudentPack / 16; i += kThreadsX) dst[i] = src[i];
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    ptx::grid_dep_launch();  // after the TMEM allocation, so that the next launch's cannot come before it
    const uint32_t tbase = *tmem_slot;
    const uint32_t sbase = ptx::smem_u32(smem);
    int64_t pos = p.total_rows * (int64_t)blockIdx.x / gridDim.x;
    const int64_t end = p.total_rows * (int64_t)(blockIdx.x + 1) / gridDim.x;
    SxItem it;
    static_assert(40 + 2 * 176 + 120 <= 4 * 128, "register budget exceeds the launch allocation");

    // Producer of kTasks tasks a thread, from e = first on, 128 apart: 8 channels (e & 1) of pixel e >> 1
    // of every staged row. The loads of the row after next are issued before this row's are split (two
    // rows in flight). Warps 12-15 take the 256 tasks of pixels 0..127, a lane each and two in turn; the four
    // of pixels 128 and 129 are warp 1's (a third turn for them made one producer warp the slowest role).
    auto produce = [&](auto tasks, int first) {
        constexpr int kTasks = decltype(tasks)::value;
        const int off = BWD ? -2 : 0, src_h = BWD ? p.H : p.H + 2, src_w = BWD ? p.W : p.W + 2;
        uint32_t s = 0, ph = 0;
        while (sx_next(p, pos, end, it)) {
            const int nst = it.rows + 2;
            const float* src = p.in + (int64_t)it.z * src_h * src_w * 16;
            float4 v[2][kTasks][2];
            auto load = [&](int u, float4 (&d)[kTasks][2]) {
                const int y = it.y0 + u + off;
#pragma unroll
                for (int i = 0; i < kTasks; ++i) {
                    const int e = first + 128 * i, x = it.x0 + (e >> 1) + off;
                    d[i][0] = d[i][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (e < 2 * 130 && u < nst && y >= 0 && y < src_h && x >= 0 && x < src_w) {
                        const float4* a = reinterpret_cast<const float4*>(src + ((int64_t)y * src_w + x) * 16 + (e & 1) * 8);
                        d[i][0] = a[0];
                        d[i][1] = a[1];
                    }
                }
            };
            auto put = [&](int u, float4 (&d)[kTasks][2]) {
                if (u >= nst) return;
                x_wait(&row_empty[s], ph ^ 1, abort_flag, p.err, p.wait_ns);
                uint8_t* dst = smem + oRingX + s * kSlotX;
#pragma unroll
                for (int i = 0; i < kTasks; ++i) {
                    const int e = first + 128 * i;
                    if (e < 2 * 130) {
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            uint4 w;
                            w.x = take_part(d[i][0].x, d[i][0].y);
                            w.y = take_part(d[i][0].z, d[i][0].w);
                            w.z = take_part(d[i][1].x, d[i][1].y);
                            w.w = take_part(d[i][1].z, d[i][1].w);
                            *reinterpret_cast<uint4*>(dst + k * kPart + ((e & 1) * kP + (e >> 1)) * 16) = w;
                        }
                    }
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0 && !p.fault_stall) ptx::mbar_arrive(&row_full[s]);
                if (++s == kRingX) {
                    s = 0;
                    ph ^= 1;
                }
            };
            load(0, v[0]);
            load(1, v[1]);
            for (int u = 0; u < nst; u += 2) {
                put(u, v[0]);
                load(u + 2, v[0]);
                put(u + 1, v[1]);
                load(u + 3, v[1]);
            }
        }
    };

    if (warp < 4) {
        ptx::setmaxnreg_dec<40>();
        if (warp == 1) produce(std::integral_constant<int, 1>{}, 256 + lane);
        if (warp == 0) {
            // ================= MMA issuer ============================================================
            const uint64_t adesc = ptx::smem_desc(sbase + oRingX, kP * 16, 128);
            const uint64_t bdesc = ptx::smem_desc(sbase + oBx, kNx * 16, 128);
            const uint32_t a_hi = (uint32_t)(adesc >> 32), b_hi = (uint32_t)(bdesc >> 32);
            const uint32_t lead = lane == 0;
            // running ring positions (slot and phase): this warp's own chain of instructions is what
            // bounds a row once the producers keep up, and a remainder or quotient costs several
            uint32_t rs = 0, rph = 0, as = 0, aph = 0;  // next staged row's slot, next accumulator
            bool ok = true;
            auto wait_row = [&] {
                ok = ok && x_wait(&row_full[rs], rph, abort_flag, p.err, p.wait_ns);
                ok = ok && x_wait(&acc_free[as], aph ^ 1, abort_flag, p.err, p.wait_ns);
            };
            while (sx_next(p, pos, end, it)) {
                const int nst = __shfl_sync(0xffffffffu, it.rows, 0) + 2;
                uint64_t* last_empty = nullptr;
                uint64_t* last_full = nullptr;
                wait_row();
                for (int u = 0; u < nst; ++u) {
                    ptx::tc_fence_after();
                    const uint32_t on = ok ? lead : 0u, d = tbase + as * kNx;
                    const uint32_t a = (uint32_t)adesc + rs * (uint32_t)(kSlotX >> 4);
                    uint64_t* my_empty = &row_empty[rs];
                    uint64_t* my_full = &acc_full[as];
                    if (++rs == kRingX) {
                        rs = 0;
                        rph ^= 1;
                    }
                    if (++as == kBufsX) {
                        as = 0;
                        aph ^= 1;
                    }
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
                        const uint32_t b = (uint32_t)bdesc + ((kx * 2 * kNx * 16) >> 4);
                        ptx::mma_bf16_acc(on, d, a + kx, a_hi, b, b_hi, ptx::idesc_f32acc(ptx::kFmtBF16, 128, 144),
                                          kx > 0 ? 1u : 0u);
                        ptx::mma_bf16_if(on, d + 48, a + (kPart >> 4) + kx, a_hi, b, b_hi,
                                         ptx::idesc_f32acc(ptx::kFmtBF16, 128, 96));
                        ptx::mma_bf16_if(on, d + 96, a + (2 * kPart >> 4) + kx, a_hi, b, b_hi,
                                         ptx::idesc_f32acc(ptx::kFmtBF16, 128, 48));
                        if (kx == 0 && u > 0) {
                            ptx::mma_commit_if(lead, last_empty);
                            ptx::mma_commit_if(lead, last_full);
                        }
                        if (kx == 1 && u + 1 < nst) wait_row();
                    }
                    last_empty = my_empty;
                    last_full = my_full;
                }
                ptx::mma_commit_if(lead, last_empty);
                ptx::mma_commit_if(lead, last_full);
            }
            if (lane == 0) x_drain(fin, p.err, p.wait_ns);
            __syncwarp();
        }
    } else if (warp < 12) {
        ptx::setmaxnreg_inc<176>();
        // ================= epilogue ===================================================================
        const int px = tid & 127, g = (warp - 4) >> 2;  // channels 8 g .. 8 g + 7
        const uint32_t lanes = (uint32_t)(32 * (warp & 3)) << 16;
        float* xch = reinterpret_cast<float*>(smem + oXch);
        float* red = reinterpret_cast<float*>(smem + oRed);
        uint32_t q = 0, turn = 0;
        float s0[8], s1[8];  // conv rows u, u - 1 so far
        // one staged row's contributions: the completed conv row u - 2 in `done`
        auto row = [&](float (&done)[8]) {
            const uint32_t bf = q % kBufsX;
            x_wait(&acc_full[bf], (q / kBufsX) & 1, abort_flag, p.err, p.wait_ns);
            ptx::tc_fence_after();
            const uint32_t ta = tbase + lanes + bf * kNx + 8u * g;
            float v[3][3][8];
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int m = 0; m < 3; ++m) ptx::tmem_ld8_nowait(ta + (uint32_t)(48 * m + 16 * k), v[k][m]);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
                for (int m = 0; m < 3; ++m) ptx::keep8(v[k][m]);
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&acc_free[bf]);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                done[c] = s1[c] + (v[2][0][c] + (v[2][1][c] + v[2][2][c]));
                s1[c] = s0[c] + (v[1][0][c] + (v[1][1][c] + v[1][2][c]));
                s0[c] = v[0][0][c] + (v[0][1][c] + v[0][2][c]);
            }
        };
        if constexpr (!BWD) {
            float b2[8], hw[8], gw[8], db[8], loss = 0.f, gb = 0.f;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                b2[c] = p.fw[kSB2 + 8 * g + c];
                hw[c] = p.fw[kSWH + 8 * g + c];
                gw[c] = db[c] = 0.f;
            }
            const float hb = p.fw[kSBH];
            while (sx_next(p, pos, end, it)) {
                const int nst = it.rows + 2, x = it.x0 + px;
                const bool col_ok = x < p.W;
                const int64_t pix0 = ((int64_t)it.z * p.H + it.y0) * p.W + x;  // conv row 0 of the item
                const float* trow = INFER ? nullptr : p.target + ((int64_t)(p.zmap ? p.zmap[it.z] : it.z) * p.H + it.y0) * p.W + x;
#pragma unroll
                for (int c = 0; c < 8; ++c) s0[c] = s1[c] = 0.f;
                float t = 0.f;
                for (int u = 0; u < nst; ++u, ++q) {
                    const float t_next = !INFER && col_ok && u >= 1 && u + 1 < nst ? __ldg(trow + (int64_t)(u - 1) * p.W) : 0.f;
                    float h2[8];
                    row(h2);
                    if (u >= 2) {
                        float z = 0.f;
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            h2[c] = fmaxf(h2[c] + b2[c], 0.f);
                            z = fmaf(hw[c], h2[c], z);
                        }
                        // the groups' halves of the head sum meet; two buffers in turn, so that one
                        // rendezvous per row keeps a row's readers from the next but one's writers
                        float* xc = xch + turn * 256;
                        turn ^= 1;
                        xc[g * 128 + px] = z;
                        asm volatile("bar.sync 2, 256;" ::: "memory");
                        z = (xc[px] + xc[128 + px]) + hb;
                        if constexpr (INFER) {
                            if (g == (u & 1) && col_ok && !*abort_flag) {  // the groups take rows in turn
                                const float pr = 1.0f / (1.0f + expf(-z));
                                const int64_t i = (int64_t)it.z * p.out_slice + (int64_t)(it.y0 + u - 2) * p.out_pitch + x;
                                if (p.out_u8)
                                    static_cast<uint8_t*>(p.out)[i] = (uint8_t)fminf(floorf(255.0f * pr + 0.5f), 255.0f);
                                else
                                    static_cast<float*>(p.out)[i] = pr;
                            }
                        } else {
                            const float pr = 1.0f / (1.0f + expf(-z));
                            const float e = pr - t;
                            const float dz = col_ok ? 2.0f * p.inv_n * e * pr * (1.0f - pr) : 0.f;
                            if (g == 0 && col_ok) {
                                loss = fmaf(e, e, loss);
                                gb += dz;
                            }
                            float dy[8];
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                gw[c] = fmaf(dz, h2[c], gw[c]);
                                dy[c] = h2[c] > 0.f ? dz * hw[c] : 0.f;
                                db[c] += dy[c];
                            }
                            if (col_ok && !*abort_flag) {
                                float4* o = reinterpret_cast<float4*>(p.dy2 + (pix0 + (int64_t)(u - 2) * p.W) * 16 + 8 * g);
                                o[0] = make_float4(dy[0], dy[1], dy[2], dy[3]);
                                o[1] = make_float4(dy[4], dy[5], dy[6], dy[7]);
                            }
                        }
                    }
                    t = t_next;
                }
            }
            if constexpr (!INFER) {
                // partials per CTA: [loss, db2[16], dWh[16], dbh]
                float all[18];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    all[c] = db[c];
                    all[8 + c] = gw[c];
                }
                all[16] = loss;
                all[17] = gb;
                float* out = reinterpret_cast<float*>(smem + oXch) + 128 * g;  // free: every row's exchange is over
                asm volatile("bar.sync 2, 256;" ::: "memory");
                group_sum(all, red, g, warp & 3, lane, out);
                asm volatile("bar.sync %0, 128;" ::"r"(3 + g) : "memory");
                float* part = p.partial + (int64_t)blockIdx.x * kX3FwdWidth;
                if (px < 8) {
                    part[1 + 8 * g + px] = out[px];
                    part[17 + 8 * g + px] = out[8 + px];
                }
                if (g == 0 && px == 0) {
                    part[0] = out[16];
                    part[33] = out[17];
                }
            }
        } else {
            // dy1 = (h1 > 0) conv row; dW1[co][ky][kx] += dy1[co] x(y + ky, x + kx), channel pairs packed
            float2 acc[9][4], db[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                db[c] = make_float2(0.f, 0.f);
#pragma unroll
                for (int k = 0; k < 9; ++k) acc[k][c] = make_float2(0.f, 0.f);
            }
            while (sx_next(p, pos, end, it)) {
                const int nst = it.rows + 2, x = it.x0 + px;
                const bool col_ok = x < p.out_w;
                const uint16_t* mrow = p.mask + ((int64_t)it.z * p.out_h + it.y0) * p.out_w + x;
                const uint8_t* img = p.img + (int64_t)(p.zmap ? p.zmap[it.z] : it.z) * p.H * p.W;
                int sc[3];
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) sc[kx] = sx_refl(x + kx - 2, p.W);
                float w[3][3];  // x at input rows (of the conv row) ky, taps kx
                uint8_t nb[3];
                auto fetch = [&](int r) {  // image row that conv row r - 2's ky = 2 reads: y0 + r, mirrored by 2
                    const uint8_t* src = img + (int64_t)sx_refl(it.y0 + r - 2, p.H) * p.W;
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) nb[kx] = __ldg(src + sc[kx]);
                };
#pragma unroll
                for (int c = 0; c < 8; ++c) s0[c] = s1[c] = 0.f;
#pragma unroll
                for (int ky = 0; ky < 3; ++ky)
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) w[ky][kx] = 0.f;
                fetch(0);
                uint32_t m = 0;
                for (int u = 0; u < nst; ++u, ++q) {
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
                        w[0][kx] = w[1][kx];
                        w[1][kx] = w[2][kx];
                        w[2][kx] = lut[nb[kx]];  // row y0 + u
                    }
                    if (u + 1 < nst) fetch(u + 1);
                    const uint32_t m_next = col_ok && u >= 1 && u + 1 < nst ? mrow[(int64_t)(u - 1) * p.out_w] : 0u;
                    float dy[8];
                    row(dy);
                    if (u >= 2) {
#pragma unroll
                        for (int c = 0; c < 8; ++c) dy[c] = (m >> (8 * g + c)) & 1u ? dy[c] : 0.f;
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float2 d = make_float2(dy[2 * c], dy[2 * c + 1]);
                            db[c].x += d.x;
                            db[c].y += d.y;
#pragma unroll
                            for (int ky = 0; ky < 3; ++ky)
#pragma unroll
                                for (int kx = 0; kx < 3; ++kx)
                                    acc[ky * 3 + kx][c] =
                                        __ffma2_rn(d, make_float2(w[ky][kx], w[ky][kx]), acc[ky * 3 + kx][c]);
                        }
                    }
                    m = m_next;
                }
            }
            // partials per CTA: [144 (co, ky, kx)] then db1[16]
            float all[80];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    all[(2 * c) * 9 + k] = acc[k][c].x;
                    all[(2 * c + 1) * 9 + k] = acc[k][c].y;
                }
                all[72 + 2 * c] = db[c].x;
                all[72 + 2 * c + 1] = db[c].y;
            }
            float* out = xch + 128 * g;
            group_sum(all, red, g, warp & 3, lane, out);
            asm volatile("bar.sync %0, 128;" ::"r"(3 + g) : "memory");
            float* part = p.partial + (int64_t)blockIdx.x * 160;
            if (px < 72) part[72 * g + px] = out[px];
            if (px < 8) part[144 + 8 * g + px] = out[72 + px];
        }
    } else {
        ptx::setmaxnreg_dec<120>();
        // ================= producers ==================================================================
        produce(std::integral_constant<int, 2>{}, tid - 384);
    }

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == 0) ptx::tmem_dealloc(tbase, 512);
}

struct SxConv1 {
    const uint8_t* in;   // slice zmap[z] (z without a map) at in_slice, rows in_pitch apart, H x W
    const int* zmap;
    int64_t in_slice, in_pitch;
    int H, W;
    int y0, x0;          // slice coordinates of the outputs' first row and column, plus 1
    int H1, W1;          // rows and columns of h1
    const float* fw;
    float* h1;           // [z][H1][W1][16]
    uint16_t* mask;      // bit c of [z][H1][W1]: h1[c] > 0 (NULL: not wanted)
    int n_strips;        // of 32 columns
    int64_t total;       // z x n_strips x H1
};

// conv1 + ReLU from the uint8 slice: h1 [B][H+2][W+2][16] FP32 and its mask (bit c: h1[c] > 0). HBM
// writes bound it (66 B per pixel: 85 us on a batch of 32 x 512 x 512; 154 measured, 205 with weights
// broadcast from shared memory). A warp walks down a 32-column strip; a lane keeps all 144 weights
// (packed by channel pairs), its 3x3 input window and the bytes of the next four rows in registers.
__global__ void __launch_bounds__(256, 1) st_conv1(const __grid_constant__ SxConv1 a) {
    __shared__ float lut[256];
    lut[threadIdx.x] = (float)threadIdx.x / 255.0f;
    __syncthreads();
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * 8, me = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    int64_t pos = a.total * me / nw;
    const int64_t end = a.total * (me + 1) / nw;
    const int H1 = a.H1, W1 = a.W1;
    const float* fw = a.fw;
    float2 w[9][8], b[8];  // fw: W1t[tap][co], b1
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        b[c] = make_float2(fw[kSB1 + 2 * c], fw[kSB1 + 2 * c + 1]);
#pragma unroll
        for (int k = 0; k < 9; ++k) w[k][c] = make_float2(fw[k * 16 + 2 * c], fw[k * 16 + 2 * c + 1]);
    }
    while (pos < end) {
        const int64_t col = pos / H1;
        const int y0 = (int)(pos - col * H1), z = (int)(col / a.n_strips), x = (int)(col % a.n_strips) * 32 + lane;
        const int rows = (int)min((int64_t)(H1 - y0), end - pos);
        pos += rows;
        const uint8_t* src = a.in + (int64_t)(a.zmap ? a.zmap[z] : z) * a.in_slice;
        int sc[3];
#pragma unroll
        for (int kx = 0; kx < 3; ++kx) sc[kx] = sx_refl(x + kx - 2 + a.x0, a.W);
        float win[3][3];
        uint8_t nb[4][3];  // four rows of bytes in flight
        auto fetch = [&](int r, uint8_t (&n)[3]) {
            const uint8_t* row = src + (int64_t)sx_refl(y0 + r - 2 + a.y0, a.H) * a.in_pitch;
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) n[kx] = __ldg(row + sc[kx]);
        };
#pragma unroll
        for (int ky = 0; ky < 3; ++ky)
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) win[ky][kx] = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) fetch(i, nb[i]);
        auto step = [&](int r, uint8_t (&n)[3]) {
            if (r >= rows + 2) return;
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) {
                win[0][kx] = win[1][kx];
                win[1][kx] = win[2][kx];
                win[2][kx] = lut[n[kx]];
            }
            if (r + 4 < rows + 2) fetch(r + 4, n);
            if (r < 2) return;
            float2 acc[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] = b[c];
#pragma unroll
            for (int k = 0; k < 9; ++k)
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    acc[c] = __ffma2_rn(make_float2(win[k / 3][k % 3], win[k / 3][k % 3]), w[k][c], acc[c]);
            if (x < W1) {
                const int64_t pix = ((int64_t)z * H1 + y0 + r - 2) * W1 + x;
                uint32_t m = 0;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    m |= (acc[c].x > 0.f ? 1u : 0u) << (2 * c) | (acc[c].y > 0.f ? 1u : 0u) << (2 * c + 1);
                    acc[c] = make_float2(fmaxf(acc[c].x, 0.f), fmaxf(acc[c].y, 0.f));
                }
                float4* o = reinterpret_cast<float4*>(a.h1 + pix * 16);
#pragma unroll
                for (int c = 0; c < 4; ++c) o[c] = make_float4(acc[2 * c].x, acc[2 * c].y, acc[2 * c + 1].x, acc[2 * c + 1].y);
                if (a.mask) a.mask[pix] = (uint16_t)m;
            }
        };
#pragma unroll 1
        for (int r = 0; r < rows + 2; r += 4) {
            step(r, nb[0]);
            step(r + 1, nb[1]);
            step(r + 2, nb[2]);
            step(r + 3, nb[3]);
        }
    }
}

// conv2's weight gradient dW2[co][ci][ky][kx] = sum dy2[co](y, x) h1[ci](y + ky, x + kx) over 16x16
// pixel tiles. FP32 FMA issue bounds it (2,304 per pixel). Lane: input channels 2 (l & 7), + 1 as a
// pair, output channels 4 (l >> 3) .. + 3; a warp takes two tile rows: 36 packed FMAs per pixel for
// three 8-byte window loads and one 16-byte load (scalar FMAs over two output channels: 18 for five
// loads). A ninth warp brings the next tile's 37 KB meanwhile, by bulk copies of whole tile rows; 2 CTAs
// per SM. (With the copies issued by the computing warps, a rendezvous per tile cost 25 %.)
// 32 x 512 x 512: 588 us, of which the FMAs are 517.
constexpr int kG2H = 18 * 18 * 16, kG2D = 16 * 16 * 16;  // floats per tile buffer
constexpr int kG2Smem = 2 * (kG2H + kG2D) * 4 + 48;

__global__ void __maxnreg__(112) st_grad2(const float* dy2, const float* h1, int B, int H, int W, float* partial,
                                                   int* err) {
    extern __shared__ __align__(128) float sm[];
    uint64_t* full = reinterpret_cast<uint64_t*>(sm + 2 * (kG2H + kG2D));
    uint64_t* empty = full + 2;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(full + 4);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, cp = lane & 7, cg = lane >> 3;
    const int tx_n = (W + 15) / 16, ty_n = (H + 15) / 16;
    const int64_t tiles = (int64_t)B * tx_n * ty_n;
    ptx::grid_dep_launch();
    if (t == 0) {
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(&full[i], 1);
            ptx::mbar_init(&empty[i], 8);
        }
        *abort_flag = 0;
        ptx::mbar_fence_init();
    }
    // what a short tile leaves uncovered is finite (stale or zero) in h1 and zero in dy2
    for (int i = t; i < 2 * (kG2H + kG2D); i += 288) sm[i] = 0.f;
    ptx::fence_proxy_async_smem();
    __syncthreads();
    ptx::grid_dep_wait();
    float2 acc[9][4];
    if (warp == 8) {
        uint32_t n = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; ok && tile < tiles; tile += gridDim.x, ++n) {
            const int buf = n & 1;
            const int zi = (int)(tile / ((int64_t)tx_n * ty_n));
            const int rem = (int)(tile - (int64_t)zi * tx_n * ty_n);
            const int y0 = (rem / tx_n) * 16, x0 = (rem % tx_n) * 16;
            const int dr = min(16, H - y0), dc = min(16, W - x0);  // rows, columns of dy2; h1 has two more of each
            ok = x_wait(&empty[buf], ((n >> 1) & 1) ^ 1, abort_flag, err, kXWaitNs);
            if (!ok) break;
            float* sh = sm + buf * (kG2H + kG2D);
            float* sd = sh + kG2H;
            if (dr < 16 || dc < 16) {
                for (int i = lane; i < 256 * 4; i += 32) {
                    const int px = i >> 2;
                    if ((px >> 4) >= dr || (px & 15) >= dc)
                        *reinterpret_cast<float4*>(sd + 4 * i) = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                ptx::fence_proxy_async_smem();  // a later tile's copies overwrite them
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_expect_tx(&full[buf], (uint32_t)(dr * dc + (dr + 2) * (dc + 2)) * 64u);
            __syncwarp();
            if (lane < dr)
                ptx::bulk_copy_g2s(sd + lane * 16 * 16, dy2 + (((int64_t)zi * H + y0 + lane) * W + x0) * 16,
                                   (uint32_t)dc * 64u, &full[buf]);
            if (lane < dr + 2)
                ptx::bulk_copy_g2s(sh + lane * 18 * 16, h1 + (((int64_t)zi * (H + 2) + y0 + lane) * (W + 2) + x0) * 16,
                                   (uint32_t)(dc + 2) * 64u, &full[buf]);
        }
        // copies still in flight (only where the CTA gave up) land before it ends
        const uint64_t t0 = x_gtime();
        for (uint32_t r = n > 2 ? n - 2 : 0; r < n; ++r)
            while (!ptx::mbar_test(&full[r & 1], (r >> 1) & 1) && x_gtime() - t0 <= kXWaitNs) {
            }
    } else {
#pragma unroll
    for (int k = 0; k < 9; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[k][j] = make_float2(0.f, 0.f);
    uint32_t n = 0;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++n) {
        const int buf = n & 1;
        x_wait(&full[buf], (n >> 1) & 1, abort_flag, err, kXWaitNs);
        const float* sh = sm + buf * (kG2H + kG2D) + 2 * cp;
        const float* sd = sm + buf * (kG2H + kG2D) + kG2H + 4 * cg;
#pragma unroll 1
        for (int py = 2 * warp; py < 2 * warp + 2; ++py) {
            float2 w[3][3];  // h1 at rows py + ky, columns px + kx
            auto h_at = [&](int ky, int c) { return *reinterpret_cast<const float2*>(sh + ((py + ky) * 18 + c) * 16); };
#pragma unroll
            for (int ky = 0; ky < 3; ++ky)
#pragma unroll
                for (int kx = 0; kx < 2; ++kx) w[ky][kx + 1] = h_at(ky, kx);
#pragma unroll
            for (int px = 0; px < 16; ++px) {
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) {
                    w[ky][0] = w[ky][1];
                    w[ky][1] = w[ky][2];
                    w[ky][2] = h_at(ky, px + 2);
                }
                const float4 d = *reinterpret_cast<const float4*>(sd + (py * 16 + px) * 16);
                const float2 dd[4] = {make_float2(d.x, d.x), make_float2(d.y, d.y), make_float2(d.z, d.z),
                                      make_float2(d.w, d.w)};
#pragma unroll
                for (int k = 0; k < 9; ++k)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[k][j] = __ffma2_rn(w[k / 3][k % 3], dd[j], acc[k][j]);
            }
        }
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&empty[buf]);
    }
    }
    __syncthreads();
    // the eight warps' sums, in order
    static_assert(8 * 2304 * 4 <= kG2Smem, "the warps' sums fit the tile buffers");
    if (warp < 8) {
#pragma unroll
        for (int k = 0; k < 9; ++k)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
            sm[warp * 2304 + ((4 * cg + j) * 16 + 2 * cp) * 9 + k] = acc[k][j].x;
            sm[warp * 2304 + ((4 * cg + j) * 16 + 2 * cp + 1) * 9 + k] = acc[k][j].y;
        }
    }
    __syncthreads();
    for (int i = t; i < 2304; i += 288) {
        float v = sm[i];
#pragma unroll
        for (int r = 1; r < 8; ++r) v += sm[r * 2304 + i];
        partial[(int64_t)blockIdx.x * 2304 + i] = v;
    }
}

// Every parameter's gradient and the loss from the CTAs' partial sums, in FP64 and a fixed order: thread
// (l, j) of a block adds CTAs j, j + 32, ... of output l of 32 consecutive ones (coalesced loads, ten at
// most, all in flight), then warp j adds the 32 sums of output j.
__global__ void __launch_bounds__(1024) st_reduce(const float* fwd, const float* g2, const float* bwd, float inv_n,
                                                  float* grad, float* loss) {
    __shared__ double sh[32][33];
    ptx::grid_dep_launch();
    ptx::grid_dep_wait();
    const int l = threadIdx.x & 31, j = threadIdx.x >> 5;
    {
        const int o = blockIdx.x * 32 + l;
        const float* src = nullptr;
        int n = kX3Grid, width = 0;
        if (o < kSW2) {  // W1, b1
            src = bwd + o;
            width = 160;
        } else if (o < kSB2) {
            src = g2 + (o - kSW2);
            n = kX3GridG2;
            width = 2304;
        } else if (o <= kSN) {  // b2, head; the loss after the last parameter
            src = fwd + (o == kSN ? 0 : 1 + o - kSB2);
            width = kX3FwdWidth;
        }
        double s = 0.0;
        if (src) {
#pragma unroll 10
            for (int c = j; c < n; c += 32) s += (double)src[(int64_t)c * width];
        }
        sh[j][l] = s;
    }
    __syncthreads();
    // warp j: output 32 blockIdx + j, its 32 partial sums across the lanes
    double s = sh[l][j];
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
    const int o = blockIdx.x * 32 + j;
    if (l == 0) {
        if (o == kSN)
            *loss = (float)(s * (double)inv_n);
        else if (o < kSN)
            grad[o] = (float)s;
    }
}

template <int MODE>
mb_status launch_sx(const SxParams& q, cudaStream_t st) {
    static std::atomic<uint64_t> smem_set{0};
    MB_TRY(set_smem_once(smem_set, st_x3<MODE>, kSmemX));
    constexpr bool BWD = MODE == SX_BWD;
    SxParams p = q;
    p.out_h = BWD ? p.H + 2 : p.H;
    p.out_w = BWD ? p.W + 2 : p.W;
    p.n_strips = (p.out_w + 127) / 128;
    p.total_rows = (int64_t)p.B * p.n_strips * p.out_h;
    const char* stall = getenv("MB_FAULT_STALL");
    p.fault_stall = (stall && stall[0] == '1') ? 1 : 0;
    p.wait_ns = p.fault_stall ? 200000000ull : kXWaitNs;
    // inference: one range per SM, or fewer when a range would get under 2 rows; the training grids are fixed
    const unsigned grid = MODE == SX_INFER ? (unsigned)std::max<int64_t>(1, std::min<int64_t>(kX3Grid, (p.total_rows + 1) / 2)) : kX3Grid;
    MB_CUDA(launch_dependent(st_x3<MODE>, grid, kThreadsX, kSmemX, st, p));
    count_launch();
    MB_CUDA(cudaGetLastError());
    return MB_OK;
}

}  // namespace

mb_status student_x3_grad(const StudentX3& a, cudaStream_t st) {
    const int strips = (a.W + 2 + 31) / 32;
    SxConv1 c{};
    c.in = a.in;
    c.zmap = a.zmap;
    c.in_slice = (int64_t)a.H * a.W;
    c.in_pitch = a.W;
    c.H = a.H;
    c.W = a.W;
    c.H1 = a.H + 2;
    c.W1 = a.W + 2;
    c.fw = a.fw;
    c.h1 = a.h1;
    c.mask = a.mask;
    c.n_strips = strips;
    c.total = (int64_t)a.B * strips * c.H1;
    MB_CUDA(launch_dependent(st_conv1, kX3Grid, 256, 0, st, c));
    count_launch();
    SxParams p{};
    p.fw = a.fw;
    p.B = a.B;
    p.H = a.H;
    p.W = a.W;
    p.zmap = a.zmap;
    p.err = a.err;
    p.in = a.h1;
    p.wpack = a.pack;
    p.target = a.target;
    p.dy2 = a.dy2;
    p.inv_n = a.inv_n;
    p.partial = a.part_fwd;
    MB_TRY(launch_sx<SX_FWD>(p, st));
    static std::atomic<uint64_t> smem_set{0};
    MB_TRY(set_smem_once(smem_set, st_grad2, kG2Smem));
    MB_CUDA(launch_dependent(st_grad2, kX3GridG2, 288, kG2Smem, st, a.dy2, a.h1, a.B, a.H, a.W, a.part_g2, a.err));
    count_launch();
    p.in = a.dy2;
    p.wpack = a.pack + kX3StudentPack;
    p.mask = a.mask;
    p.img = a.in;
    p.partial = a.part_bwd;
    MB_TRY(launch_sx<SX_BWD>(p, st));
    MB_CUDA(launch_dependent(st_reduce, (kSN + 1 + 31) / 32, 1024, 0, st, a.part_fwd, a.part_g2, a.part_bwd, a.inv_n, a.grad,
                             a.loss));
    count_launch();
    MB_CUDA(cudaGetLastError());
    return MB_OK;
}

// Probabilities of a region of z slices: h1 of the region and one pixel around it, then conv2, head and
// sigmoid. h1: [z][rows + 2][cols + 2][16] floats.
mb_status student_x3_infer(const StudentX3Region& a, cudaStream_t st) {
    SxConv1 c{};
    c.in = a.in;
    c.in_slice = a.in_slice;
    c.in_pitch = a.in_pitch;
    c.H = a.h;
    c.W = a.w;
    c.y0 = a.y0;
    c.x0 = a.x0;
    c.H1 = a.rows + 2;
    c.W1 = a.cols + 2;
    c.fw = a.fw;
    c.h1 = a.h1;
    c.n_strips = (c.W1 + 31) / 32;
    c.total = (int64_t)a.z * c.n_strips * c.H1;
    // an ordinary launch for the first chunk of a call: later launches read the weights before their wait
    if (a.first)
        st_conv1<<<kX3Grid, 256, 0, st>>>(c);
    else
        MB_CUDA(launch_dependent(st_conv1, kX3Grid, 256, 0, st, c));
    count_launch();
    MB_CUDA(cudaGetLastError());
    SxParams p{};
    p.in = a.h1;
    p.fw = a.fw;
    p.B = a.z;
    p.H = a.rows;
    p.W = a.cols;
    p.out = a.out;
    p.out_pitch = a.out_pitch;
    p.out_slice = a.out_slice;
    p.out_u8 = a.out_u8;
    p.err = a.err;
    return launch_sx<SX_INFER>(p, st);
}

}  // namespace mb
