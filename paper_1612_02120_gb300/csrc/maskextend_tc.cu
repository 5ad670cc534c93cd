// maskextend_tc.cu - MaskExtend's five max-out convolutions (Sec. 3.2) on the 5th-generation tensor
// cores, FP16 operands and FP32 accumulation; the last one ends with the 1x1 64->3 head and the
// 3-class softmax in its epilogue.
//
// Implicit GEMM per output row y and 128-pixel column strip x0 of a conv with dilation D:
//   D[128 px][N] = sum over taps (ky, kx) and K chunks kc of  A[128 px][16 ch] x B[N][16 ch]^T
// N = 2 x features (the max-out pairs, channels 2c and 2c+1 -> feature c), K = input channels
// padded to a multiple of 16 (12 -> 16, 40 -> 48, 56 -> 64). A for tap (ky, kx) is staged input row
// y + D ky at pixels x0 + D kx .. + 127: one staged row in the no-swizzle K-major layout
// [8-channel chunk][pixel][16 B], the column tap a (D kx x 16)-byte shift of the descriptor.
//
// The weights of the deeper layers (up to 16 taps x 64 x 128 FP16 = 256 KB) do not fit in shared
// memory beside the staged rows, so B is streamed in units of 4 taps (2 for the widest layer) and
// reused over a group of R output rows of one residue class y mod D (R TMEM accumulators: 8 at
// N = 64, else 4). A group's taps run ky-major: step ky reads staged rows m + ky .. m + ky + R - 1,
// so the window of staged rows slides by one row per step. In step 0 the rows are issued one after
// the other (all four taps of ky = 0 resident), so an accumulator is only waited for when its row
// starts while the epilogue drains the previous group's rows in the same order. The issuing thread
// polls one mbarrier per weight unit and per staged row and commits once per unit, per staged row
// and per group: with the tensor pipe reading shared memory at its full rate, each poll or commit
// costs tens of cycles of MMA issue.
//
// Features in global memory are what the next conv reads, already max-filtered, chunk-planar:
// [row][8-channel chunk][column][16 B], so a staged row is a few contiguous runs that one warp fetches
// with bulk copies. (Eight producer warps gathering 4 x 16 B per pixel took ~9,000 cycles for a row of
// the last layer, a quarter of its launch before the first group was staged, and while they ran an MMA
// took 85-100 cycles of the issuing thread against 65 alone.) The epilogue owns the values the filter
// needs: a CTA walks one residue class, so the vertical partner y + D is the next row it drains, and the
// horizontal one x + D is in the same strip. A strip of 128 conv columns yields 128 - D filtered ones, an
// item one conv row more than filtered rows. The maxima are of values already rounded to FP16, so the
// maps are bitwise those of filtering on the load.
//
// 16 sections of 512 x 512, us: 4,766 with gathering producers; 4,595 with whole-warp issue loops; 4,222 with
// rows by bulk copies; 3,138 with two issuing warps, the loader's lanes, ranges without divisions and dependent
// launches (23, 33, 45, 47, 46 a section for the five layers). The multiplies alone are 1,390 at the BF16 rate:
// N = 96 .. 128 MMAs read shared memory at its full 128 B per cycle, beside the streamed weights.
//
// Warp roles (384 threads, 1 CTA per SM, persistent over work items):
//   warps 0, 3   lane 0 issues the MMAs of the even / odd rows of a group (warp 0 also owns TMEM)
//   warp 1       lane 0 streams the weight units into their ring with bulk copies (completion counted
//                on the unit's mbarrier)
//   warp 2       lane c fetches chunk c of the staged rows (as many ahead as shared memory allows, up to 12)
//   warps 4-11   epilogue, two groups of 4 warps, each half of the feature chunks: TMEM -> registers,
//                + bias, max-out, FP16, max-filter, store. Last layer: the first group alone, the 1x1
//                conv to 3 classes and the softmax, FP32 probabilities
// Every mbarrier wait is bounded (a global-timer limit), after which the CTA records
// MB_ERR_TIMEOUT in a mapped host word, stops issuing work, waits (bounded) for its bulk copies in
// flight and frees its TMEM.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "tc_ptx.cuh"

namespace mb {

namespace {

constexpr int kMThreads = 384;
constexpr int kMBRing = 3;   // weight units in flight (a unit is 4 or 2 tap tiles)
constexpr uint64_t kMWaitNs = 4000000000ull;

template <int KC, int N, int D, bool HEAD>
struct MCfg {
    static constexpr int kChunks = 2 * KC;              // 8-channel chunks per staged pixel
    static constexpr int kMP = 128 + 3 * D;              // staged pixels per row
    static constexpr int kOutChunks = N / 16;            // 8-feature chunks of the output
    static constexpr int kARow = kChunks * kMP * 16;     // bytes per staged row
    static constexpr int kBTap = kChunks * N * 16;       // bytes per tap tile [chunk][N][16 B]
    static constexpr int kConsts = N + (HEAD ? 3 * 64 + 3 : 0);  // biases (+ head W[3][64], b[3])
    // output rows per group = TMEM accumulators (512 columns, 64 or 128 apart)
    static constexpr int kR = N <= 64 ? 8 : 4;
    static constexpr int kAccStride = 512 / kR;
    // taps per weight unit (one mbarrier, one release): a whole step's 4 taps, or 2 for the widest
    static constexpr int kBU = KC == 4 ? 2 : 4;
    static constexpr int kBUnit = kBU * kBTap;
    // staged rows: kR in use by a step, the rest filled ahead (as many as fit, up to 12)
    // the strip-edge exchange: 2 rows in turn x output chunks x 4 warps x D pixels x 16 B
    static constexpr int kXch = HEAD ? 0 : 2 * kOutChunks * 4 * D * 16;
    static constexpr int kEpi = HEAD ? 128 : 256;        // epilogue threads
    static constexpr int kStrip = HEAD ? 128 : 128 - D;  // output columns of a strip
    static constexpr int kMore = HEAD ? 0 : 1;           // conv rows of an item beyond its output rows
    static constexpr int kFixed = kMBRing * kBUnit + kXch + kConsts * 4 + 16 + (2 * kMBRing + kR + 3) * 8 + 16;
    static constexpr int kARing = (227 * 1024 - kFixed) / (kARow + 16) < 12 ? (227 * 1024 - kFixed) / (kARow + 16) : 12;
    static constexpr int oA = 0;
    static constexpr int oB = oA + kARing * kARow;
    static constexpr int oXch = oB + kMBRing * kBUnit;
    static constexpr int oConst = oXch + kXch;
    static constexpr int oBar = oConst + ((kConsts * 4 + 15) & ~15);
    static constexpr int kBars = 2 * kARing + 2 * kMBRing + 1 + kR + 2;
    static constexpr int oMisc = oBar + kBars * 8;
    static constexpr int kSmem = oMisc + 16;
    static_assert(kARing >= kR + 1, "staged-row ring");
    static_assert(N % 16 == 0 && N <= 128, "MMA N");
    static_assert(kSmem <= 227 * 1024, "shared memory");
};

struct MeTcParams {
    const __half* in;       // features [row][chunk][in_pitch][8] FP16, src_chunks chunks
    __half* out;            // layers: features in the same layout, N / 16 chunks
    float* probs;           // head: [3][out_h][out_pitch] FP32, planes probs_plane apart
    const uint8_t* wpack;   // 16 tap tiles, then the FP32 constants
    int* err;
    int64_t in_pitch, out_pitch, probs_plane;  // pixels
    int src_chunks;         // 8-channel chunks of the input (the operand's further ones stay zero)
    int out_h, out_w;       // what is written: filtered features; the head: the maps
    int n_strips;
    int total_rows;         // strip-rows of the launch: n_strips x out_h (< 2^31, checked)
    int per_cta, extra;     // total_rows = per_cta x CTAs + extra: the first `extra` CTAs take one more
    int fault_stall;        // test injection: the loaders withhold their copies
    uint64_t wait_ns;
};

__device__ __forceinline__ uint64_t gtime() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err,
                                         uint64_t limit_ns) {
    if (ptx::mbar_test(bar, parity)) return true;  // a completed phase costs one poll
    if (*abort_flag) return false;
    const uint64_t t0 = gtime();
    uint32_t n = 0;
    while (!ptx::mbar_test(bar, parity)) {
        if ((++n & 255u) == 0) {
            if (*abort_flag) return false;
            if (gtime() - t0 > limit_ns) {
                *abort_flag = 1;
                *(volatile int*)err = MB_ERR_TIMEOUT;
                return false;
            }
        }
    }
    return true;
}

struct MeItem {
    int ry, x0, m0, rows;  // written rows y = ry + D (m0 + j), j < rows
};

// Work split: the launch's strip-rows, in (residue class ry, strip, row) order, are cut into one
// equal contiguous range per CTA (every CTA gets the same number of rows, no tail wave); a CTA's
// items are the parts of its range in one (ry, strip) column. Residue class ry has
// hr = ceil((out_h - ry) / D) rows per strip, i.e. base + 1 for ry < rem and base after
// (out_h = D base + rem), so n_strips (ry base + min(ry, rem)) strip-rows precede it. Every role of
// a CTA walks the same sequence. A layer's item of n filtered rows is n + 1 conv rows; an item of n
// conv rows stages n + 3 input rows.
struct MeCursor {
    int g, hi;  // next strip-row, end of this CTA's range
};

__device__ __forceinline__ MeCursor me_begin(const MeTcParams& p) {
    MeCursor c;
    const int b = blockIdx.x;
    c.g = b * p.per_cta + min(b, p.extra);
    c.hi = c.g + p.per_cta + (b < p.extra ? 1 : 0);
    return c;
}

template <int D, int STRIP>
__device__ __forceinline__ bool me_next(const MeTcParams& p, MeCursor& c, MeItem& it) {
    if (c.g >= c.hi) return false;
    const int base = p.out_h / D, rem = p.out_h % D;
    auto before = [&](int ry) { return p.n_strips * (ry * base + min(ry, rem)); };
    int ry = 0;
    while (ry + 1 < D && before(ry + 1) <= c.g) ++ry;
    const int hr = base + (ry < rem ? 1 : 0);  // > 0: before(ry) <= g < before(ry + 1)
    const int off = c.g - before(ry);
    const int strip = off / hr;
    it.ry = ry;
    it.x0 = strip * STRIP;
    it.m0 = off - strip * hr;
    it.rows = min(hr - it.m0, c.hi - c.g);
    c.g += it.rows;
    return true;
}

__device__ __forceinline__ uint4 hmax4(uint4 a, uint4 b) {
    uint4 r;
    const __half2* x = reinterpret_cast<const __half2*>(&a);
    const __half2* y = reinterpret_cast<const __half2*>(&b);
    __half2* o = reinterpret_cast<__half2*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = __hmax2(x[i], y[i]);
    return r;
}

template <int KC, int N, int D, bool HEAD>
__global__ void __launch_bounds__(kMThreads, 1) me_tc_conv(const __grid_constant__ MeTcParams p) {
    using C = MCfg<KC, N, D, HEAD>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* a_full = reinterpret_cast<uint64_t*>(smem + C::oBar);
    uint64_t* a_empty = a_full + C::kARing;
    uint64_t* b_full = a_empty + C::kARing;
    uint64_t* b_empty = b_full + kMBRing;
    uint64_t* acc_full = b_empty + kMBRing;  // one per CTA: a group's accumulators are complete
    uint64_t* acc_free = acc_full + 1;       // per accumulator: drained by the epilogue
    uint64_t* fin = acc_free + C::kR;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::oMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::oMisc + 4);
    const float* cst = reinterpret_cast<const float*>(smem + C::oConst);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // known to be the same in all lanes

    if (tid == 0) {
        for (int i = 0; i < C::kARing; ++i) {
            ptx::mbar_init(&a_full[i], 1);
            ptx::mbar_init(&a_empty[i], 2);
        }
        for (int i = 0; i < kMBRing; ++i) {
            ptx::mbar_init(&b_full[i], 1);
            ptx::mbar_init(&b_empty[i], 2);
        }
        ptx::mbar_init(acc_full, 2);
        for (int i = 0; i < C::kR; ++i) ptx::mbar_init(&acc_free[i], C::kEpi);
        ptx::mbar_init(fin, 1);
        ptx::mbar_init(fin + 1, 1);
        *abort_flag = 0;
        ptx::mbar_fence_init();
    }
    {
        const float* src = reinterpret_cast<const float*>(p.wpack + 16 * C::kBTap);
        float* dst = reinterpret_cast<float*>(smem + C::oConst);
        for (int i = tid; i < C::kConsts; i += kMThreads) dst[i] = __ldg(src + i);
        // channels that the operand has beyond the input's stay zero
        uint4* a = reinterpret_cast<uint4*>(smem + C::oA);
        const int pad = (C::kChunks - p.src_chunks) * C::kMP;
        for (int i = tid; i < C::kARing * pad; i += kMThreads)
            a[(i / pad) * (C::kARow / 16) + p.src_chunks * C::kMP + i % pad] = make_uint4(0, 0, 0, 0);
        ptx::fence_proxy_async_smem();
    }
    if (warp == 0) {
        ptx::tmem_alloc(tmem_slot, 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    // the next launch may set itself up on SMs that are done (only now: its TMEM could otherwise be
    // taken before this launch's)
    ptx::grid_dep_launch();
    const uint32_t tbase = *tmem_slot;
    const uint32_t sbase = ptx::smem_u32(smem);

    if (warp == 0 || warp == 3) {
        // ================= MMA issuers ================================================================
        // The whole warp walks the loop on uniform values, lane 0 issuing: a divergent branch would
        // move every operand of every MMA through vector registers. One thread issues an MMA per 80-93
        // cycles, the tensor pipe takes one per 48 (N = 64) to 64 (N = 128); a row's accumulator is its
        // own, so two warps share the rows of a group (each accumulator's MMAs stay in one thread's order).
            const int odd = warp == 3;
            const uint64_t adesc = ptx::smem_desc(sbase + C::oA, C::kMP * 16, 128);
            const uint64_t bdesc = ptx::smem_desc(sbase + C::oB, N * 16, 128);
            const uint32_t adesc0 = (uint32_t)adesc, a_hi = (uint32_t)(adesc >> 32);
            const uint32_t bdesc0 = (uint32_t)bdesc, b_hi = (uint32_t)(bdesc >> 32);
            const uint32_t lead = lane == 0;
            constexpr uint32_t idesc = ptx::idesc_f32acc(ptx::kFmtF16, 128, N);
            constexpr int kR = C::kR, kBU = C::kBU;
            uint32_t a_seq = 0, u_seq = 0;
            uint32_t free_par = 0;  // bit j: parity of the next use of accumulator j
            bool ok = true;
            // Row j of every group accumulates in TMEM columns kAccStride j (a group always starts
            // at accumulator 0, so a group cannot complete before the epilogue has taken the one
            // before it). Rows are runtime loops and only taps and K chunks are unrolled (the tap
            // shift D kx and the chunk kc are compile-time offsets): a short issue loop stays in
            // the instruction cache beside the other roles' code.
            auto mma_taps = [&](uint32_t ad, uint32_t dcol, uint32_t bd, auto kx0, auto ntaps, auto zero_first) {
                const uint32_t on = ok ? lead : 0u;
#pragma unroll
                for (int t = 0; t < decltype(ntaps)::value; ++t)
#pragma unroll
                    for (int kc = 0; kc < KC; ++kc) {
                        const int kx = decltype(kx0)::value + t;
                        const uint32_t al = ad + (uint32_t)((D * kx * 16 + kc * 2 * C::kMP * 16) >> 4);
                        const uint32_t bl = bd + (uint32_t)(((kx % kBU) * C::kBTap + kc * 2 * N * 16) >> 4);
                        if (decltype(zero_first)::value && t == 0 && kc == 0)
                            ptx::mma_bf16_acc(on, dcol, al, a_hi, bl, b_hi, idesc, 0u);
                        else
                            ptx::mma_bf16_if(on, dcol, al, a_hi, bl, b_hi, idesc);
                    }
            };
            auto unit_desc = [&](uint32_t q) { return bdesc0 + (((q % kMBRing) * C::kBUnit) >> 4); };
            auto wait_unit = [&](uint32_t q) {
                ok = ok && wait_bar(&b_full[q % kMBRing], (q / kMBRing) & 1, abort_flag, p.err, p.wait_ns);
            };
            MeCursor cur = me_begin(p);
            MeItem it;
            while (me_next<D, C::kStrip>(p, cur, it)) {
                const int rows = it.rows + C::kMore;
                const int groups = (rows + kR - 1) / kR;
                int a_known = 0;  // staged rows [0, a_known) of the item are known full
                int a_rel = 0;    // staged rows [0, a_rel) are released
                auto release_upto = [&](int last) {
                    for (; a_rel <= last; ++a_rel) ptx::mma_commit_if(lead, &a_empty[(a_seq + a_rel) % C::kARing]);
                };
                for (int g = 0; g < groups; ++g) {
                    const int rg = min(kR, rows - kR * g);
                    for (int ky = 0; ky < 4; ++ky) {
                        const int s = kR * g + ky;  // staged rows s .. s + rg - 1
                        for (; a_known < s + rg; ++a_known) {
                            const uint32_t q = a_seq + a_known;
                            ok = ok && wait_bar(&a_full[q % C::kARing], (q / C::kARing) & 1, abort_flag, p.err, p.wait_ns);
                        }
                        const uint32_t aslot0 = (a_seq + s) % C::kARing;
                        auto arow = [&](int j) {
                            const uint32_t sl = aslot0 + j < (uint32_t)C::kARing ? aslot0 + j : aslot0 + j - C::kARing;
                            return adesc0 + ((sl * C::kARow) >> 4);
                        };
                        if (ky == 0) {
                            // the step's weight units, then rows one after the other, each waiting
                            // only for its own accumulator
                            for (int u = 0; u < 4 / kBU; ++u) wait_unit(u_seq + u);
                            const uint32_t bd0 = unit_desc(u_seq), bd1 = unit_desc(u_seq + (4 / kBU) - 1);
                            for (int j = odd; j < rg; j += 2) {
                                ok = ok && wait_bar(&acc_free[j], ((free_par >> j) & 1) ^ 1, abort_flag, p.err,
                                                    p.wait_ns);
                                free_par ^= 1u << j;
                                ptx::tc_fence_after();
                                const uint32_t ad = arow(j);
                                const uint32_t dcol = tbase + (uint32_t)(C::kAccStride * j);
                                {
                                    if constexpr (kBU == 4) {
                                        mma_taps(ad, dcol, bd0, std::integral_constant<int, 0>{},
                                                 std::integral_constant<int, 4>{}, std::true_type{});
                                    } else {
                                        mma_taps(ad, dcol, bd0, std::integral_constant<int, 0>{},
                                                 std::integral_constant<int, 2>{}, std::true_type{});
                                        mma_taps(ad, dcol, bd1, std::integral_constant<int, 2>{},
                                                 std::integral_constant<int, 2>{}, std::false_type{});
                                    }
                                }
                            }
                            for (int u = 0; u < 4 / kBU; ++u) ptx::mma_commit_if(lead, &b_empty[(u_seq + u) % kMBRing]);
                            u_seq += 4 / kBU;
                        } else {
                            for (int u = 0; u < 4 / kBU; ++u) {
                                wait_unit(u_seq);
                                ptx::tc_fence_after();
                                const uint32_t bd = unit_desc(u_seq);
                                {
                                    for (int j = odd; j < rg; j += 2) {
                                        const uint32_t ad = arow(j);
                                        const uint32_t dcol = tbase + (uint32_t)(C::kAccStride * j);
                                        if constexpr (kBU == 4) {
                                            mma_taps(ad, dcol, bd, std::integral_constant<int, 0>{},
                                                     std::integral_constant<int, 4>{}, std::false_type{});
                                        } else if (u == 0) {
                                            mma_taps(ad, dcol, bd, std::integral_constant<int, 0>{},
                                                     std::integral_constant<int, 2>{}, std::false_type{});
                                        } else {
                                            mma_taps(ad, dcol, bd, std::integral_constant<int, 2>{},
                                                     std::integral_constant<int, 2>{}, std::false_type{});
                                        }
                                    }
                                }
                                ptx::mma_commit_if(lead, &b_empty[u_seq % kMBRing]);
                                ++u_seq;
                            }
                        }
                        // staged row s is not read by any later step
                        release_upto(s);
                    }
                    ptx::mma_commit_if(lead, acc_full);
                    // rows before the next group's first are done; after the last group, all rows
                    release_upto(g + 1 < groups ? kR * (g + 1) - 1 : rows + 2);
                }
                a_seq += rows + 3;
            }
            if (lane == 0) {
                uint64_t* my = fin + odd;
                ptx::mma_commit(my);
                const uint64_t t0 = gtime();
                while (!ptx::mbar_test(my, 0)) {
                    if (gtime() - t0 > p.wait_ns) {
                        *(volatile int*)p.err = MB_ERR_TIMEOUT;
                        break;
                    }
                }
            }
        __syncwarp();
    } else if (HEAD ? (warp >= 4 && warp < 8) : warp >= 4) {
        // ================= epilogue ===================================================================
        const int px = tid & 127;  // TMEM lane = pixel of the strip
        const uint32_t lanes = (uint32_t)(32 * (warp & 3)) << 16;
        uint32_t n_groups = 0;
        MeCursor cur = me_begin(p);
        MeItem it;
        auto wait_group = [&](int j) {  // at a group's first row: all its accumulators are complete together
            if (j % C::kR == 0) {
                wait_bar(acc_full, n_groups & 1, abort_flag, p.err, p.wait_ns);
                ++n_groups;
                ptx::tc_fence_after();
            }
        };
        if constexpr (HEAD) {
            while (me_next<D, C::kStrip>(p, cur, it)) {
                const int x = it.x0 + px;
                for (int j = 0; j < it.rows; ++j) {
                    wait_group(j);
                    const uint32_t s = j % C::kR;
                    const uint32_t ta = tbase + lanes + (uint32_t)C::kAccStride * s;
                    const int y = it.ry + D * (it.m0 + j);
                    // features c = 0..63 -> logits z_k = b_k + sum_c W[k][c] f_c, in order of c
                    const float* hw = cst + N;
                    float z0 = hw[192], z1 = hw[193], z2 = hw[194];
#pragma unroll
                    for (int q = 0; q < N / 32; ++q) {
                        float v[32];
                        ptx::tmem_ld32(ta + 32u * q, v);
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const int c = 16 * q + i;
                            const float f = fmaxf(v[2 * i] + cst[2 * c], v[2 * i + 1] + cst[2 * c + 1]);
                            z0 = fmaf(hw[c], f, z0);
                            z1 = fmaf(hw[64 + c], f, z1);
                            z2 = fmaf(hw[128 + c], f, z2);
                        }
                    }
                    ptx::tc_fence_before();
                    ptx::mbar_arrive(&acc_free[s]);
                    const float m = fmaxf(z0, fmaxf(z1, z2));
                    const float e0 = expf(z0 - m), e1 = expf(z1 - m), e2 = expf(z2 - m);
                    const float den = e0 + e1 + e2;
                    if (x < p.out_w && !*abort_flag) {
                        float* o = p.probs + (int64_t)y * p.out_pitch + x;
                        o[0] = e0 / den;
                        o[p.probs_plane] = e1 / den;
                        o[2 * p.probs_plane] = e2 / den;
                    }
                }
            }
        } else {
            // chunks C0 .. C0 + NC - 1: conv channels 16 C0 .. -> features 8 C0 ..
            auto run = [&](auto c0_, auto nc_) {
                constexpr int C0 = decltype(c0_)::value, NC = decltype(nc_)::value;
                const int pw = warp & 3, bar = 2 + (C0 > 0);
                uint4* xch = reinterpret_cast<uint4*>(smem + C::oXch) + C0 * 4 * D;
                uint4 prev[NC];
                uint32_t turn = 0;
                while (me_next<D, C::kStrip>(p, cur, it)) {
                    const int x = it.x0 + px;
                    const bool col_ok = px < C::kStrip && x < p.out_w;
                    for (int j = 0; j <= it.rows; ++j) {
                        wait_group(j);
                        const uint32_t s = j % C::kR;
                        const uint32_t ta = tbase + lanes + (uint32_t)C::kAccStride * s + 16u * C0;
                        uint4 w[NC];
#pragma unroll
                        for (int c = 0; c < NC; ++c) {
                            float v[16];
                            ptx::tmem_ld16(ta + 16u * c, v);
                            uint32_t r[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const float4 b = *reinterpret_cast<const float4*>(cst + 16 * (C0 + c) + 4 * i);
                                const __half2 h2 = __floats2half2_rn(fmaxf(v[4 * i] + b.x, v[4 * i + 1] + b.y),
                                                                     fmaxf(v[4 * i + 2] + b.z, v[4 * i + 3] + b.w));
                                r[i] = *reinterpret_cast<const uint32_t*>(&h2);
                            }
                            w[c] = make_uint4(r[0], r[1], r[2], r[3]);
                        }
                        ptx::tc_fence_before();
                        ptx::mbar_arrive(&acc_free[s]);
                        if (j > 0) {
                            // vertical maximum; then the horizontal partner: D lanes on, for the last D
                            // lanes of a warp the next warp's first ones, through shared memory (two
                            // buffers in turn, over item boundaries too: one rendezvous per row)
                            uint4* xc = xch + turn * C::kOutChunks * 4 * D;
                            turn ^= 1;
#pragma unroll
                            for (int c = 0; c < NC; ++c) {
                                prev[c] = hmax4(prev[c], w[c]);
                                if (lane < D) xc[(c * 4 + pw) * D + lane] = prev[c];
                            }
                            asm volatile("bar.sync %0, 128;" ::"r"(bar) : "memory");
                            __half* o = p.out + (((int64_t)(it.ry + D * (it.m0 + j - 1)) * C::kOutChunks + C0) * p.out_pitch + x) * 8;
#pragma unroll
                            for (int c = 0; c < NC; ++c) {
                                uint4 nb;
                                nb.x = __shfl_down_sync(0xffffffffu, prev[c].x, D);
                                nb.y = __shfl_down_sync(0xffffffffu, prev[c].y, D);
                                nb.z = __shfl_down_sync(0xffffffffu, prev[c].z, D);
                                nb.w = __shfl_down_sync(0xffffffffu, prev[c].w, D);
                                if (lane >= 32 - D && pw < 3) nb = xc[(c * 4 + pw + 1) * D + lane - (32 - D)];
                                if (col_ok && !*abort_flag)
                                    *reinterpret_cast<uint4*>(o + (int64_t)c * p.out_pitch * 8) = hmax4(prev[c], nb);
                            }
                        }
#pragma unroll
                        for (int c = 0; c < NC; ++c) prev[c] = w[c];
                    }
                }
            };
            constexpr int kFirst = (C::kOutChunks + 1) / 2;
            if (warp < 8)
                run(std::integral_constant<int, 0>{}, std::integral_constant<int, kFirst>{});
            else
                run(std::integral_constant<int, kFirst>{}, std::integral_constant<int, C::kOutChunks - kFirst>{});
        }
    } else if (warp == 1) {
        // ================= B producer: weight units, in the issuer's order ==========================
        if (lane == 0) {
            uint32_t issued = 0;
            bool go = true;
            MeCursor cur = me_begin(p);
            MeItem it;
            while (go && me_next<D, C::kStrip>(p, cur, it)) {
                const int groups = (it.rows + C::kMore + C::kR - 1) / C::kR;
                for (int g = 0; go && g < groups; ++g)
                    for (int t0 = 0; go && t0 < 16; t0 += C::kBU) {
                        const uint32_t slot = issued % kMBRing;
                        go = wait_bar(&b_empty[slot], ((issued / kMBRing) & 1) ^ 1, abort_flag, p.err, p.wait_ns);
                        if (go && !p.fault_stall) {
                            ptx::mbar_arrive_expect_tx(&b_full[slot], C::kBUnit);
                            for (int t = 0; t < C::kBU; ++t)
                                ptx::bulk_copy_g2s(smem + C::oB + slot * C::kBUnit + t * C::kBTap,
                                                   p.wpack + (size_t)(t0 + t) * C::kBTap, C::kBTap, &b_full[slot]);
                            ++issued;
                        }
                    }
            }
            // the copies still in flight land before the CTA exits (bounded, abort or not)
            for (uint32_t q = issued > (uint32_t)kMBRing ? issued - kMBRing : 0; q < issued; ++q) {
                const uint64_t t0 = gtime();
                while (!ptx::mbar_test(&b_full[q % kMBRing], (q / kMBRing) & 1))
                    if (gtime() - t0 > p.wait_ns) {
                        *(volatile int*)p.err = MB_ERR_TIMEOUT;
                        break;
                    }
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ================= A loader: staged input rows ==============================================
        // (lane c fetches chunk c: one thread's 2 to 7 copies per row took 540-950 cycles)
        uint32_t q = 0;
        bool go = !p.fault_stall;
        ptx::grid_dep_wait();  // the rows are the previous launch's output
        MeCursor cur = me_begin(p);
        MeItem it;
        while (go && me_next<D, C::kStrip>(p, cur, it)) {
            const int nst = it.rows + C::kMore + 3;
            for (int u = 0; u < nst; ++u, ++q) {
                const uint32_t slot = q % C::kARing;
                go = wait_bar(&a_empty[slot], ((q / C::kARing) & 1) ^ 1, abort_flag, p.err, p.wait_ns);
                go = __all_sync(0xffffffffu, go);
                if (!go) break;
                if (lane == 0) ptx::mbar_arrive_expect_tx(&a_full[slot], (uint32_t)(p.src_chunks * C::kMP * 16));
                __syncwarp();
                if (lane < p.src_chunks)
                    ptx::bulk_copy_g2s(
                        smem + C::oA + slot * C::kARow + lane * C::kMP * 16,
                        p.in + (((int64_t)(it.ry + D * (it.m0 + u)) * p.src_chunks + lane) * p.in_pitch + it.x0) * 8,
                        C::kMP * 16, &a_full[slot]);
            }
        }
        // the copies still in flight land before the CTA exits (bounded, abort or not)
        if (lane == 0) {
            const uint64_t t0 = gtime();
            for (uint32_t r = q > (uint32_t)C::kARing ? q - C::kARing : 0; r < q; ++r)
                while (!ptx::mbar_test(&a_full[r % C::kARing], (r / C::kARing) & 1) && gtime() - t0 <= p.wait_ns) {
                }
        }
        __syncwarp();
    }

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == 0) ptx::tmem_dealloc(tbase, 512);
}

uint16_t f16_bits(float f) {
    const __half h = __float2half_rn(f);
    uint16_t b;
    memcpy(&b, &h, 2);
    return b;
}

// Pack conv layer W[n][cin][4][4], b[n] (n < N conv channels) as 16 tap tiles: tile t = 4 ky + kx is
// [chunk kc][row n][8 FP16], input channel 8 kc + e (zero beyond cin); then the N FP32 biases and,
// for the last layer, the head W[3][64] and b[3].
void me_tc_pack(const float* W, const float* b, int cin, int n, int kc, const float* head, std::vector<uint8_t>& out) {
    const int chunks = 2 * kc, tap = chunks * n * 16;
    const size_t consts = (size_t)n + (head ? 3 * 64 + 3 : 0);
    out.assign((size_t)16 * tap + consts * 4, 0);
    for (int o = 0; o < n; ++o)
        for (int ci = 0; ci < cin; ++ci)
            for (int t = 0; t < 16; ++t) {
                const uint16_t h = f16_bits(W[((size_t)o * cin + ci) * 16 + t]);
                memcpy(out.data() + (size_t)t * tap + ((size_t)(ci / 8) * n + o) * 16 + (ci % 8) * 2, &h, 2);
            }
    float* c = reinterpret_cast<float*>(out.data() + (size_t)16 * tap);
    for (int o = 0; o < n; ++o) c[o] = b[o];
    if (head)
        for (int i = 0; i < 3 * 64 + 3; ++i) c[n + i] = head[i];
}

template <int KC, int N, int D, bool HEAD>
mb_status launch_me_tc(const MeTcParams& q, cudaStream_t st) {
    using C = MCfg<KC, N, D, HEAD>;
    static int n_sms = 0;
    if (n_sms == 0) {
        int dev = 0;
        MB_CUDA(cudaGetDevice(&dev));
        MB_CUDA(cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev));
    }
    static std::atomic<uint64_t> smem_set{0};
    MB_TRY(set_smem_once(smem_set, me_tc_conv<KC, N, D, HEAD>, C::kSmem));
    // one range per SM, or fewer when a range would get under 2 rows
    const int grid = std::max(1, std::min(n_sms, (q.total_rows + 1) / 2));
    MeTcParams p = q;
    p.per_cta = q.total_rows / grid;
    p.extra = q.total_rows % grid;
    // the launch's set-up (barriers, constants, TMEM, the first weights) overlaps the end of the one
    // before it; its rows are read after that one's completion (grid_dep_wait)
    MB_CUDA(launch_dependent(me_tc_conv<KC, N, D, HEAD>, (unsigned)grid, kMThreads, C::kSmem, st, p));
    count_launch();
    MB_CUDA(cudaGetLastError());
    return MB_OK;
}

// Layer table: input channels, K chunks of 16, N (= 2 x features), dilation.
constexpr int kMeCin[5] = {12, 32, 40, 48, 56};
constexpr int kMeKc[5] = {1, 2, 3, 3, 4};
constexpr int kMeN[5] = {64, 80, 96, 112, 128};

struct MeTcState {
    uint8_t* d_wpack[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    int* h_err = nullptr;
    int* d_err = nullptr;
};

}  // namespace

mb_status me_tc_prepare(mb_net* net) {
    MeTcState* S = reinterpret_cast<MeTcState*>(net->me_state);
    if (!S) {
        S = new (std::nothrow) MeTcState();
        if (!S) {
            set_error("host allocation failed");
            return MB_ERR_OOM;
        }
        net->me_state = S;
    }
    // API layout: per conv W [N][cin][4][4], b [N]; then the head W [3][64], b [3]
    const float* P = net->host_params.data();
    const float* head = P;
    for (int l = 0; l < 5; ++l) head += (size_t)kMeN[l] * kMeCin[l] * 16 + kMeN[l];
    std::vector<uint8_t> pk;
    for (int l = 0; l < 5; ++l) {
        const size_t nw = (size_t)kMeN[l] * kMeCin[l] * 16;
        me_tc_pack(P, P + nw, kMeCin[l], kMeN[l], kMeKc[l], l == 4 ? head : nullptr, pk);
        P += nw + kMeN[l];
        if (!S->d_wpack[l]) MB_TRY(dev_alloc((void**)&S->d_wpack[l], pk.size()));
        MB_CUDA(cudaMemcpy(S->d_wpack[l], pk.data(), pk.size(), cudaMemcpyHostToDevice));
    }
    if (!S->h_err) {
        if (fault_oom()) {
            set_error("pinned allocation failed (MB_FAULT_OOM injected)");
            return MB_ERR_OOM;
        }
        MB_CUDA(cudaHostAlloc((void**)&S->h_err, sizeof(int), cudaHostAllocMapped));
        *S->h_err = 0;
        MB_CUDA(cudaHostGetDevicePointer((void**)&S->d_err, S->h_err, 0));
    }
    return MB_OK;
}

void me_tc_release(mb_net* net) {
    MeTcState* S = reinterpret_cast<MeTcState*>(net->me_state);
    if (!S) return;
    for (uint8_t* w : S->d_wpack) dev_free(w);
    if (S->h_err) cudaFreeHost(S->h_err);
    delete S;
    net->me_state = nullptr;
}

mb_status me_tc_poll_error(mb_net* net) {
    MeTcState* S = reinterpret_cast<MeTcState*>(net->me_state);
    if (S && S->h_err && *(volatile int*)S->h_err) {
        *(volatile int*)S->h_err = 0;
        set_error("a MaskExtend tensor-core launch gave up waiting (device-side wait limit)");
        return MB_ERR_TIMEOUT;
    }
    return MB_OK;
}

static const int kMeD[5] = {1, 2, 4, 8, 16};

static int me_tc_strips(int layer, int64_t cols) {
    const int strip = layer == 4 ? 128 : 128 - kMeD[layer];
    return (int)((cols + strip - 1) / strip);
}

int64_t me_tc_in_pitch(int layer, int64_t cols) {
    const int d = kMeD[layer], strip = layer == 4 ? 128 : 128 - d;
    return (int64_t)(me_tc_strips(layer, cols) - 1) * strip + 128 + 3 * d;
}

mb_status me_tc_layer(mb_net* net, int layer, const void* in, int64_t in_pitch, void* out, int64_t out_pitch, int rows,
                      int cols, float* probs, int64_t probs_plane, cudaStream_t st) {
    MeTcState* S = reinterpret_cast<MeTcState*>(net->me_state);
    if (!S || !S->d_wpack[layer]) {
        set_error("MaskExtend tensor-core weights not prepared");
        return MB_ERR_NOT_READY;
    }
    if (in_pitch < me_tc_in_pitch(layer, cols)) {
        set_error("MaskExtend: feature pitch too small");
        return MB_ERR_INVALID_ARG;
    }
    MeTcParams p{};
    p.in = static_cast<const __half*>(in);
    p.out = static_cast<__half*>(out);
    p.probs = probs;
    p.wpack = S->d_wpack[layer];
    p.err = S->d_err;
    p.in_pitch = in_pitch;
    p.out_pitch = out_pitch;
    p.probs_plane = probs_plane;
    p.src_chunks = layer == 0 ? 2 : (kMeCin[layer] + 7) / 8;
    p.out_h = rows;
    p.out_w = cols;
    p.n_strips = me_tc_strips(layer, cols);
    if ((int64_t)p.n_strips * rows > 0x7fffffffLL) {
        set_error("MaskExtend: too many strip-rows for one launch");
        return MB_ERR_SHAPE;
    }
    p.total_rows = p.n_strips * rows;
    const char* stall = getenv("MB_FAULT_STALL");
    p.fault_stall = (stall && stall[0] == '1') ? 1 : 0;
    p.wait_ns = p.fault_stall ? 200000000ull : kMWaitNs;
    switch (layer) {
        case 0: return launch_me_tc<1, 64, 1, false>(p, st);
        case 1: return launch_me_tc<2, 80, 2, false>(p, st);
        case 2: return launch_me_tc<3, 96, 4, false>(p, st);
        case 3: return launch_me_tc<3, 112, 8, false>(p, st);
        default: return launch_me_tc<4, 128, 16, true>(p, st);
    }
}

}  // namespace mb
