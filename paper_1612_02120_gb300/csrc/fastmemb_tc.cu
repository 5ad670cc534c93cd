// fastmemb_tc.cu - FastMemb's dense form (Sec. 2.2) on the 5th-generation tensor cores: the
// 32->64 dilated convolutions (+ bias, max-out over channel pairs, the 2x2 max-filter behind them)
// and the 32->2 head (+ the 2-class softmax).
//
// Implicit GEMM per conv row y and 128-pixel column strip x0, conv dilation d:
//   D[128 px][N] = sum over 16 taps (ky, kx) and 2 K-halves of
//                  A_{ky,kx}[128 px][16 ch] x B_{ky,kx}[N][16 ch]^T
// A_{ky,kx} is input row y + d ky, pixels x0 + d kx .. x0 + d kx + 127, taken from one staged row
// in the no-swizzle K-major layout [channel chunk][pixel][16 B]: the column tap is a (d kx x 16)-
// byte shift of the descriptor's start address, so 4 staged rows feed all 32 MMAs of a row.
// Conv rows are walked in steps of d (one residue class y mod d at a time, the max-pooling
// fragments of Sec. 2.2), so each staged row serves 4 consecutive conv rows and is loaded once.
//
// Features in global memory are what the next conv reads, already max-filtered, chunk-planar:
// [slice][row][chunk of 8 channels][column][16 B]. A staged row is then 4 contiguous runs of
// 128 + 3d pixels, fetched by 4 bulk copies of one thread straight into the operand layout, where
// eight producer warps gathering 4 x 16 B per pixel through registers used to bound every layer
// (1024 x 1024 x 8, per launch: BF16 layers 795 us, FP16 638 us, head 509 us). The max-filter moves
// to the epilogue that owns the values: a CTA walks one residue class, so a row's vertical partner
// y + d is the next row it drains (kept in registers), and the horizontal partner x + d is in the
// same strip (one exchange through shared memory). A strip of 128 conv columns yields 128 - d
// filtered ones, and an item one conv row more than filtered rows. Maxima of values already rounded
// to 16 bits are the same in any order, so the maps are bitwise those of filtering on the load.
//
// Two operand types, one template: BF16 and FP16 (both kind::f16 MMAs, A and B of the same type).
// BF16 weights are split W = W_hi + W_lo, both BF16 (W_lo = BF16(W - W_hi)), and stacked along N,
// so each MMA applies both and the result carries BF16 activation rounding only; FP16's 11-bit
// significand makes the split unnecessary for the layers (64 columns per row tap):
//   BF16 layers: 128 columns per row tap ky, n (hi) and 64 + n (lo) of conv channel n
//   FP16 layers: 64 columns per row tap (column n = conv channel n)
//   head:   16 columns per row tap: 0, 1 (hi of classes 0, 1) and 2, 3 (lo); the rest zero
//           (both types keep the split here: the head's MMAs cost the same with it).
// Row taps are stacked along N, T at a time (4; 2 for the BF16 layers, N = 256 either way): staged
// row u is multiplied once per (tap group, kx, K-half) into the accumulators of conv rows u .. u-3,
// a ring of row accumulators (8; 4 for the BF16 layers), one MMA per window, two where it wraps the
// ring. Every MMA accumulates; the epilogue zeroes the used columns of an accumulator after draining
// it. Stacking halves the MMAs that the BF16 layers issue (one row tap per MMA: 755 us). Their ring of
// 4 holds exactly one window, so a staged row's taps 2, 3 go first: they touch only rows already
// started, and conv row u-4 drains meanwhile.
//
// Measured on 1024 x 1024 x 8 (3 nm: 2048 x 2048 x 2), us per launch, producer warps -> this: BF16
// layers 795 -> 621 (2,350 cycles per staged row for 2,048 of MMAs), FP16 layers 638 -> 373 (1,410
// for 1,076; a quarter of the DRAM rate), heads 510 / 555 -> 155.
//
// Warp roles (persistent over work items; layers 384 threads, 1 CTA per SM; head 256 threads, 2):
//   warp 0      TMEM owner; lane 0 issues the MMAs (16-bit operands -> FP32 in TMEM)
//   warp 1      lane 0 fetches staged rows (bulk copies, up to 8 rows ahead)
//   warps 4-7   epilogue: TMEM -> registers; layers: conv channels 0-31, (hi + lo) + bias, max-out,
//               16-bit rounding, max-filter, store; head: z_c = hi + lo + bias,
//               p = 1 / (1 + exp(z0 - z1)), FP32 or uint8 store
//   warps 8-11  layers: the same for conv channels 32-63 (its own barrier; the halves never meet)
// Every mbarrier wait is bounded (a global-timer limit), after which the CTA records
// MB_ERR_TIMEOUT in a mapped host word, stops issuing work, waits for its copies in flight and
// frees its TMEM.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <climits>
#include <string.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "tc_ptx.cuh"

namespace mb {

namespace {

constexpr int kFRing = 8;                // staged rows in flight
constexpr uint64_t kFWaitNs = 4000000000ull;

template <bool HEAD, bool F16>
struct FCfg {
    static constexpr int N = HEAD ? 16 : (F16 ? 64 : 128);  // columns per row tap = per row accumulator
    static constexpr int kTaps = !HEAD && !F16 ? 2 : 4;     // row taps stacked in one MMA
    static constexpr int kTapGroups = 4 / kTaps;
    static constexpr int kBRows = kTaps * N;                // B rows per block
    static constexpr int kBlock = 2 * kBRows * 16;          // [2 chunks][kBRows][16 B] per (kx, K-half, tap group)
    static constexpr int kBBytes = 8 * kTapGroups * kBlock;
    static constexpr int kAcc = !HEAD && !F16 ? 4 : 8;      // ring of row accumulators
    static constexpr int kTmemCols = kAcc * N;
    static constexpr int kMaxD = HEAD ? 16 : 8;       // largest dilation (FastMemb_3nm)
    static constexpr int kFP = 128 + 3 * kMaxD;       // pixels per staged row
    static constexpr int kSlot = 4 * kFP * 16;        // bytes per staged row (4 chunks of 8 16-bit channels)
    static constexpr int kEpi = HEAD ? 128 : 256;     // epilogue threads
    static constexpr int kThreads = 128 + kEpi;
    // the head's shared memory and TMEM (106 KB, 128 columns) leave room for a second CTA, whose
    // rows hide the first one's hand-offs
    static constexpr int kCtas = HEAD ? 2 : 1;
    static constexpr int oB = 0;
    static constexpr int oRing = oB + kBBytes;
    static constexpr int oStage = oRing + kFRing * kSlot;  // layers: 2 rows of [4 chunks][128 px][16 B]
    static constexpr int oBias = oStage + (HEAD ? 0 : 2 * 4 * 128 * 16);
    static constexpr int oBar = oBias + 64 * 4;
    static constexpr int kBars = 2 * kFRing + kAcc + 1;
    static constexpr int oMisc = oBar + kBars * 8;
    static constexpr int kSmem = oMisc + 16;
    static_assert(kCtas * (kSmem + 1024) <= 228 * 1024 && kSmem <= 227 * 1024, "shared memory");
    static_assert(kTmemCols == 128 || kTmemCols == 256 || kTmemCols == 512, "TMEM allocation");
};

struct FmTcParams {
    const uint16_t* in;        // features of the previous stage, [slice][row][chunk][column][8] BF16 or FP16
    void* out;                 // layers: features in the same layout; head: FP32 or uint8 [slice][y][x]
    const uint8_t* wpack;      // B operands then 64 FP32 biases
    int* err;
    int64_t in_slice, in_pitch, out_slice, out_pitch;  // elements per slice, columns per row
    int rows_h, cols_w;        // what is written: filtered rows / columns (layers), map rows / columns (head)
    int d;                     // conv dilation, and that of the max-filter behind it
    int nz, n_strips;          // strips of strip_of(d) columns
    int64_t total_rows;        // strip-rows of the launch: nz x n_strips x rows_h
    int out_u8;                // head: uint8 output round(255 p)
    int fault_stall;           // test injection: the loader withholds its rows
    uint64_t wait_ns;
};

// Columns that one 128-column strip of conv outputs yields.
template <bool HEAD>
__host__ __device__ __forceinline__ int strip_of(int d) {
    return HEAD ? 128 : 128 - d;
}

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

struct FmItem {
    int z, ry, x0, m0, rows;  // rows y = ry + d (m0 + j), j < rows, of what is written
};

// Work split: the launch's strip-rows, in (slice z, residue class ry, strip, row) order, are cut
// into one equal contiguous range per CTA (no tail wave); a CTA's items are the parts of its range
// in one (z, ry, strip) column. Residue class ry has hr = ceil((rows_h - ry) / d) rows per strip:
// base + 1 for ry < rem and base after (rows_h = d base + rem), so n_strips (ry base + min(ry, rem))
// strip-rows of a slice precede it. Every role of a CTA walks the same sequence. A layer's item of
// n filtered rows is n + 1 conv rows; an item of n conv rows stages n + 3 input rows.
struct FmCursor {
    int64_t g, hi;  // next strip-row, end of this CTA's range
};

__device__ __forceinline__ FmCursor fm_begin(const FmTcParams& p) {
    FmCursor c;
    c.g = p.total_rows * (int64_t)blockIdx.x / gridDim.x;
    c.hi = p.total_rows * (int64_t)(blockIdx.x + 1) / gridDim.x;
    return c;
}

template <bool HEAD>
__device__ __forceinline__ bool fm_next(const FmTcParams& p, FmCursor& c, FmItem& it) {
    if (c.g >= c.hi) return false;
    const int64_t per_slice = (int64_t)p.n_strips * p.rows_h;
    it.z = (int)(c.g / per_slice);
    const int r = (int)(c.g - (int64_t)it.z * per_slice);  // strip-row within the slice
    const int base = p.rows_h / p.d, rem = p.rows_h % p.d;
    auto before = [&](int ry) { return p.n_strips * (ry * base + min(ry, rem)); };
    int ry = 0;
    while (ry + 1 < p.d && before(ry + 1) <= r) ++ry;
    const int hr = base + (ry < rem ? 1 : 0);  // > 0: before(ry) <= r < before(ry + 1)
    const int off = r - before(ry);
    const int strip = off / hr;
    it.ry = ry;
    it.x0 = strip * strip_of<HEAD>(p.d);
    it.m0 = off - strip * hr;
    it.rows = (int)min((int64_t)(hr - it.m0), c.hi - c.g);
    c.g += it.rows;
    return true;
}

// element-wise max of 8 packed 16-bit values
template <bool F16>
__device__ __forceinline__ uint4 bmax(uint4 a, uint4 b) {
    using T2 = typename std::conditional<F16, __half2, __nv_bfloat162>::type;
    uint4 r;
    const T2* x = reinterpret_cast<const T2*>(&a);
    const T2* y = reinterpret_cast<const T2*>(&b);
    T2* o = reinterpret_cast<T2*>(&r);
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = __hmax2(x[i], y[i]);
    return r;
}

template <bool HEAD, bool F16>
__global__ void __launch_bounds__(FCfg<HEAD, F16>::kThreads, FCfg<HEAD, F16>::kCtas) fm_tc_conv(const __grid_constant__ FmTcParams p) {
    using C = FCfg<HEAD, F16>;
    constexpr uint32_t kFmt = F16 ? ptx::kFmtF16 : ptx::kFmtBF16;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* row_full = reinterpret_cast<uint64_t*>(smem + C::oBar);
    uint64_t* row_done = row_full + kFRing;
    uint64_t* acc_free = row_done + kFRing;
    uint64_t* fin = acc_free + C::kAcc;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::oMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::oMisc + 4);
    const float* bias = reinterpret_cast<const float*>(smem + C::oBias);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __reduce_max_sync(0xffffffffu, tid >> 5);  // known to be the same in all lanes

    if (tid == 0) {
        for (int i = 0; i < kFRing; ++i) {
            ptx::mbar_init(&row_full[i], 1);
            ptx::mbar_init(&row_done[i], 1);
        }
        for (int i = 0; i < C::kAcc; ++i) ptx::mbar_init(&acc_free[i], C::kEpi);
        ptx::mbar_init(fin, 1);
        *abort_flag = 0;
        ptx::mbar_fence_init();
    }
    {
        const uint4* src = reinterpret_cast<const uint4*>(p.wpack);
        uint4* dst = reinterpret_cast<uint4*>(smem + C::oB);
        for (int i = tid; i < C::kBBytes / 16; i += C::kThreads) dst[i] = __ldg(src + i);
        const uint4* bsrc = reinterpret_cast<const uint4*>(p.wpack + C::kBBytes);
        uint4* bdst = reinterpret_cast<uint4*>(smem + C::oBias);
        for (int i = tid; i < 64 * 4 / 16; i += C::kThreads) bdst[i] = __ldg(bsrc + i);
    }
    if (warp == 0) {
        ptx::tmem_alloc(tmem_slot, C::kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    // the next launch may set itself up on SMs that are done (its TMEM is taken after this one's); this
    // one's set-up overlaps the end of the launch whose features it reads
    ptx::grid_dep_launch();
    const uint32_t tbase = __reduce_max_sync(0xffffffffu, *tmem_slot);  // the same in all lanes, known to be
    const uint32_t sbase = ptx::smem_u32(smem);
    const int d = p.d;
    constexpr int kMore = HEAD ? 0 : 1;  // conv rows of an item beyond its written rows
    // every MMA accumulates (a staged row adds to up to 4 rows at once): the used accumulator columns
    // start at zero, and the epilogue re-zeroes them after each drain
    if (warp >= 4 && warp < 8) {
        const uint32_t lanes = (uint32_t)(32 * (warp - 4)) << 16;
        for (int c = 0; c < C::kTmemCols; c += HEAD ? C::N : 32) {
            if constexpr (HEAD)
                ptx::tmem_st4_zero(tbase + lanes + (uint32_t)c);
            else
                ptx::tmem_st32_zero(tbase + lanes + (uint32_t)c);
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    ptx::grid_dep_wait();

    if (warp == 0) {
        // ================= MMA issuer ================================================================
        // Staged row u of an item feeds conv rows u - ky for ky = 0..3. Staged row q of the CTA's
        // sequence starts conv row q in accumulator slot K-1 - q mod K (the last three staged rows of
        // an item start none), so the rows of a tap group sit in increasing slots; a window that
        // wraps the ring is split in two MMAs. Only rows of the item are written.
        //
        // The issuing thread is the bottleneck of a short row, not the tensor pipe: its MMAs cost
        // 50-100 cycles each to issue, a poll of a completed barrier and a commit 100 (FP16 layers:
        // 1,880 cycles per row for 1,076 of MMAs). So a row has one commit (staged row read, conv row
        // u-3 complete) and one wait (the loader fills a slot only when the accumulator of the same
        // position is drained, so a full row implies a free accumulator; the BF16 layers' ring of 4
        // waits for it separately), both taken between MMAs; the full window is straight-line code;
        // and the whole warp walks the loop on uniform values, lane 0 issuing.
        constexpr int K = C::kAcc, T = C::kTaps, G = C::kTapGroups;
        // instruction descriptor of a window of n row taps (no table: an indexed one is local memory)
        auto idn = [](int n) { return ptx::idesc_f32acc(kFmt, 128, 0) | ((uint32_t)(C::N >> 3) * n) << 17; };
        const uint64_t adesc = ptx::smem_desc(sbase + C::oRing, C::kFP * 16, 128);
        const uint64_t bdesc = ptx::smem_desc(sbase + C::oB, C::kBRows * 16, 128);
        const uint32_t a_hi = (uint32_t)(adesc >> 32), b_hi = (uint32_t)(bdesc >> 32);
        constexpr uint32_t kStep = (uint32_t)(G * C::kBlock) >> 4;  // B block to block
        constexpr uint32_t kHalf = (uint32_t)(2 * C::kFP * 16) >> 4;  // A K-half to K-half
        const uint32_t lead = lane == 0;
        uint32_t q = 0;  // staged row of the CTA's sequence
        bool ok = true;
        auto wait_row = [&](uint32_t r) {
            ok = ok && wait_bar(&row_full[r % kFRing], (r / kFRing) & 1, abort_flag, p.err, p.wait_ns);
        };
        FmCursor cur = fm_begin(p);
        FmItem it;
        while (fm_next<HEAD>(p, cur, it)) {
            const int rows = it.rows + kMore;
            const int nst = rows + 3;
            wait_row(q);
            ptx::tc_fence_after();
            for (int u = 0; u < nst; ++u, ++q) {
                const uint32_t arow = (uint32_t)adesc + (((q % kFRing) * C::kSlot) >> 4);
#pragma unroll
                for (int tg = G - 1; tg >= 0; --tg) {
                    const int lo = max(T * tg, u - rows + 1), hi = min(T * tg + T - 1, u);
                    const uint32_t s0 = (uint32_t)(K - 1) - (q - lo) % (uint32_t)K, on = ok ? lead : 0u;
                    const int nb = hi - lo + 1;
                    const int n1 = min(nb, K - (int)s0);  // taps before the ring wraps
                    const uint32_t d1 = tbase + (uint32_t)C::N * s0;
                    const uint32_t b1 = (uint32_t)bdesc + (uint32_t)((tg * C::kBlock + (lo - T * tg) * C::N * 16) >> 4);
                    // between the MMAs: the commit of the previous row, then the waits for what comes next
                    auto between = [&](int i) {
                        if (tg == G - 1 && i == 0 && u > 0) ptx::mma_commit_if(lead, &row_done[(q - 1) % kFRing]);
                        if (G == 2 && tg == 1 && i == 6)
                            ok = ok && wait_bar(&acc_free[q % K], ((q / K) & 1) ^ 1, abort_flag, p.err, p.wait_ns);
                        if (tg == 0 && i == 4 && u + 1 < nst) wait_row(q + 1);
                    };
                    if (n1 == T) {  // the full window in one piece: straight-line, fixed shape
                        constexpr uint32_t id = ptx::idesc_f32acc(kFmt, 128, T * C::N);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            ptx::mma_bf16_if(on, d1, arow + (i & 1) * kHalf + (uint32_t)((i >> 1) * d), a_hi,
                                             b1 + i * kStep, b_hi, id);
                            between(i);
                        }
                    } else {
                        const uint32_t id1 = idn(n1), id2 = idn(nb - n1), on1 = nb > 0 ? on : 0u, on2 = n1 < nb ? on : 0u;
                        const uint32_t b2 = b1 + ((uint32_t)(n1 * C::N * 16) >> 4);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const uint32_t ai = arow + (i & 1) * kHalf + (uint32_t)((i >> 1) * d);
                            ptx::mma_bf16_if(on1, d1, ai, a_hi, b1 + i * kStep, b_hi, id1);
                            ptx::mma_bf16_if(on2, tbase, ai, a_hi, b2 + i * kStep, b_hi, id2);
                            between(i);
                        }
                    }
                    ptx::tc_fence_after();
                }
            }
            ptx::mma_commit_if(lead, &row_done[(q - 1) % kFRing]);
        }
        if (lane == 0) {
            ptx::mma_commit(fin);
            const uint64_t t0 = gtime();
            while (!ptx::mbar_test(fin, 0)) {
                if (gtime() - t0 > p.wait_ns) {
                    *(volatile int*)p.err = MB_ERR_TIMEOUT;
                    break;
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= loader: staged rows into the A ring =========================================
        // A staged row is 4 chunk runs of 128 + 3d pixels (x0 is any pixel: 16 B each, so every copy
        // is 16-byte aligned). The rows' pitch covers the last strip's overrun; pixels past the
        // domain only reach outputs that are not stored.
        if (lane == 0) {
            const uint32_t bytes = (uint32_t)(128 + 3 * d) * 16u;
            uint32_t q = 0;
            bool ok = true;
            FmCursor cur = fm_begin(p);
            FmItem it;
            while (ok && fm_next<HEAD>(p, cur, it)) {
                const uint16_t* src = p.in + (int64_t)it.z * p.in_slice + (int64_t)it.x0 * 8;
                const int nst = it.rows + kMore + 3;
                for (int u = 0; u < nst; ++u, ++q) {
                    const uint32_t slot = q % kFRing;
                    // ring of 8 accumulators: row q - 8's is drained, which its MMAs' end precedes
                    ok = wait_bar(C::kAcc == kFRing ? &acc_free[slot] : &row_done[slot], ((q / kFRing) & 1) ^ 1, abort_flag,
                                  p.err, p.wait_ns);
                    if (!ok || p.fault_stall) break;
                    const uint16_t* row = src + (int64_t)(it.ry + d * (it.m0 + u)) * 4 * p.in_pitch * 8;
                    uint8_t* dst = smem + C::oRing + slot * C::kSlot;
                    ptx::mbar_arrive_expect_tx(&row_full[slot], 4 * bytes);
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        ptx::bulk_copy_g2s(dst + c * C::kFP * 16, row + (int64_t)c * p.in_pitch * 8, bytes,
                                           &row_full[slot]);
                }
                ok = ok && !p.fault_stall;
            }
            // copies still in flight (a CTA that gives up leaves rows unread) land before the CTA ends
            const uint64_t t0 = gtime();
            for (uint32_t r = q > kFRing ? q - kFRing : 0; r < q; ++r)
                while (!ptx::mbar_test(&row_full[r % kFRing], (r / kFRing) & 1) && gtime() - t0 <= p.wait_ns) {
                }
        }
        __syncwarp();
    } else if (HEAD ? (warp >= 4 && warp < 8) : warp >= 4) {
        // ================= epilogue ===================================================================
        const int px = tid & 127;  // TMEM lane = pixel of the strip
        const uint32_t lanes = (uint32_t)(32 * (warp & 3)) << 16;
        uint32_t q = 0;  // staged row of the CTA's sequence that starts the conv row
        auto wait_conv = [&](uint32_t r) {  // conv row r is complete once staged row r + 3 has been multiplied
            wait_bar(&row_done[(r + 3) % kFRing], ((r + 3) / kFRing) & 1, abort_flag, p.err, p.wait_ns);
            ptx::tc_fence_after();
        };
        auto skip_tail = [&] {  // the item's last three staged rows start no conv row: their slots are free
            for (int t = 0; t < 3; ++t, ++q) ptx::mbar_arrive(&acc_free[q % C::kAcc]);
        };
        FmCursor cur = fm_begin(p);
        FmItem it;
        if constexpr (HEAD) {
            while (fm_next<HEAD>(p, cur, it)) {
                const int x = it.x0 + px;
                for (int j = 0; j < it.rows; ++j, ++q) {
                    wait_conv(q);
                    const uint32_t ta = tbase + lanes + (uint32_t)C::N * ((uint32_t)(C::kAcc - 1) - q % (uint32_t)C::kAcc);
                    const int y = it.ry + d * (it.m0 + j);
                    float c[4];
                    ptx::tmem_ld4(ta, c);
                    ptx::tmem_st4_zero(ta);
                    ptx::tc_fence_before();
                    ptx::mbar_arrive(&acc_free[q % C::kAcc]);
                    const float z0 = (c[0] + c[2]) + bias[0], z1 = (c[1] + c[3]) + bias[1];
                    const float prob = 1.0f / (1.0f + expf(z0 - z1));
                    if (x < p.cols_w && !*abort_flag) {
                        const int64_t idx = (int64_t)it.z * p.out_slice + (int64_t)y * p.out_pitch + x;
                        if (p.out_u8)
                            static_cast<uint8_t*>(p.out)[idx] = (uint8_t)fminf(floorf(255.0f * prob + 0.5f), 255.0f);
                        else
                            static_cast<float*>(p.out)[idx] = prob;
                    }
                }
                skip_tail();
            }
        } else {
            const int half = (warp - 4) >> 2;  // conv channels 32 half .. 32 half + 31
            float b[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) b[c] = bias[32 * half + c];
            uint4* stage = reinterpret_cast<uint4*>(smem + C::oStage) + 2 * half * 128;
            const int partner = px + d < 128 ? px + d : px;
            uint4 prev[2] = {};
            uint32_t turn = 0;  // exchange buffer: two in turn, over item boundaries too, so that one
                                // rendezvous per row keeps a row's readers from the next but one's writers
            while (fm_next<HEAD>(p, cur, it)) {
                const int x = it.x0 + px;
                const bool col_ok = px < 128 - d && x < p.cols_w;
                uint16_t* out = static_cast<uint16_t*>(p.out) + (int64_t)it.z * p.out_slice +
                                ((int64_t)2 * half * p.out_pitch + x) * 8;
                for (int j = 0; j <= it.rows; ++j, ++q) {
                    wait_conv(q);
                    const uint32_t ta = tbase + lanes + 32u * half +
                                        (uint32_t)C::N * ((uint32_t)(C::kAcc - 1) - q % (uint32_t)C::kAcc);
                    float hi[32];
                    ptx::tmem_ld32(ta, hi);
                    ptx::tmem_st32_zero(ta);
                    if constexpr (!F16) {
                        float lo[32];  // column 64 + n
                        ptx::tmem_ld32(ta + 64u, lo);
                        ptx::tmem_st32_zero(ta + 64u);
#pragma unroll
                        for (int c = 0; c < 32; ++c) hi[c] += lo[c];
                    }
                    ptx::tc_fence_before();
                    ptx::mbar_arrive(&acc_free[q % C::kAcc]);
                    uint4 w[2];
                    uint32_t* wr = reinterpret_cast<uint32_t*>(w);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const float a0 = fmaxf(hi[4 * c] + b[4 * c], hi[4 * c + 1] + b[4 * c + 1]);
                        const float a1 = fmaxf(hi[4 * c + 2] + b[4 * c + 2], hi[4 * c + 3] + b[4 * c + 3]);
                        if constexpr (F16) {
                            const __half2 v = __floats2half2_rn(a0, a1);
                            wr[c] = *reinterpret_cast<const uint32_t*>(&v);
                        } else {
                            const __nv_bfloat162 v = __floats2bfloat162_rn(a0, a1);
                            wr[c] = *reinterpret_cast<const uint32_t*>(&v);
                        }
                    }
                    if (j > 0) {
                        const uint4 m0 = bmax<F16>(prev[0], w[0]), m1 = bmax<F16>(prev[1], w[1]);
                        uint4* st = stage + turn * 512;
                        turn ^= 1;
                        st[px] = m0;
                        st[128 + px] = m1;
                        asm volatile("bar.sync %0, 128;" ::"r"(2 + half) : "memory");
                        const uint4 f0 = bmax<F16>(m0, st[partner]), f1 = bmax<F16>(m1, st[128 + partner]);
                        if (col_ok && !*abort_flag) {
                            uint16_t* o = out + (int64_t)(it.ry + d * (it.m0 + j - 1)) * 4 * p.out_pitch * 8;
                            *reinterpret_cast<uint4*>(o) = f0;
                            *reinterpret_cast<uint4*>(o + p.out_pitch * 8) = f1;
                        }
                    }
                    prev[0] = w[0];
                    prev[1] = w[1];
                }
                skip_tail();
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == 0) ptx::tmem_dealloc(tbase, C::kTmemCols);
}

uint16_t bf16_bits_rn(float f) {
    uint32_t u;
    memcpy(&u, &f, 4);
    if ((u & 0x7f800000u) == 0x7f800000u) return (uint16_t)(u >> 16);
    u += 0x7fffu + ((u >> 16) & 1u);
    return (uint16_t)(u >> 16);
}

float bf16_value(uint16_t b) {
    const uint32_t u = (uint32_t)b << 16;
    float f;
    memcpy(&f, &u, 4);
    return f;
}

uint16_t f16_bits_rn(float f) {
    const __half h = __float2half_rn(f);
    uint16_t u;
    memcpy(&u, &h, 2);
    return u;
}

float f16_value(uint16_t b) {
    __half h;
    memcpy(&h, &b, 2);
    return __half2float(h);
}

// Pack a conv 4x4 32->C layer W[c][ci][ky][kx], b[c] as B operands: blocks of [chunk kc][row][8
// 16-bit], ci = 16 h + 8 kc + e, per (column tap kx, K-half h, group of T row taps); in a block, row
// N (ky mod T) + c. Part 0 of a weight is T(W), part 1 T(W - T(W)) for T = BF16 (layers and head) or
// FP16 (the head only: FP16 layers carry part 0 alone), 64 rows (layers) or 2 (head) further on.
// Then 64 FP32 biases.
template <bool HEAD, bool F16>
void fm_pack(const float* W, const float* b, int channels, std::vector<uint8_t>& out) {
    using C = FCfg<HEAD, F16>;
    constexpr bool kLo = HEAD || !F16;
    out.assign(C::kBBytes + 64 * 4, 0);
    for (int c = 0; c < channels; ++c)
        for (int ci = 0; ci < 32; ++ci)
            for (int ky = 0; ky < 4; ++ky)
                for (int kx = 0; kx < 4; ++kx) {
                    const int h = ci / 16, kc = (ci % 16) / 8, e = ci % 8;
                    const float w = W[((c * 32 + ci) * 4 + ky) * 4 + kx];
                    const uint16_t whi = F16 ? f16_bits_rn(w) : bf16_bits_rn(w);
                    const uint16_t wlo =
                        F16 ? f16_bits_rn(w - f16_value(whi)) : bf16_bits_rn(w - bf16_value(whi));
                    const int rhi = C::N * (ky % C::kTaps) + c, rlo = rhi + (HEAD ? 2 : 64);
                    const int blk_i = (kx * 2 + h) * C::kTapGroups + ky / C::kTaps;
                    uint8_t* blk = out.data() + blk_i * C::kBlock + kc * C::kBRows * 16;
                    memcpy(blk + rhi * 16 + e * 2, &whi, 2);
                    if (kLo) memcpy(blk + rlo * 16 + e * 2, &wlo, 2);
                }
    std::vector<float> bias(64, 0.f);
    for (int c = 0; c < channels; ++c) bias[c] = b[c];
    memcpy(out.data() + C::kBBytes, bias.data(), 64 * 4);
}

template <bool HEAD, bool F16>
mb_status launch_fm_tc(const FmTcParams& p, cudaStream_t st) {
    using C = FCfg<HEAD, F16>;
    static int n_sms = 0;
    if (n_sms == 0) {
        int dev = 0;
        MB_CUDA(cudaGetDevice(&dev));
        MB_CUDA(cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev));
    }
    static std::atomic<uint64_t> smem_set{0};
    MB_TRY(set_smem_once(smem_set, fm_tc_conv<HEAD, F16>, C::kSmem));
    // one range per resident CTA, or fewer when a range would get under 2 rows (each costs 4 more
    // staged rows: a launch this small is latency, not throughput)
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)n_sms * C::kCtas, (p.total_rows + 1) / 2));
    MB_CUDA(launch_dependent(fm_tc_conv<HEAD, F16>, (unsigned)grid, C::kThreads, C::kSmem, st, p));
    count_launch();
    MB_CUDA(cudaGetLastError());
    return MB_OK;
}

}  // namespace

struct FmTcState {
    uint8_t* d_wpack[4] = {nullptr, nullptr, nullptr, nullptr};  // the 32->64 convs, then the head
    int* h_err = nullptr;
    int* d_err = nullptr;
};

mb_status fm_tc_prepare(mb_net* net) {
    FmTcState* S = reinterpret_cast<FmTcState*>(net->fm_state);
    if (!S) {
        S = new (std::nothrow) FmTcState();
        if (!S) {
            set_error("host allocation failed");
            return MB_ERR_OOM;
        }
        net->fm_state = S;
    }
    // API layout: W1 [64][1][4][4], b1 [64], then per 32->64 conv W [64][32][4][4], b [64], then the
    // head W [2][32][4][4], b [2]
    const int nc = fastmemb_convs(net->family);
    const float* P = net->host_params.data() + 64 * 16 + 64;
    std::vector<uint8_t> pk;
    const bool f16 = net->prec == MB_PREC_FP16;
    for (int l = 0; l < nc - 1; ++l) {
        const bool head = l == nc - 2;
        const int co = head ? 2 : 64;
        if (!head)
            f16 ? fm_pack<false, true>(P, P + co * 32 * 16, co, pk) : fm_pack<false, false>(P, P + co * 32 * 16, co, pk);
        else
            f16 ? fm_pack<true, true>(P, P + co * 32 * 16, co, pk) : fm_pack<true, false>(P, P + co * 32 * 16, co, pk);
        P += co * 32 * 16 + co;
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

void fm_tc_release(mb_net* net) {
    FmTcState* S = reinterpret_cast<FmTcState*>(net->fm_state);
    if (!S) return;
    for (uint8_t* w : S->d_wpack) dev_free(w);
    if (S->h_err) cudaFreeHost(S->h_err);
    delete S;
    net->fm_state = nullptr;
}

mb_status fm_tc_poll_error(mb_net* net) {
    FmTcState* S = reinterpret_cast<FmTcState*>(net->fm_state);
    if (S && S->h_err && *(volatile int*)S->h_err) {
        *(volatile int*)S->h_err = 0;
        set_error("a FastMemb tensor-core launch gave up waiting (device-side wait limit)");
        return MB_ERR_TIMEOUT;
    }
    return MB_OK;
}

int fm_tc_strips(bool head, int64_t cols, int d) {
    const int s = head ? strip_of<true>(d) : strip_of<false>(d);
    return (int)((cols + s - 1) / s);
}

int64_t fm_tc_in_pitch(bool head, int64_t cols, int d) {
    const int s = head ? strip_of<true>(d) : strip_of<false>(d);
    return (int64_t)(fm_tc_strips(head, cols, d) - 1) * s + 128 + 3 * d;
}

mb_status fm_tc_layer(mb_net* net, int layer, const void* in, int64_t in_slice, int64_t in_pitch, void* out,
                      int64_t out_slice, int64_t out_pitch, int rows, int cols, int d, int nz, int out_u8,
                      cudaStream_t st) {
    FmTcState* S = reinterpret_cast<FmTcState*>(net->fm_state);
    if (!S || !S->d_wpack[layer]) {
        set_error("FastMemb tensor-core weights not prepared");
        return MB_ERR_NOT_READY;
    }
    const bool head = layer == fastmemb_convs(net->family) - 2;
    if (in_pitch < fm_tc_in_pitch(head, cols, d) || d > (head ? FCfg<true, true>::kMaxD : FCfg<false, true>::kMaxD)) {
        set_error("FastMemb: feature pitch too small or dilation too large");
        return MB_ERR_INVALID_ARG;
    }
    FmTcParams p{};
    p.in = static_cast<const uint16_t*>(in);
    p.out = out;
    p.wpack = S->d_wpack[layer];
    p.err = S->d_err;
    p.in_slice = in_slice;
    p.in_pitch = in_pitch;
    p.out_slice = out_slice;
    p.out_pitch = out_pitch;
    p.rows_h = rows;
    p.cols_w = cols;
    p.d = d;
    p.nz = nz;
    p.out_u8 = out_u8;
    p.n_strips = fm_tc_strips(head, cols, d);
    p.total_rows = (int64_t)nz * p.n_strips * rows;
    const char* stall = getenv("MB_FAULT_STALL");
    p.fault_stall = (stall && stall[0] == '1') ? 1 : 0;
    p.wait_ns = p.fault_stall ? 200000000ull : kFWaitNs;
    if (net->prec == MB_PREC_FP16) return head ? launch_fm_tc<true, true>(p, st) : launch_fm_tc<false, true>(p, st);
    return head ? launch_fm_tc<true, false>(p, st) : launch_fm_tc<false, false>(p, st);
}

}  // namespace mb
