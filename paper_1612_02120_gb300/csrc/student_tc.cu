// student_tc.cu - inference of the distilled student (the fast pass of the multi-pass idea, Sec. 1)
// in one fused kernel on the 5th-generation tensor cores, for BF16 student nets:
//   x = u/255 (mirror-padded by 2) -> conv3x3 1->16 + b, ReLU -> conv3x3 16->16 + b, ReLU
//   -> conv1x1 16->1 + b -> sigmoid
// Both convolutions are implicit GEMMs per 128-pixel strip row (M = 128 pixels, operands in the
// no-swizzle K-major layout [8-element chunk][pixel][16 B]):
// Rows are handed from role to role two at a time.
//   layer 1  D1[px][r][co] = sum_kx A1[px + kx][k] x W1[co][k - r][kx], rows r = 0, 1 of the pair, with
//            A1[q][k] = u(row - 1 + k, q): the pair's four input rows are stacked along K (an input byte
//            is exact in BF16), its two output rows along N, the column tap kx is a kx x 16-byte shift
//            of the descriptor start; 3 MMAs (N = 32, K = 16) per pair.
//            The epilogue scales by 1/255 in FP32, adds the bias, rounds to BF16 and applies ReLU
//            into a ring of staged feature rows.
//   layer 2  each staged row r is multiplied once per column tap kx with the three row taps stacked
//            along N (N = 48: blocks for output rows r-2, r-1, r with row taps 2, 1, 0), accumulating
//            into a ring of 6 x 2 row accumulators (windows that wrap the ring are split in two MMAs).
//            The epilogue adds the bias, applies ReLU, the head and the sigmoid in FP32 and stores.
// A strip covers 126 output columns (128 layer-1 pixels, the last two only feed the column taps).
//
// What bounds it: the shared-memory pipe (86 % busy: an MMA of N = 48 reads 4 KB of pixels for 1.5 KB
// of weights) and, close behind, instruction issue (61 %) and the ALU (50 %: max and BF16 packing). 8
// slices of 4096 x 4096: 1,921 us with rows handed over singly and one diverged lane issuing (a
// wait, a commit and every MMA's operands through vector registers per row); 1,508 in pairs with whole
// warps walking the issue loops; 1,424 with layer 1's two rows in one MMA; 1,238 with those loops on
// branches known to be uniform (and no spills); 1,210 with ReLU on packed pairs. Measured and not
// taken: a layer-2 epilogue of two warp groups, a row each (1,307: the roles then share 64 registers a
// thread), and fewer registers for the builders to the epilogue's profit (2,123: the builders spill).
//
// Warp roles (384 threads, two CTAs per SM, persistent over work items):
//   warp 0      TMEM owner (256 columns: layer-2 ring 0..191, layer-1 ring 192..255); issues the
//               layer-1 MMAs
//   warp 3      issues the layer-2 MMAs (a warp stalls ~100 cycles on each commit; with two issuing
//               warps the tensor core keeps working meanwhile)
//   warps 1-2   operand builders: keep four input rows per column in registers and write the
//               layer-1 operand (one 8-byte store per pixel per pair)
//   warps 4-7   layer-1 epilogue (TMEM lane = layer-1 pixel)
//   warps 8-11  layer-2 epilogue and head (TMEM lane = output pixel)
// Every mbarrier wait is bounded (a global-timer limit), after which the CTA records
// MB_ERR_TIMEOUT in a mapped host word, stops issuing work and frees its TMEM.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "internal.h"
#include "tc_ptx.cuh"

namespace mb {

namespace {

constexpr int kSThreads = 384;
constexpr int kSW = 126;                  // output columns per strip
constexpr int kSPitch = 136;              // pixels per operand row (128 + the column taps' overrun)
constexpr int kSRowB = 2 * kSPitch * 16;  // bytes per operand row: 2 chunks (K = 16 BF16)
// rings in row pairs (every role hands rows over two at a time)
constexpr int kNA1 = 3;                   // layer-1 operand row pairs in flight
constexpr int kNS = 4;                    // staged layer-1 feature row pairs
constexpr int kKL = 2;                    // layer-1 accumulator pairs, 32 TMEM columns each
constexpr int kKA = 6;                    // layer-2 accumulator pairs, 32 TMEM columns each
constexpr int kSTmem = 256;
constexpr int kL1Col = 32 * kKA;          // first TMEM column of the layer-1 ring
constexpr int kB1Tap = 2 * 32 * 16;       // per column tap: [2 chunks][row of the pair, co][16 B]
constexpr int kB1 = 3 * kB1Tap;
constexpr int kB2Group = 2 * 48 * 16;     // per column tap: [2 chunks][48 rows][16 B]
constexpr int kB2 = 3 * kB2Group;
constexpr int kSConst = 64;               // b1[16] | b2[16] | head w[16] | head b | 1/255
constexpr int kCB1 = 0, kCB2 = 16, kCWH = 32, kCBH = 48, kCInv = 49;
constexpr int oSB1 = 0;
constexpr int oSB2 = oSB1 + kB1;
constexpr int oSA1 = oSB2 + kB2;
constexpr int oSS = oSA1 + kNA1 * kSRowB;
constexpr int oSConst = oSS + kNS * 2 * kSRowB;
constexpr int oSBar = oSConst + kSConst * 4;
constexpr int kSBars = 2 * kNA1 + 2 * kKL + 2 * kNS + 2 * kKA + 2;
constexpr int oSMisc = oSBar + kSBars * 8;
constexpr int kSUsed = oSMisc + 16;
// Requested shared memory: at most two CTAs fit on an SM, so their TMEM (2 x 256 columns) always
// fits and no CTA waits in tcgen05.alloc.
constexpr int kSSmem = 80 * 1024;
constexpr int kWpack = kB1 + kB2 + kSConst * 4;
constexpr uint64_t kSWaitNs = 4000000000ull;
// forward layout of the student's parameters (as packed for the CUDA-core path)
constexpr int kFW1 = 0, kFB1 = 144, kFW2 = 160, kFB2 = 2464, kFWH = 2480, kFBH = 2496;
static_assert(kSUsed <= kSSmem && 3 * kSSmem > 227 * 1024, "shared memory");
static_assert(oSA1 % 16 == 0 && oSS % 16 == 0 && oSBar % 8 == 0, "alignment");
static_assert(2 * kSTmem <= 512 && kL1Col + 32 * kKL <= kSTmem, "TMEM of two CTAs");

struct StTcParams {
    const uint8_t* in;        // slice z at in + z in_slice; row pitch in_pitch
    void* out;                // region output, [z][rows][cols] with out_pitch / out_slice
    const uint8_t* wpack;     // B operands then the FP32 constants
    int* err;
    int64_t in_slice, in_pitch, out_slice, out_pitch;
    int h, w;                 // slice
    int y0, x0, rows, cols;   // region
    int n_strips;
    int col_pairs;            // row pairs of a strip: ceil(rows / 2)
    int64_t total_pairs;      // row pairs of the launch: z x n_strips x col_pairs
    int out_u8;
    int fault_stall;
    uint64_t wait_ns;
};

__device__ __forceinline__ uint64_t gtime() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// A completed phase costs one poll: the abort flag is read only once the phase is found incomplete.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err,
                                         uint64_t limit_ns) {
    if (ptx::mbar_test(bar, parity)) return true;
    if (*abort_flag) return false;
    const uint64_t t0 = gtime();
    uint32_t n = 0;
    // mbarrier.try_wait suspends the thread for a while by itself; no extra sleep between polls
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

__device__ __forceinline__ int refl(int t, int n) { return t < 0 ? -t : (t >= n ? 2 * (n - 1) - t : t); }

struct StItem {
    int z, m0, rows, s0, ncol;  // region rows m0 .. m0 + rows - 1 (m0 even), columns s0 .. s0 + ncol - 1
    int pairs;                  // output row pairs; an odd last row's partner is computed and not stored
};

// Work split: the launch's strip row pairs, in (slice, strip, pair) order, are cut into one equal
// contiguous range per CTA (no tail wave); a CTA's items are the parts of its range in one (slice,
// strip) column. Every role of a CTA walks the same sequence.
struct StCursor {
    int64_t g, hi;  // next strip row pair, end of this CTA's range
};

__device__ __forceinline__ StCursor st_begin(const StTcParams& p) {
    StCursor c;
    c.g = p.total_pairs * (int64_t)blockIdx.x / gridDim.x;
    c.hi = p.total_pairs * (int64_t)(blockIdx.x + 1) / gridDim.x;
    return c;
}

__device__ __forceinline__ bool st_next(const StTcParams& p, StCursor& c, StItem& it) {
    if (c.g >= c.hi) return false;
    const int64_t col = c.g / p.col_pairs;  // (slice, strip) column
    it.z = (int)(col / p.n_strips);
    const int strip = (int)(col - (int64_t)it.z * p.n_strips);
    const int pair = (int)(c.g - col * p.col_pairs);
    // (the shuffle makes it known to be the same in all lanes: role loops stay on uniform branches)
    it.pairs = __shfl_sync(0xffffffffu, (int)min((int64_t)(p.col_pairs - pair), c.hi - c.g), 0);
    it.m0 = 2 * pair;
    it.rows = min(p.rows - it.m0, 2 * it.pairs);
    it.s0 = strip * kSW;
    it.ncol = min(kSW, p.cols - it.s0);
    c.g += it.pairs;
    return true;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

// max(x, 0) of a BF16 pair (after the rounding it gives the same as before it, in half the instructions)
__device__ __forceinline__ uint32_t relu2(uint32_t v) {
    const __nv_bfloat162 h = __hmax2(*reinterpret_cast<__nv_bfloat162*>(&v), __float2bfloat162_rn(0.f));
    return *reinterpret_cast<const uint32_t*>(&h);
}

__global__ void __launch_bounds__(kSThreads, 2) st_tc_infer(const __grid_constant__ StTcParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    uint64_t* a1_full = reinterpret_cast<uint64_t*>(smem + oSBar);
    uint64_t* a1_empty = a1_full + kNA1;
    uint64_t* l1_full = a1_empty + kNA1;
    uint64_t* l1_free = l1_full + kKL;
    uint64_t* s_full = l1_free + kKL;
    uint64_t* s_empty = s_full + kNS;
    uint64_t* l2_full = s_empty + kNS;
    uint64_t* l2_free = l2_full + kKA;
    uint64_t* fin = l2_free + kKA;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + oSMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + oSMisc + 4);
    const float* cst = reinterpret_cast<const float*>(smem + oSConst);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // known to be the same in all lanes

    if (tid == 0) {
        for (int i = 0; i < kNA1; ++i) {
            ptx::mbar_init(&a1_full[i], 2);
            ptx::mbar_init(&a1_empty[i], 1);
        }
        for (int i = 0; i < kKL; ++i) {
            ptx::mbar_init(&l1_full[i], 1);
            ptx::mbar_init(&l1_free[i], 4);
        }
        for (int i = 0; i < kNS; ++i) {
            ptx::mbar_init(&s_full[i], 4);
            ptx::mbar_init(&s_empty[i], 1);
        }
        for (int i = 0; i < kKA; ++i) {
            ptx::mbar_init(&l2_full[i], 1);
            ptx::mbar_init(&l2_free[i], 4);
        }
        ptx::mbar_init(fin, 1);
        ptx::mbar_init(fin + 1, 1);
        *abort_flag = 0;
        ptx::mbar_fence_init();
    }
    {
        // both operand rings start zero: the second K chunk of the layer-1 operand and the pixels
        // past 127 of every row (read by the column taps, never written) stay zero
        uint4* r = reinterpret_cast<uint4*>(smem + oSA1);
        for (int i = tid; i < (kNA1 + 2 * kNS) * kSRowB / 16; i += kSThreads) r[i] = make_uint4(0, 0, 0, 0);
    }
    if (warp == 0) {
        ptx::tmem_alloc(tmem_slot, kSTmem);
        ptx::tmem_relinquish();
    }
    ptx::grid_dep_wait();  // the operands are the packing launch's, which this one's set-up overlaps
    {
        const uint4* src = reinterpret_cast<const uint4*>(p.wpack);
        uint4* dst = reinterpret_cast<uint4*>(smem + oSB1);
        for (int i = tid; i < (kB1 + kB2) / 16; i += kSThreads) dst[i] = src[i];
        const float* csrc = reinterpret_cast<const float*>(p.wpack + kB1 + kB2);
        float* cdst = reinterpret_cast<float*>(smem + oSConst);
        for (int i = tid; i < kSConst; i += kSThreads) cdst[i] = csrc[i];
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tbase = *tmem_slot;
    const uint32_t sbase = ptx::smem_u32(smem);
    if (warp >= 8) {
        // every layer-2 accumulator starts at zero (its MMAs only accumulate)
        const uint32_t lanes = (uint32_t)(32 * (warp - 8)) << 16;
        for (int sl = 0; sl < kKA; ++sl) ptx::tmem_st32_zero(tbase + lanes + 32u * sl);
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();

    if (warp == 0 || warp == 3) {
        // ================= MMA issuers: warp 0 layer 1, warp 3 layer 2 ================================
        // Each issues, commits and finally drains only its own MMAs; they meet only through the
        // layer-1 epilogue (layer 1 runs ahead as far as its accumulators allow). The per-row chain of
        // waits, MMAs and commits of one thread is what bounds the issue of MMAs this small, so a wait
        // and a commit serve two rows, and the whole warp walks uniform code with lane 0 issuing.
        const uint32_t lead = lane == 0;
        constexpr uint32_t id16 = ptx::idesc_f32acc(ptx::kFmtBF16, 128, 16);
        constexpr uint32_t id32 = ptx::idesc_f32acc(ptx::kFmtBF16, 128, 32);
        constexpr uint32_t id48 = ptx::idesc_f32acc(ptx::kFmtBF16, 128, 48);
        bool ok = true;
        if (warp == 0) {
            const uint64_t ad64 = ptx::smem_desc(sbase + oSA1, kSPitch * 16, 128);
            const uint64_t bd64 = ptx::smem_desc(sbase + oSB1, 32 * 16, 128);
            const uint32_t a_lo = (uint32_t)ad64, a_hi = (uint32_t)(ad64 >> 32);
            const uint32_t b_lo = (uint32_t)bd64, b_hi = (uint32_t)(bd64 >> 32);
            uint32_t as = 0, aph = 0;  // operand pair slot and phase
            uint32_t ls = 0, lph = 0;  // accumulator pair slot and phase
            StCursor cur = st_begin(p);
            StItem it;
            while (st_next(p, cur, it)) {
                for (int k = 0; k <= it.pairs; ++k) {
                    ok = ok && wait_bar(&a1_full[as], aph, abort_flag, p.err, p.wait_ns);
                    ok = ok && wait_bar(&l1_free[ls], lph ^ 1, abort_flag, p.err, p.wait_ns);
                    ptx::tc_fence_after();
                    const uint32_t on = ok ? lead : 0u;
                    const uint32_t al = a_lo + as * (uint32_t)(kSRowB >> 4);
                    const uint32_t dc = tbase + kL1Col + 32u * ls;
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx)
                        ptx::mma_bf16_acc(on, dc, al + kx, a_hi, b_lo + (uint32_t)((kx * kB1Tap) >> 4), b_hi, id32,
                                          kx ? 1u : 0u);
                    ptx::mma_commit_if(lead, &l1_full[ls]);
                    ptx::mma_commit_if(lead, &a1_empty[as]);
                    if (++as == kNA1) {
                        as = 0;
                        aph ^= 1;
                    }
                    if (++ls == kKL) {
                        ls = 0;
                        lph ^= 1;
                    }
                }
            }
        } else {
            // Staged row u of an item feeds output rows u-2+i, i = 0..2, with row tap 2-i. Staged pair k
            // starts output pair k (rows 2k, 2k + 1) and completes pair k - 1: its first row covers
            // columns (pair k - 1: both rows) (pair k: first row), its second row (pair k - 1: second
            // row) (pair k: both rows), 48 contiguous TMEM columns each unless pair k is slot 0.
            const uint64_t ad64 = ptx::smem_desc(sbase + oSS, kSPitch * 16, 128);
            const uint64_t bd64 = ptx::smem_desc(sbase + oSB2, 48 * 16, 128);
            const uint32_t a_lo = (uint32_t)ad64, a_hi = (uint32_t)(ad64 >> 32);
            const uint32_t b_lo = (uint32_t)bd64, b_hi = (uint32_t)(bd64 >> 32);
            uint32_t ss = 0, sph = 0;  // staged pair slot and phase
            uint32_t as = 0, aph = 0;  // slot and phase of the next output pair to start
            uint32_t ws = kKA - 1;     // slot of the output pair that completes next
            // row r of the staged pair x weight blocks i .. (N / 16 of them) onto TMEM column dc
            auto taps = [&](uint32_t on, uint32_t al, int r, int i, uint32_t dc, uint32_t id) {
#pragma unroll
                for (int kx = 0; kx < 3; ++kx)
                    ptx::mma_bf16_if(on, dc, al + (uint32_t)((r * kSRowB) >> 4) + kx, a_hi,
                                     b_lo + (uint32_t)((kx * kB2Group) >> 4) + 16u * i, b_hi, id);
            };
            StCursor cur = st_begin(p);
            StItem it;
            while (st_next(p, cur, it)) {
                const int P = it.pairs;
                for (int k = 0; k <= P; ++k) {
                    ok = ok && wait_bar(&s_full[ss], sph, abort_flag, p.err, p.wait_ns);
                    if (k < P)  // output pair k starts here: its accumulators must have been drained
                        ok = ok && wait_bar(&l2_free[as], aph ^ 1, abort_flag, p.err, p.wait_ns);
                    ptx::tc_fence_after();
                    const uint32_t on = ok ? lead : 0u;
                    const uint32_t al = a_lo + ss * (uint32_t)((2 * kSRowB) >> 4);
                    const uint32_t dw = tbase + 32u * ws, da = tbase + 32u * as;
                    if (k > 0 && k < P && as != 0) {
                        taps(on, al, 0, 0, dw, id48);
                        taps(on, al, 1, 0, dw + 16u, id48);
                    } else {
                        if (k > 0) {
                            taps(on, al, 0, 0, dw, id32);
                            taps(on, al, 1, 0, dw + 16u, id16);
                        }
                        if (k < P) {
                            taps(on, al, 0, 2, da, id16);
                            taps(on, al, 1, 1, da, id32);
                        }
                    }
                    if (k > 0) {
                        ptx::mma_commit_if(lead, &l2_full[ws]);
                        if (++ws == kKA) ws = 0;
                    }
                    ptx::mma_commit_if(lead, &s_empty[ss]);
                    if (++ss == kNS) {
                        ss = 0;
                        sph ^= 1;
                    }
                    if (k == 0) ws = as;
                    if (k < P && ++as == kKA) {
                        as = 0;
                        aph ^= 1;
                    }
                }
            }
        }
        if (lane == 0) {
            uint64_t* f = fin + (warp == 0 ? 0 : 1);
            ptx::mma_commit(f);
            const uint64_t t0 = gtime();
            while (!ptx::mbar_test(f, 0)) {
                if (gtime() - t0 > p.wait_ns) {
                    *(volatile int*)p.err = MB_ERR_TIMEOUT;
                    break;
                }
            }
        }
        __syncwarp();
    } else if (warp == 1 || warp == 2) {
        // ================= layer-1 operand builder ====================================================
        // Operand k of an item belongs to the layer-1 rows r, r + 1, r = y0 + m0 - 1 + 2 k: pixel q holds
        // the input bytes of rows r - 1 .. r + 2 (elements 0..3 of K chunk 0) at column x0 + s0 - 2 + q,
        // both mirror-padded at the slice borders. Builder thread b (warps 1-2) owns pixels b, b + 64 and,
        // b < 2, b + 128; it keeps the four rows of a pair in registers and has the loads of the kLd
        // pairs after them in flight (rows further on are bulk-prefetched into L2). A loaded byte is
        // converted only when its row enters the window: converting it at the load would stall the
        // thread on the load. An integer up to 255 is exact in BF16 (the upper half of its FP32 bits).
        const int bt = tid - 32;
        const int nj = warp == 1 ? 3 : 2;
        uint32_t slot = 0, sph = 0;  // operand pair slot and its phase
        StCursor cur = st_begin(p);
        StItem it;
        while (st_next(p, cur, it)) {
            const int last = it.rows + 3;  // input rows 0 .. rows + 3 of the item
            const uint8_t* src = p.in + (int64_t)it.z * p.in_slice;
            const int c0 = p.x0 + it.s0 - 2;
            const int nin = min(130, it.ncol + 4);  // input columns the strip's outputs depend on
            const int rbase = p.y0 + it.m0 - 2;
            int col[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) col[i] = bt + 64 * i < nin ? refl(c0 + bt + 64 * i, p.w) : 0;
            // raw bytes; columns past the strip read column 0 (they feed only outputs that are not stored)
            auto load_row = [&](int i, uint32_t (&v)[3]) {
                const uint8_t* row = src + (int64_t)refl(rbase + min(i, last), p.h) * p.in_pitch;
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    if (j < nj) v[j] = (uint32_t)__ldg(row + col[j]);
            };
            auto conv = [&](uint32_t v) { return __float_as_uint((float)v); };  // raw byte -> FP32 bits
            constexpr int kPf = 8;  // input rows prefetched at a time, by one thread each
            auto prefetch_row = [&](int i) {
                if (i > last) return;
                const uint8_t* base = src + (int64_t)refl(rbase + i, p.h) * p.in_pitch;
                const uintptr_t lo = (uintptr_t)(base + max(0, c0)) & ~(uintptr_t)15;
                const uintptr_t hi = (uintptr_t)(base + min(p.w, c0 + nin)) & ~(uintptr_t)15;
                if (hi > lo) ptx::prefetch_l2_bulk((const void*)lo, (uint32_t)(hi - lo));
            };
            if (bt < 2 * kPf) prefetch_row(4 + bt);
            constexpr int kLd = 2;  // row pairs whose loads are in flight
            uint32_t f0[3], f1[3], f2[3], f3[3], pend[kLd][2][3];
            load_row(0, f0);
            load_row(1, f1);
            load_row(2, f2);
            load_row(3, f3);
#pragma unroll
            for (int t = 0; t < kLd; ++t) {  // rows past the last are clamped to it
                load_row(4 + 2 * t, pend[t][0]);
                load_row(5 + 2 * t, pend[t][1]);
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                f0[j] = conv(f0[j]);
                f1[j] = conv(f1[j]);
                f2[j] = conv(f2[j]);
                f3[j] = conv(f3[j]);
            }
            for (int k0 = 0; k0 <= it.pairs; k0 += kLd) {
#pragma unroll
                for (int t = 0; t < kLd; ++t) {
                    const int k = k0 + t;
                    if (k > it.pairs) break;
                    if (k > 0 && 2 * k % kPf == 0 && bt < kPf) prefetch_row(2 * k + 4 + kPf + bt);
                    wait_bar(&a1_empty[slot], sph ^ 1, abort_flag, p.err, p.wait_ns);
                    uint8_t* dst = smem + oSA1 + slot * kSRowB + bt * 16;
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        if (j < 2 || bt < 2)
                            *reinterpret_cast<uint2*>(dst + 1024 * j) =
                                make_uint2(__byte_perm(f0[j], f1[j], 0x7632), __byte_perm(f2[j], f3[j], 0x7632));
                    }
                    ptx::fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0 && !p.fault_stall) ptx::mbar_arrive(&a1_full[slot]);
                    if (++slot == kNA1) {
                        slot = 0;
                        sph ^= 1;
                    }
                    // the next pair's window; the loads of the pair kLd further take these rows' place
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        if (j < nj) {
                            f0[j] = f2[j];
                            f1[j] = f3[j];
                            f2[j] = conv(pend[t][0][j]);
                            f3[j] = conv(pend[t][1][j]);
                        }
                    load_row(2 * k + 4 + 2 * kLd, pend[t][0]);
                    load_row(2 * k + 5 + 2 * kLd, pend[t][1]);
                }
            }
        }
    } else if (warp >= 4 && warp < 8) {
        // ================= layer-1 epilogue: x 1/255, bias, ReLU, BF16 -> staged feature ring =======
        const int px = tid - 128;
        const uint32_t lanes = (uint32_t)(32 * (warp - 4)) << 16;
        const float2 inv = make_float2(cst[kCInv], cst[kCInv]);
        float2 b1r[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) b1r[c] = make_float2(cst[kCB1 + 2 * c], cst[kCB1 + 2 * c + 1]);
        uint32_t sl = 0, lph = 0, ss = 0, sph = 0;  // accumulator and staged pair slots, their phases
        StCursor cur = st_begin(p);
        StItem it;
        while (st_next(p, cur, it)) {
            for (int k = 0; k <= it.pairs; ++k) {
                wait_bar(&l1_full[sl], lph, abort_flag, p.err, p.wait_ns);
                ptx::tc_fence_after();
                float d[32];
                ptx::tmem_ld32(tbase + lanes + kL1Col + 32u * sl, d);
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&l1_free[sl]);
                if (++sl == kKL) {
                    sl = 0;
                    lph ^= 1;
                }
                uint32_t wd[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const float2 v = __ffma2_rn(make_float2(d[2 * c], d[2 * c + 1]), inv, b1r[c % 8]);
                    wd[c] = relu2(pack_bf16x2(v.x, v.y));
                }
                wait_bar(&s_empty[ss], sph ^ 1, abort_flag, p.err, p.wait_ns);
                uint8_t* dst = smem + oSS + ss * 2 * kSRowB + px * 16;
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    *reinterpret_cast<uint4*>(dst + r * kSRowB) =
                        make_uint4(wd[8 * r], wd[8 * r + 1], wd[8 * r + 2], wd[8 * r + 3]);
                    *reinterpret_cast<uint4*>(dst + r * kSRowB + kSPitch * 16) =
                        make_uint4(wd[8 * r + 4], wd[8 * r + 5], wd[8 * r + 6], wd[8 * r + 7]);
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&s_full[ss]);
                if (++ss == kNS) {
                    ss = 0;
                    sph ^= 1;
                }
            }
        }
    } else if (warp >= 8) {
        // ================= layer-2 epilogue: bias, ReLU, head, sigmoid, store ========================
        const int px = tid - 256;  // TMEM lane = output pixel of the strip
        const uint32_t lanes = (uint32_t)(32 * (warp - 8)) << 16;
        uint32_t sl = 0, aph = 0;  // accumulator pair slot and its phase
        // the head's constants in registers (shared-memory reads would repeat every row: the waits
        // are compiler barriers)
        float2 b2r[8];
        float whr[16];
#pragma unroll
        for (int c = 0; c < 8; ++c) b2r[c] = make_float2(cst[kCB2 + 2 * c], cst[kCB2 + 2 * c + 1]);
#pragma unroll
        for (int c = 0; c < 16; ++c) whr[c] = cst[kCWH + c];
        const float bhr = cst[kCBH];
        StCursor cur = st_begin(p);
        StItem it;
        while (st_next(p, cur, it)) {
            const bool col = px < it.ncol;
            int64_t idx = (int64_t)it.z * p.out_slice + (int64_t)it.m0 * p.out_pitch + it.s0 + px;
            for (int k = 0; k < it.pairs; ++k, idx += 2 * p.out_pitch) {
                wait_bar(&l2_full[sl], aph, abort_flag, p.err, p.wait_ns);
                const bool live = !*abort_flag;  // read early: its latency overlaps the drain
                ptx::tc_fence_after();
                float d[32];
                const uint32_t ta = tbase + lanes + 32u * sl;
                ptx::tmem_ld32(ta, d);
                ptx::tmem_st32_zero(ta);
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&l2_free[sl]);
                if (++sl == kKA) {
                    sl = 0;
                    aph ^= 1;
                }
                float2 z = make_float2(bhr, bhr);  // the pair's two rows
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float2 u = __fadd2_rn(make_float2(d[2 * c], d[2 * c + 1]), b2r[c]);
                    const float2 v = __fadd2_rn(make_float2(d[16 + 2 * c], d[17 + 2 * c]), b2r[c]);
                    z = __ffma2_rn(make_float2(whr[2 * c], whr[2 * c]), make_float2(fmaxf(u.x, 0.f), fmaxf(v.x, 0.f)), z);
                    z = __ffma2_rn(make_float2(whr[2 * c + 1], whr[2 * c + 1]),
                                   make_float2(fmaxf(u.y, 0.f), fmaxf(v.y, 0.f)), z);
                }
                // the correctly rounded reciprocal is the correctly rounded quotient 1 / x
                const float p0 = __frcp_rn(1.0f + expf(-z.x)), p1 = __frcp_rn(1.0f + expf(-z.y));
                if (col && live) {
                    const bool two = 2 * k + 1 < it.rows;
                    if (p.out_u8) {
                        uint8_t* o = static_cast<uint8_t*>(p.out) + idx;
                        o[0] = (uint8_t)fminf(floorf(255.0f * p0 + 0.5f), 255.0f);
                        if (two) o[p.out_pitch] = (uint8_t)fminf(floorf(255.0f * p1 + 0.5f), 255.0f);
                    } else {
                        float* o = static_cast<float*>(p.out) + idx;
                        o[0] = p0;
                        if (two) o[p.out_pitch] = p1;
                    }
                }
            }
        }
    }

    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == 0) ptx::tmem_dealloc(tbase, kSTmem);
}

// Operands and constants from the forward-layout parameters (W1t[tap][co], b1, W2t[ci][tap][co], b2,
// wh, bh; tap = 3 ky + kx):
//   B1, per column tap kx: [chunk][n][8] BF16, n = 16 r + co, element k holding W1[co][k - r][kx]
//   B2, per column tap kx: [chunk][n][8] BF16, n = 16 i + co, element ci holding W2[co][ci][2 - i][kx]
//   constants: b1, b2, head weights, head bias, 1/255
__global__ void __launch_bounds__(1024) st_tc_pack(const float* fwd, uint8_t* wpack) {
    ptx::grid_dep_launch();
    __nv_bfloat16* b1 = reinterpret_cast<__nv_bfloat16*>(wpack);
    for (int i = threadIdx.x; i < kB1 / 2; i += blockDim.x) {
        const int kx = i / 512, rem = i % 512, n = (rem / 8) % 32, co = n % 16;
        const int ky = (rem / 256) * 8 + rem % 8 - n / 16;
        b1[i] = __float2bfloat16_rn(ky >= 0 && ky < 3 ? fwd[kFW1 + (ky * 3 + kx) * 16 + co] : 0.f);
    }
    __nv_bfloat16* b2 = reinterpret_cast<__nv_bfloat16*>(wpack + kB1);
    for (int i = threadIdx.x; i < kB2 / 2; i += blockDim.x) {
        const int kx = i / 768, rem = i % 768, ci = (rem / 384) * 8 + rem % 8, n = (rem / 8) % 48;
        const int ky = 2 - n / 16, co = n % 16;
        b2[i] = __float2bfloat16_rn(fwd[kFW2 + (ci * 9 + ky * 3 + kx) * 16 + co]);
    }
    float* c = reinterpret_cast<float*>(wpack + kB1 + kB2);
    for (int i = threadIdx.x; i < kSConst; i += blockDim.x) {
        float v = 0.f;
        if (i < 16) v = fwd[kFB1 + i];
        else if (i < 32) v = fwd[kFB2 + (i - 16)];
        else if (i < 48) v = fwd[kFWH + (i - 32)];
        else if (i == kCBH) v = fwd[kFBH];
        else if (i == kCInv) v = 1.0f / 255.0f;
        c[i] = v;
    }
}

struct StTcState {
    uint8_t* d_wpack = nullptr;
    int* h_err = nullptr;
    int* d_err = nullptr;
    int n_sms = 0;
};

}  // namespace

void st_tc_release(mb_net* net) {
    StTcState* S = reinterpret_cast<StTcState*>(net->st_state);
    if (!S) return;
    dev_free(S->d_wpack);
    if (S->h_err) cudaFreeHost(S->h_err);
    delete S;
    net->st_state = nullptr;
}

mb_status st_tc_poll_error(mb_net* net) {
    StTcState* S = reinterpret_cast<StTcState*>(net->st_state);
    if (S && S->h_err && *(volatile int*)S->h_err) {
        *(volatile int*)S->h_err = 0;
        set_error("a student tensor-core launch gave up waiting (device-side wait limit)");
        return MB_ERR_TIMEOUT;
    }
    return MB_OK;
}

mb_status st_tc_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w, int64_t in_pitch,
                       int64_t in_slice, int64_t y0, int64_t x0, int64_t rows, int64_t cols, void* out,
                       int64_t out_pitch, int64_t out_slice, mb_out_type ot, cudaStream_t st) {
    if (z == 0 || rows == 0 || cols == 0) return MB_OK;
    StTcState* S = reinterpret_cast<StTcState*>(net->st_state);
    if (!S) {
        S = new (std::nothrow) StTcState();
        if (!S) {
            set_error("host allocation failed");
            return MB_ERR_OOM;
        }
        net->st_state = S;
    }
    if (!S->d_wpack) MB_TRY(dev_alloc((void**)&S->d_wpack, kWpack));
    if (!S->h_err) {
        if (fault_oom()) {
            set_error("pinned allocation failed (MB_FAULT_OOM injected)");
            return MB_ERR_OOM;
        }
        MB_CUDA(cudaHostAlloc((void**)&S->h_err, sizeof(int), cudaHostAllocMapped));
        *S->h_err = 0;
        MB_CUDA(cudaHostGetDevicePointer((void**)&S->d_err, S->h_err, 0));
    }
    MB_TRY(st_tc_poll_error(net));
    if (!S->n_sms) {
        int dev = 0;
        MB_CUDA(cudaGetDevice(&dev));
        MB_CUDA(cudaDeviceGetAttribute(&S->n_sms, cudaDevAttrMultiProcessorCount, dev));
    }
    static std::atomic<uint64_t> smem_set{0};
    MB_TRY(set_smem_once(smem_set, st_tc_infer, kSSmem));
    // the forward copy changes while the student trains: pack it on every call
    // (the inference launch sets itself up meanwhile: 64 x 64 17.2 -> 12.9 us, 1024 x 1024 27.4 -> 23.7)
    st_tc_pack<<<1, 1024, 0, st>>>(net->d_simt, S->d_wpack);
    count_launch();
    MB_CUDA(cudaGetLastError());
    StTcParams p{};
    p.in = in;
    p.out = out;
    p.wpack = S->d_wpack;
    p.err = S->d_err;
    p.in_slice = in_slice;
    p.in_pitch = in_pitch;
    p.out_slice = out_slice;
    p.out_pitch = out_pitch;
    p.h = (int)h;
    p.w = (int)w;
    p.y0 = (int)y0;
    p.x0 = (int)x0;
    p.rows = (int)rows;
    p.cols = (int)cols;
    p.out_u8 = ot == MB_OUT_U8 ? 1 : 0;
    p.n_strips = (int)((cols + kSW - 1) / kSW);
    const int64_t slots = (int64_t)S->n_sms * 2;
    p.col_pairs = (int)((rows + 1) / 2);
    p.total_pairs = z * p.n_strips * p.col_pairs;
    const char* stall = getenv("MB_FAULT_STALL");
    p.fault_stall = (stall && stall[0] == '1') ? 1 : 0;
    p.wait_ns = p.fault_stall ? 200000000ull : kSWaitNs;
    // one range per CTA slot, or fewer when a range would get under 4 row pairs
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(slots, (p.total_pairs + 3) / 4));
    MB_CUDA(launch_dependent(st_tc_infer, (unsigned)grid, kSThreads, kSSmem, st, p));
    count_launch();
    return MB_OK;
}

}  // namespace mb
