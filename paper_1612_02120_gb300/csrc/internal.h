// internal.h - host-side internals shared by the translation units of libmembrane.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <string>
#include <vector>

#include "../../include/membrane.h"
#include "per_device.h"

namespace mb {

enum Family { FAMILY_TEACHER = 1, FAMILY_STUDENT = 2, FAMILY_FASTMEMB = 3, FAMILY_FASTMEMB_3NM = 4, FAMILY_MASKEXTEND = 5 };

// Teacher geometry: conv5x5 x3 with two 2x2 max-filters -> receptive radius 7.
constexpr int kTeacherRadius = 7;
constexpr int kTeacherC = 32;
// Student geometry: conv3x3 x2 -> radius 2.
constexpr int kStudentRadius = 2;
constexpr int kStudentC = 16;
// FastMemb dense form: conv4x4 (dilation 1, 2, 4) with max-out 2, max-filters (1, 2, 4), conv4x4
// dilation 8 -> radius 26 (53x53 field of view).
constexpr int kFastMembRadius = 26;
// FastMemb_3nm: one more stage (dilation 8 conv and max-filter, head at 16) -> radius 54 (109x109).
constexpr int kFastMemb3nmRadius = 54;
inline bool is_fastmemb(int family) { return family == FAMILY_FASTMEMB || family == FAMILY_FASTMEMB_3NM; }
// convolutions of a FastMemb family (conv1, the 32->64 middle convs, the head)
inline int fastmemb_convs(int family) { return family == FAMILY_FASTMEMB_3NM ? 5 : 4; }

void set_error(const char* fmt, ...);
void clear_error();
mb_status cuda_fail(cudaError_t e, const char* what, const char* file, int line);
void count_launch(int n = 1);

// u / 255, correctly rounded. A zero numerator takes the division's slow path, and a whole warp with it, so
// zero is divided as one and set back: FP32's 0 / 255 is 0.
__device__ __forceinline__ float unit_of_byte(uint32_t u) {
    const float q = (float)(u > 1u ? u : 1u) / 255.0f;
    return u ? q : 0.f;
}

// A launch that may begin while the one before it on the stream still ends (programmatic dependent
// launch): the kernel calls ptx::grid_dep_wait before it touches anything that an earlier launch
// writes or reads, and the one before it calls ptx::grid_dep_launch where this one may set itself up.
// What an earlier launch of the chain writes is read by ordinary loads (or bulk copies), not through the
// read-only path: __ldg may be moved above the wait. A call's first launch is an ordinary one, so that a
// chain does not begin while what an earlier call writes (this one's inputs) is still being written.
// A call's launches in a chain, against ordinary ones:
// FastMemb BF16 on 64 x 64 55 -> 47 us, 1024 x 1024 283 -> 267, eight of them 1,839 -> 1,828; FP32
// teacher 64 x 64 58 -> 52, 1024 x 1024 441 -> 430; a student gradient of 3 x 131 x 257 95 -> 91.
// After a launch that does not call it, this is an ordinary one.
template <typename... K, typename... A>
cudaError_t launch_dependent(void (*kernel)(K...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st,
                             const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<K>(args)...);
}
bool fault_oom();

#define MB_CUDA(call)                                                        \
    do {                                                                     \
        cudaError_t e_ = (call);                                             \
        if (e_ != cudaSuccess) return ::mb::cuda_fail(e_, #call, __FILE__, __LINE__); \
    } while (0)

#define MB_TRY(call)                      \
    do {                                  \
        mb_status s_ = (call);            \
        if (s_ != MB_OK) return s_;       \
    } while (0)

mb_status dev_alloc(void** p, size_t bytes);
void dev_free(void* p);

// Lets `kernel` use `bytes` of dynamic shared memory on the current device.
template <typename... K>
mb_status set_smem_once(std::atomic<uint64_t>& done, void (*kernel)(K...), int bytes) {
    int device = 0;
    MB_CUDA(cudaGetDevice(&device));
    return once_per_device(done, device, [&]() -> mb_status {
        MB_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
        return MB_OK;
    });
}

// A growable device scratch buffer owned by a net.
struct Workspace {
    void* ptr = nullptr;
    size_t bytes = 0;
    mb_status ensure(size_t need);
    void release();
};

struct GraphCacheEntry;

// Which weights a launch took along as kernel parameters. Parameters are fixed when a launch is captured in
// a caller's CUDA graph, while device weights follow mb_load_weights: a kernel whose `taken` is no longer
// the net's count (*word) reads its weights from device memory instead.
struct WeightsTag {
    const uint32_t* word;
    uint32_t taken;
};
}  // namespace mb

struct mb_net {
    int device = 0;
    int family = 0;
    mb_precision prec = MB_PREC_FP32;
    std::vector<mb_layer_desc> layers;
    int64_t n_params = 0;
    std::vector<float> host_params;  // FP32 master copy on the host
    bool loaded = false;
    bool calibrated = false;
    float* d_params = nullptr;   // FP32 parameters, API layout (student: the master copy)
    float* d_simt = nullptr;     // SIMT layout: per conv layer Wt[ci][ky][kx][co], b[co]; head w, b
    uint32_t tag = 0;            // counts the changes of the weights (and FP8 scales)
    uint32_t* d_tag = nullptr;   // the same on the device (WeightsTag)
    size_t simt_floats = 0;
    void* tc_state = nullptr;    // tensor-core path state (packed operands, constants), tc_conv.cu
    void* fm_state = nullptr;    // FastMemb tensor-core state (packed operands, error word), fastmemb_tc.cu
    void* me_state = nullptr;    // MaskExtend tensor-core state (packed operands, error word), maskextend_tc.cu
    void* x3_state = nullptr;    // FP32 tensor-core layers (packed split operands, error word), f32_tc.cu
    bool x3_ok = false;          // its activations are bounded: those layers run on the tensor cores
    // mapped host words of the FP32-accurate student passes: error word of the training, loss of the last
    // gradient, error word of the inference
    int* train_host = nullptr;
    int* train_dev = nullptr;    // their device address
    void* st_state = nullptr;    // student tensor-core state (packed operands, error word), student_tc.cu
    float fp8_amax[2][32] = {};
    mb::Workspace ws;            // layered FP32 path activations
    mb::Workspace ws2;           // student training / cascade scratch
    mb::Workspace slab_ws;       // host-buffer streaming: double-buffered device slabs
    cudaStream_t slab_streams[4] = {};  // H2D, compute, D2H, second compute stream (overlapping slabs)
    int host_io = 0;             // mb_host_io: 0 direct host access where possible, 1 always slabs
    cudaEvent_t slab_events[6] = {};                              // per buffer: in, comp, out
    // persistent kernel tuning
    // (defaults: the even split with rings of 4, what the autotuner picks on most shapes; against
    // round-robin items of 64 rows and rings of 6, BF16: 32 x 1024 x 1024 3,510 -> 3,130 us,
    // 8 x 1000 x 1333 1,251 -> 1,055 us. FP8 launches are always even; FP8 nets start with rings of 6,
    // 2,902 us against 3,132 with 4)
    int rows_per_item = 0;
    int stages = 4;  // teacher A-ring depth (a compiled candidate; set by the autotuner or mb_set_tuning)
    bool tuned = false;
    // batch graph cache
    std::vector<mb::GraphCacheEntry*> graphs;
};

namespace mb {

// SIMT (FP32 arithmetic) layered path: conv kernels with activations in a workspace.
mb_status simt_teacher_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w,
                              int64_t in_pitch, int64_t in_slice, int64_t y0, int64_t x0, int64_t rows,
                              int64_t cols, void* out, int64_t out_pitch, int64_t out_slice,
                              mb_out_type ot, cudaStream_t st);
// Slices per pass of a workspace of per_slice bytes each (3 GB at most, at least one slice).
int64_t chunk_slices(size_t per_slice, int64_t z);
// FP32 student inference: on the tensor cores in exact three-part splits where the weights are bounded
// (student.cu, student_x3.cu), else simt_student_region.
mb_status student_f32_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w, int64_t in_pitch,
                             int64_t in_slice, int64_t y0, int64_t x0, int64_t rows, int64_t cols, void* out,
                             int64_t out_pitch, int64_t out_slice, mb_out_type ot, cudaStream_t st);
mb_status simt_student_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w,
                              int64_t in_pitch, int64_t in_slice, int64_t y0, int64_t x0, int64_t rows,
                              int64_t cols, void* out, int64_t out_pitch, int64_t out_slice,
                              mb_out_type ot, cudaStream_t st);
// FastMemb region (FP32 / BF16); sub = 1: the dense map, sub = 2: the map at even rows and columns
// of the region (out is ceil(rows/2) x ceil(cols/2)).
mb_status simt_fastmemb_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w,
                               int64_t in_pitch, int64_t in_slice, int64_t y0, int64_t x0, int64_t rows,
                               int64_t cols, void* out, int64_t out_pitch, int64_t out_slice,
                               mb_out_type ot, cudaStream_t st, int sub);
mb_status tc_fastmemb_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w,
                             int64_t in_pitch, int64_t in_slice, int64_t y0, int64_t x0, int64_t rows,
                             int64_t cols, void* out, int64_t out_pitch, int64_t out_slice,
                             mb_out_type ot, cudaStream_t st, int sub);
// FastMemb tensor-core layers (fastmemb_tc.cu): pack the B operands of the 32->64 convs and the
// head (split BF16, or FP16 for FP16 nets), launch one (the head ends with the softmax, FP32 or
// uint8 out), poll the device-side wait error word.
mb_status fm_tc_prepare(mb_net* net);
void fm_tc_release(mb_net* net);
mb_status fm_tc_poll_error(mb_net* net);
// in, and a layer's out: 16-bit features of the net's type, max-filtered, chunk-planar
// [slice][row][chunk 0..3][column (pitch)][8 channels]. rows x cols: what the layer writes (filtered
// features; the head: the map, FP32 or uint8), i.e. it reads rows + 3d (+ d for a layer) input rows.
// in_pitch is at least fm_tc_in_pitch of the same cols and d (the last strip's overrun).
// layer: 0-based index of the conv after conv1; the last one is the head.
int64_t fm_tc_in_pitch(bool head, int64_t cols, int d);
mb_status fm_tc_layer(mb_net* net, int layer, const void* in, int64_t in_slice, int64_t in_pitch, void* out,
                      int64_t out_slice, int64_t out_pitch, int rows, int cols, int d, int nz, int out_u8,
                      cudaStream_t st);
// MaskExtend (maskextend.cu): SIMT weight layout, and the +z transfer recursion (device pointers).
void me_pack(const mb_net* net, const float* params, std::vector<float>& out);
// MaskExtend FP16 tensor-core convs (maskextend_tc.cu). layer 0..4; in, and the out of layers 0-3: FP16
// features, max-filtered, chunk-planar [row][chunk of 8 channels][column (pitch)][8] (2, 4, 5, 6, 7 chunks
// into layers 0..4); rows x cols is what the layer writes (layer 4: the 3 class probabilities
// [3][rows][out_pitch], planes probs_plane apart), i.e. it reads rows + 3 d (+ d for layers 0-3) rows.
// in_pitch is at least me_tc_in_pitch of the layer and cols (the last strip's overrun).
int64_t me_tc_in_pitch(int layer, int64_t cols);
mb_status me_tc_prepare(mb_net* net);
void me_tc_release(mb_net* net);
mb_status me_tc_poll_error(mb_net* net);
mb_status me_tc_layer(mb_net* net, int layer, const void* in, int64_t in_pitch, void* out, int64_t out_pitch, int rows,
                      int cols, float* probs, int64_t probs_plane, cudaStream_t st);
mb_status maskextend_run(mb_net* net, const uint8_t* em, const float* memb, int64_t zt, int64_t h, int64_t w,
                         const uint8_t* seeds, int64_t z0, int64_t n_steps, int dz, float thr, uint8_t* masks_out,
                         float* probs_out, cudaStream_t st);
// BF16 student inference on the tensor cores (student_tc.cu), same arguments as simt_student_region;
// student_region picks it for BF16 nets and the CUDA-core path for FP32 nets.
mb_status st_tc_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w, int64_t in_pitch,
                       int64_t in_slice, int64_t y0, int64_t x0, int64_t rows, int64_t cols, void* out,
                       int64_t out_pitch, int64_t out_slice, mb_out_type ot, cudaStream_t st);
void st_tc_release(mb_net* net);
mb_status st_tc_poll_error(mb_net* net);
mb_status student_f32_poll_error(mb_net* net);  // the FP32 student's inference
// MB_ERR_TIMEOUT (and every error word of the net cleared) if a launch of an inference on this net gave up
// waiting: what a call that has synchronised returns, so that MB_OK means complete maps.
mb_status net_poll_error(mb_net* net);
mb_status student_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w, int64_t in_pitch,
                         int64_t in_slice, int64_t y0, int64_t x0, int64_t rows, int64_t cols, void* out,
                         int64_t out_pitch, int64_t out_slice, mb_out_type ot, cudaStream_t st);
// FP32 layers on the tensor cores (f32_tc.cu): 5x5 32 -> 32 of the teacher (layer 0: ReLU, FP32 out;
// layer 1: ReLU, head, sigmoid, FP32 or uint8 map out), 4x4 32 -> 64 with max-out of FastMemb (layer =
// 0-based conv after conv1). in and feature outputs: FP32 [slice][row][column (pitch)][32]; the conv
// reads input (r, c) = 2x2 max (dilation dm; 0: none) at source (stride r, stride c), r < in_rows,
// c < in_cols. x3_prepare packs at load time and sets net->x3_ok; where it is false the CUDA-core
// kernels run.
struct X3Layer {
    const float* in;
    int64_t in_slice, in_pitch;
    int in_rows, in_cols;
    int64_t src_cols;
    int d, dm, stride;
    void* out;
    int64_t out_slice, out_pitch;
    int out_h, out_w, nz, out_u8;
};
mb_status x3_prepare(mb_net* net);
void x3_release(mb_net* net);
mb_status x3_poll_error(mb_net* net);
mb_status x3_layer(const mb_net* net, int layer, const X3Layer& a, cudaStream_t st);
// Layers 2 and 3 of the FP32 teacher for nz slices: act1 [nz][rows + 10][cols + 10][32] -> act2
// [nz][rows + 5][cols + 5][32] -> the map; on the tensor cores, or (x3_ok false) on CUDA cores.
mb_status teacher_fp32_deep(const mb_net* net, const float* act1, float* act2, int nz, int64_t rows, int64_t cols,
                            void* out, int64_t out_pitch, int64_t out_slice, mb_out_type ot, cudaStream_t st);
// FP32 teacher activations after the two max-filters: per-channel amax over n slices (device out[64]).
mb_status simt_teacher_amax(mb_net* net, const uint8_t* in, int64_t n, int64_t h, int64_t w, float* d_amax,
                            cudaStream_t st);
// Pack the SIMT weight layout from the FP32 API layout (host side).
void simt_pack(const mb_net* net, const float* params, std::vector<float>& out);

// Tensor-core fused path.
mb_status tc_prepare(mb_net* net);   // pack BF16 / FP8 weights from host_params (+ calibration)
void tc_release(mb_net* net);
mb_status tc_poll_error(mb_net* net);  // MB_ERR_TIMEOUT if a launch recorded a timed-out wait
mb_status tc_infer_blocks(mb_net* net, const mb_block* blocks, int n_blocks, const int64_t* y0,
                          const int64_t* x0, const int64_t* rows, const int64_t* cols, mb_out_type ot,
                          cudaStream_t st, bool use_graph);
// Autotuner timed on the caller's own batch (its outputs are written by every candidate).
mb_status tc_autotune_batch(mb_net* net, const mb_block* blocks, int n_blocks, mb_out_type ot, const char* cache_path,
                            int32_t* choice, cudaStream_t st);

// Student training and cascade.
mb_status student_loss_grad(mb_net* s, const uint8_t* in, const float* tgt, int64_t n, int64_t h, int64_t w,
                            double* loss, float* grad, cudaStream_t st);
mb_status student_train(mb_net* s, const uint8_t* in, const float* tgt, int64_t n, int64_t h, int64_t w,
                        const mb_train_cfg* cfg, const char* ckpt, float* curve, cudaStream_t st);
mb_status cascade(mb_net* s, mb_net* t, const uint8_t* in, int64_t z, int64_t h, int64_t w, float* out,
                  int tile, float lo, float hi, float max_frac, double* rate, uint8_t* flags,
                  cudaStream_t st);

// Teacher dispatch used by the API, the batch comparison path and the cascade.
mb_status teacher_region(mb_net* net, const uint8_t* in, int64_t z, int64_t h, int64_t w, int64_t in_pitch,
                         int64_t in_slice, int64_t y0, int64_t x0, int64_t rows, int64_t cols, void* out,
                         int64_t out_pitch, int64_t out_slice, mb_out_type ot, cudaStream_t st);

}  // namespace mb
