// student_x3.h - the student's parameter layout and the interface of its tensor-core training pass.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace mb {

// Parameter offsets (API layout): W1[16][1][3][3] b1[16] W2[16][16][3][3] b2[16] Wh[16] bh.
constexpr int kSW1 = 0, kSB1 = 144, kSW2 = 160, kSB2 = 2464, kSWH = 2480, kSBH = 2496, kSN = 2497;
// Forward (SIMT) layout: W1t[1][3][3][16] b1 | W2t[16][3][3][16] b2 | Wh bh  (same block offsets)

// Fixed grids make the partial sums reproducible: one CTA per SM of a GB300, two for st_grad2.
constexpr int kX3Grid = 152, kX3GridG2 = 304;
constexpr int kX3FwdWidth = 34;                      // partials per CTA: [loss, db2[16], dWh[16], dbh]
constexpr int kX3StudentPack = 3 * 2 * 144 * 16;     // bytes of one pass's B operand

// One gradient of a batch: partial sums, then loss and gradient. part_g2: 2304 per CTA; part_bwd: dW1[144],
// db1[16] per CTA.
struct StudentX3 {
    const uint8_t* in;       // [slices][H][W]
    const float* target;     // [slices][H][W]
    const int* zmap;         // slice of each batch entry (NULL: identity)
    int B, H, W;
    const float* fw;         // forward parameters, SIMT layout
    float* h1;               // [B][H+2][W+2][16]
    uint16_t* mask;          // [B][H+2][W+2]
    float* dy2;              // [B][H][W][16]
    const uint8_t* pack;     // B operands of both passes (2 x kX3StudentPack, see student_pack)
    float *part_fwd, *part_g2, *part_bwd;
    float inv_n;
    float* grad;             // [kSN], and the mean loss
    float* loss;
    int* err;                // device address of the error word
};
mb_status student_x3_grad(const StudentX3& a, cudaStream_t st);

// One chunk of slices of an inference call (out_pitch, out_slice in elements).
struct StudentX3Region {
    const uint8_t* in;
    int64_t in_slice, in_pitch, out_pitch, out_slice;
    int z, h, w, y0, x0, rows, cols;
    const float* fw;
    float* h1;               // [z][rows + 2][cols + 2][16]
    void* out;
    int out_u8, first;       // first: the call's first chunk
    int* err;
};
mb_status student_x3_infer(const StudentX3Region& a, cudaStream_t st);

}  // namespace mb
