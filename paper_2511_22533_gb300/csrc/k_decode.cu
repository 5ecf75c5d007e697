// k_decode.cu -- K10: the convolutional stand-in grid decoder O(S) of Eq. 1
// (Sec. 4.1) and the dynamic-voxel count at the anchor step (Sec. 4.2).
//
// TRELLIS's decoder is not part of the paper; this one has the shape of an
// upsampling 3-D convolution stack: 3x3x3 convolutions with zero padding and
// ReLU, C -> 16 at D^3, nearest 2x upsampling, 16 -> 8 at (2D)^3, 2x, 8 -> 1
// at (4D)^3; sub-voxel v is occupied iff its logit > 0.  Every output is
// summed in one fixed fp32 order (bias, then tap k = 0..26 with dx fastest,
// then input channel; one rounding per * and +; taps outside the grid
// skipped), so the occupancy bits are reproducible bit for bit.  The decoder
// runs twice per sample (before and after the anchor step).
//
// What bounds it is fp32 arithmetic: 2 * 1.47e9 separate products and sums for
// eight 16^3 samples, 75 us at 128 lanes per SM (each * and + rounds, so no
// fused multiply-add and no tensor core).  Every thread holds pairs of outputs
// that take the same weight or the same input and uses paired instructions;
// nearest upsampling makes the outputs of one source cell share their inputs,
// so a thread computes the two (hidden layer) or four (last layer) of a cell,
// with channel-last activations read 16 bytes at a time.  One decode of eight
// 16^3 samples: 517 us with one output voxel per thread and channel-major
// activations, 154 us now (one sample: 108 -> 37 us).  The hidden layers run at
// 200 registers and two blocks per SM: with 128 (four blocks) the three source
// voxels spill, and the decode took 224 us against 141 (before each product was
// made to round on its own, see fmul2_alone).
#include "common.cuh"
#include "kernels.h"

namespace f3dc {

namespace {

constexpr int kDecThreads = 128;

template <int C>
F3DC_DEV void load_voxel(const float *p, float (&v)[C])
{
#pragma unroll
    for (int q = 0; q < C / 4; ++q) {
        const float4 f = __ldg(reinterpret_cast<const float4 *>(p) + q);
        v[4 * q] = f.x;
        v[4 * q + 1] = f.y;
        v[4 * q + 2] = f.z;
        v[4 * q + 3] = f.w;
    }
}

// out[b][v][co] (v on the (din UP)^3 grid) from in[b][u][ci] (u on din^3), both
// channel-last.  A thread computes 8 of the output channels (four pairs) of the
// UP voxels along x that share source column sx.
template <int CIN, int COUT, int UP>
__global__ void __launch_bounds__(kDecThreads, 2) k_conv3d(const float *in, int din, const uint16_t *w,
                                                       const uint16_t *bias, float *out, int B, float neg_zero)
{
    constexpr int G = COUT / 8;
    // [tap][ci][co], taps 16 bytes further apart: a warp fills consecutive taps
    __shared__ float4 sw[27][CIN * COUT / 4 + 1];
    __shared__ float sb[COUT];
#pragma unroll 9
    for (int q = threadIdx.x; q < COUT * CIN * 27; q += kDecThreads) {
        const int co = q / (CIN * 27), ci = (q / 27) % CIN, k = q % 27;
        reinterpret_cast<float *>(&sw[k][ci * (COUT / 4)])[co] = bf16_bits_to_f32(w[q]);
    }
    for (int q = threadIdx.x; q < COUT; q += kDecThreads) sb[q] = bf16_bits_to_f32(bias[q]);
    __syncthreads();
    griddep_launch();
    griddep_wait();
    const int d = din * UP;
    const size_t total = (size_t)B * d * d * din * G;
    const size_t q = (size_t)blockIdx.x * kDecThreads + threadIdx.x;
    if (q >= total) return;
    const int sx = (int)(q % din);
    size_t r = q / din;
    const int g = (int)(r % G);
    r /= G;
    const int y = (int)(r % d), z = (int)((r / d) % d), b = (int)(r / ((size_t)d * d));
    const float *ib = in + (size_t)b * din * din * din * CIN;
    const bool lo = sx > 0, hi = sx < din - 1;  // the neighbouring columns exist
    f32x2 acc[UP][4];
#pragma unroll
    for (int i = 0; i < UP; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[i][c] = {sb[8 * g + 2 * c], sb[8 * g + 2 * c + 1]};
#pragma unroll 1
    for (int kzy = 0; kzy < 9; ++kzy) {
        const int zz = z + kzy / 3 - 1, yy = y + kzy % 3 - 1;
        if (zz < 0 || zz >= d || yy < 0 || yy >= d) continue;
        const float *row = ib + ((size_t)(zz / UP) * din + yy / UP) * din * CIN;
        float s[3][CIN];  // columns sx - 1, sx, sx + 1 (the middle one where there is none)
        load_voxel<CIN>(row + (size_t)(lo ? sx - 1 : sx) * CIN, s[0]);
        load_voxel<CIN>(row + (size_t)sx * CIN, s[1]);
        load_voxel<CIN>(row + (size_t)(hi ? sx + 1 : sx) * CIN, s[2]);
        auto tap = [&](int kx, f32x2(&a)[4], const float(&v)[CIN]) {
            const float4 *wk = &sw[3 * kzy + kx][2 * g];
#pragma unroll
            for (int ci = 0; ci < CIN; ++ci) {
                const float4 w0 = wk[ci * (COUT / 4)], w1 = wk[ci * (COUT / 4) + 1];
                const f32x2 x = {v[ci], v[ci]};
                a[0] = fadd2(a[0], fmul2_alone(x, {w0.x, w0.y}, neg_zero));
                a[1] = fadd2(a[1], fmul2_alone(x, {w0.z, w0.w}, neg_zero));
                a[2] = fadd2(a[2], fmul2_alone(x, {w1.x, w1.y}, neg_zero));
                a[3] = fadd2(a[3], fmul2_alone(x, {w1.z, w1.w}, neg_zero));
            }
        };
        if (UP == 1) {
            if (lo) tap(0, acc[0], s[0]);
            tap(1, acc[0], s[1]);
            if (hi) tap(2, acc[0], s[2]);
        } else {
            // output 2 sx + i reads column sx + floor((i + kx - 1) / 2)
            if (lo) tap(0, acc[0], s[0]);
            tap(0, acc[UP - 1], s[1]);
            tap(1, acc[0], s[1]);
            tap(1, acc[UP - 1], s[1]);
            tap(2, acc[0], s[1]);
            if (hi) tap(2, acc[UP - 1], s[2]);
        }
    }
    float4 *o = reinterpret_cast<float4 *>(out + ((((size_t)b * d + z) * d + y) * d + (size_t)UP * sx) * COUT + 8 * g);
    auto relu = [](float v) { return v > 0.0f ? v : 0.0f; };
#pragma unroll
    for (int i = 0; i < UP; ++i)
#pragma unroll
        for (int c = 0; c < 2; ++c)
            o[i * (COUT / 4) + c] = make_float4(relu(acc[i][2 * c].x), relu(acc[i][2 * c].y), relu(acc[i][2 * c + 1].x),
                                                relu(acc[i][2 * c + 1].y));
}

// Last layer (8 -> 1 at (din * 2)^3) straight to occupancy bits.  A thread
// computes the four outputs (2 sy + j, 2 sx + i) of source cell (sy, sx) at one
// output z; the four ballots of a warp are four words (the order of the bits
// is this kernel's own).  compare != 0 counts the bits that differ from the
// stored ones into dyn[b] instead of storing.
__global__ void __launch_bounds__(kDecThreads) k_conv3d_occ(const float *in, int din, const uint16_t *w,
                                                           const uint16_t *bias, uint32_t *bits, int compare,
                                                           int64_t *dyn, int B, float neg_zero)
{
    constexpr int CIN = 8;
    __shared__ float2 sw[27][CIN];  // each weight twice, for the paired instructions
    for (int q = threadIdx.x; q < CIN * 27; q += kDecThreads) {
        const float f = bf16_bits_to_f32(w[q]);
        sw[q % 27][q / 27] = make_float2(f, f);
    }
    __syncthreads();
    griddep_launch();
    griddep_wait();
    const int d = 2 * din, lane = threadIdx.x & 31;
    // 2 din^3 = 16 N threads per sample, N a multiple of 32: a warp's outputs
    // belong to one sample, and a warp is inside the range or outside as a whole
    const size_t q = (size_t)blockIdx.x * kDecThreads + threadIdx.x;
    if (q >= (size_t)B * d * din * din) return;
    const int sx = (int)(q % din), sy = (int)((q / din) % din), z = (int)((q / ((size_t)din * din)) % d);
    const int b = (int)(q / ((size_t)din * din * d));
    const float *ib = in + (size_t)b * din * din * din * CIN;
    const bool lo = sx > 0, hi = sx < din - 1;
    const float b0 = bf16_bits_to_f32(bias[0]);
    f32x2 acc[2] = {{b0, b0}, {b0, b0}};  // output rows 2 sy, 2 sy + 1: (2 sx, 2 sx + 1)
#pragma unroll 1
    for (int kz = 0; kz < 3; ++kz) {
        const int zz = z + kz - 1;
        if (zz < 0 || zz >= d) continue;
        const float *plane = ib + (size_t)(zz / 2) * din * din * CIN;
        float s[3][3][CIN];  // rows sy - 1 .. sy + 1, columns sx - 1 .. sx + 1 (clamped)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int yy = sy + j - 1 < 0 ? 0 : (sy + j - 1 >= din ? din - 1 : sy + j - 1);
            const float *row = plane + (size_t)yy * din * CIN;
            load_voxel<CIN>(row + (size_t)(lo ? sx - 1 : sx) * CIN, s[j][0]);
            load_voxel<CIN>(row + (size_t)sx * CIN, s[j][1]);
            load_voxel<CIN>(row + (size_t)(hi ? sx + 1 : sx) * CIN, s[j][2]);
        }
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int jr = j == 0 ? (ky == 0 ? 0 : 1) : (ky == 2 ? 2 : 1);  // source row of output row j
                if (jr == 0 && sy == 0) continue;
                if (jr == 2 && sy == din - 1) continue;
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    const int c0 = kx == 0 ? 0 : 1, c1 = kx == 2 ? 2 : 1;
#pragma unroll
                    for (int ci = 0; ci < CIN; ++ci) {
                        const float2 wv = sw[9 * kz + 3 * ky + kx][ci];
                        const f32x2 n =
                            fadd2(acc[j], fmul2_alone({s[jr][c0][ci], s[jr][c1][ci]}, {wv.x, wv.y}, neg_zero));
                        // taps outside the grid are skipped
                        acc[j].x = kx == 0 && !lo ? acc[j].x : n.x;
                        acc[j].y = kx == 2 && !hi ? acc[j].y : n.y;
                    }
                }
            }
        }
    }
    uint32_t word[4];
    word[0] = __ballot_sync(0xffffffffu, acc[0].x > 0.0f);
    word[1] = __ballot_sync(0xffffffffu, acc[0].y > 0.0f);
    word[2] = __ballot_sync(0xffffffffu, acc[1].x > 0.0f);
    word[3] = __ballot_sync(0xffffffffu, acc[1].y > 0.0f);
    if (lane == 0) {
        uint4 *dst = reinterpret_cast<uint4 *>(bits) + q / 32;
        if (compare) {
            const uint4 old = *dst;
            const int flips = __popc(word[0] ^ old.x) + __popc(word[1] ^ old.y) + __popc(word[2] ^ old.z) +
                              __popc(word[3] ^ old.w);
            if (flips) atomicAdd(reinterpret_cast<unsigned long long *>(dyn + b), (unsigned long long)flips);
        } else {
            *dst = make_uint4(word[0], word[1], word[2], word[3]);
        }
    }
}

unsigned dec_grid(size_t threads) { return (unsigned)((threads + kDecThreads - 1) / kDecThreads); }

}  // namespace

size_t decode_scratch_floats(int B, int D)
{
    const size_t N = (size_t)D * D * D;
    return (size_t)B * (16 * N + 8 * 8 * N);
}

cudaError_t launch_decode_conv(const DecodeArgs &a, cudaStream_t s)
{
    if (a.B < 1 || a.D < 1 || ((size_t)a.D * a.D * a.D) % 32 != 0) return cudaErrorInvalidValue;
    const int D = a.D;
    const size_t N = (size_t)D * D * D, B = (size_t)a.B;
    float *x1 = a.scratch, *x2 = a.scratch + B * 16 * N;
    // C -> 16 at D^3 from the token-major latents S [B, N, 8]
    launch_k(k_conv3d<kChannels, 16, 1>, dim3(dec_grid(B * N * 2)), dim3(kDecThreads), 0, s, a.S, D, a.w1, a.b1, x1,
             a.B, -0.0f);
    // 16 -> 8 at (2D)^3
    launch_k(k_conv3d<16, 8, 2>, dim3(dec_grid(B * 4 * N)), dim3(kDecThreads), 0, s, (const float *)x1, D, a.w2, a.b2,
             x2, a.B, -0.0f);
    // 8 -> 1 at (4D)^3, to bits
    launch_k(k_conv3d_occ, dim3(dec_grid(B * 16 * N)), dim3(kDecThreads), 0, s, (const float *)x2, 2 * D, a.w3, a.b3,
             a.bits, a.compare, a.dyn, a.B, -0.0f);
    return cudaGetLastError();
}

}  // namespace f3dc
