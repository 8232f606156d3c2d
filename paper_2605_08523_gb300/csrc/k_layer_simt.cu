// (a3)-(a6) One layer of the centred recursion with FP32 FMA products on the
// CUDA cores: the FTSP2_FP32 mode and the FP32 refinement layers
// (FTSP2_REFINE1/2).  Same triangular 128 x 128 tile list and epilogue
// arithmetic as the tensor-core kernel (plus the Max-SP2 layers, which only
// this kernel runs); the operand is the full symmetric FP32 matrix Z_k
// (written for this layer by the previous layer's epilogue).
//
// Bound by the FP32 pipes (n^3 FMAs per chain on the triangle against 24 n^2
// bytes).  One CTA of 128 threads computes one 64 x 64 quadrant of a tile,
// 8 x 4 outputs per thread, four or five CTAs per SM:
// * the quadrants, one CTA each, spread a layer over the SMs by the hardware's
//   block scheduler (at n = 1728 the 210 tiles of 128 x 128 were 1.4 waves of
//   152 one-CTA SMs, i.e. two); the quadrant left of the diagonal of a
//   diagonal tile, and quadrants past the order, are not computed;
// * Z is symmetric, so the K-major panels Z[k][row] that the outer products
//   read are rows of Z: 16-byte cp.async copies straight into shared memory,
//   a four-deep ring of 16-row slices;
// * fma.rn.f32x2 forms two outputs per instruction: with the row pair
//   (a0, a1) and the column pair (b0, b1) the outputs (00, 11) take the pair as
//   it is and (01, 10) the swapped pair, so one swap per column pair and k
//   replaces a duplicated operand per row;
// * the sums are those of one FMA per k in increasing k over 128-element
//   chunks of K (`part`), the chunks added in order into `acc`;
// * the finished sums go through shared memory, so that in the epilogue a lane
//   owns a row of a 32 x 8 block: the blocked state is read and written in
//   512-byte runs, a direct operand row in 32-byte vectors and a mirror column
//   in 128-byte runs.
#include "epilogue.cuh"
#include "ftsp2_internal.h"

namespace ftsp2 {

constexpr int kSQ = 64;          // quadrant edge
constexpr int kSK = 16;          // K slice
constexpr int kSStages = 4;
constexpr int kSThreads = 128;
constexpr int kSWarps = kSThreads / 32;
constexpr int kSPitch = kSQ + 1; // pitch of the staged sums
static_assert(kSStages * 2 * kSK * kSQ >= kSQ * kSPitch, "the ring holds the staged sums");

typedef unsigned long long f32x2;      // two packed FP32 values

__device__ __forceinline__ void fma2(f32x2& d, f32x2 a, f32x2 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ f32x2 swap2(f32x2 v) { return (v >> 32) | (v << 32); }
__device__ __forceinline__ float lo2(f32x2 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi2(f32x2 v) { return __uint_as_float((unsigned)(v >> 32)); }

__global__ void __launch_bounds__(kSThreads, 4) layer_simt_kernel(const __grid_constant__ LayerArgs a) {
    __shared__ __align__(16) float sm[kSStages * 2 * kSK * kSQ];
    grid_wait();
    // no instance starts before status[1]: a layer below it has nothing to do
    if (a.gl < *reinterpret_cast<volatile const int*>(a.status + 1)) return;
    const int t = blockIdx.x >> 2, quad = blockIdx.x & 3;
    const Tile tl = a.tiles[t];
    int k;
    if (!tile_active(a, tl, k)) return;
    const int n = a.inst[tl.inst].n;
    const int rowA = tl.I * 128 + (quad >> 1) * kSQ, rowB = tl.J * 128 + (quad & 1) * kSQ;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (rowA > rowB || rowA >= n || rowB >= n) return;
    const float* const Op = reinterpret_cast<const float*>(a.opr[tl.chain]) + (size_t)tl.inst * a.P * a.P;
    // outputs of a thread: rows 8 ty .. + 7, columns 4 tx .. + 3 (a warp covers 32 x 32)
    const int ty = (warp >> 1) * 4 + (lane >> 3), tx = (warp & 1) * 8 + (lane & 7);
    const int nk = (n + kSK - 1) / kSK;        // slices; columns and rows n .. 16 nk - 1 are zero
    // copies of a slice: 16 rows of 64 floats of either panel, 16-byte chunks
    const int lrow = tid >> 4, lcol = (tid & 15) * 4;
    const float* const srcA = Op + (size_t)lrow * a.P + rowA + lcol;
    const float* const srcB = Op + (size_t)lrow * a.P + rowB + lcol;
    const uint32_t dst0 = smem_u32(sm) + 4u * (lrow * kSQ + lcol);
    auto load = [&](int kb) {
        const uint32_t d = dst0 + 4u * ((kb % kSStages) * 2 * kSK * kSQ);
        const size_t o = (size_t)kb * kSK * a.P, h = (size_t)(kSK / 2) * a.P;
        cp_async16(d, srcA + o);
        cp_async16(d + 4u * (kSK / 2 * kSQ), srcA + o + h);
        cp_async16(d + 4u * (kSK * kSQ), srcB + o);
        cp_async16(d + 4u * (kSK * kSQ + kSK / 2 * kSQ), srcB + o + h);
    };
#pragma unroll
    for (int s = 0; s < kSStages - 1; ++s) {
        if (s < nk) load(s);
        cp_async_commit();
    }
    // pair (i2, j2): straight = outputs (2 i2, 2 j2), (2 i2 + 1, 2 j2 + 1); crossed =
    // (2 i2, 2 j2 + 1), (2 i2 + 1, 2 j2)
    f32x2 ps[4][2], px[4][2];
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) ps[i][j] = px[i][j] = 0ull;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int kb = 0; kb < nk; ++kb) {
        cp_async_wait<kSStages - 2>();
        __syncthreads();
        if (kb + kSStages - 1 < nk) load(kb + kSStages - 1);
        cp_async_commit();
        const float* const As = sm + (kb % kSStages) * 2 * kSK * kSQ + ty * 8;
        const float* const Bs = sm + (kb % kSStages) * 2 * kSK * kSQ + kSK * kSQ + tx * 4;
#pragma unroll
        for (int kk = 0; kk < kSK; ++kk) {
            const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(As + kk * kSQ);
            const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(As + kk * kSQ + 4);
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(Bs + kk * kSQ);
            const f32x2 av[4] = {a0.x, a0.y, a1.x, a1.y}, bv[2] = {b0.x, b0.y};
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const f32x2 bs = swap2(bv[j]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    fma2(ps[i][j], av[i], bv[j]);
                    fma2(px[i][j], av[i], bs);
                }
            }
        }
        if ((kb & 7) == 7 || kb == nk - 1) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    acc[2 * i][2 * j] += lo2(ps[i][j]);
                    acc[2 * i + 1][2 * j + 1] += hi2(ps[i][j]);
                    acc[2 * i][2 * j + 1] += lo2(px[i][j]);
                    acc[2 * i + 1][2 * j] += hi2(px[i][j]);
                    ps[i][j] = px[i][j] = 0ull;
                }
        }
    }
    __syncthreads();                           // the ring is free (its last copies were waited for)
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sm[(ty * 8 + i) * kSPitch + tx * 4 + j] = acc[i][j];
    __syncthreads();
    EpiCtx e;
    make_ctx(a, tl, k, e);
    double tr = 0.0, sq = 0.0;
    // 32 x 8 blocks of the quadrant, lane = row
#pragma unroll 1
    for (int s = warp; s < 2 * kSQ / 8; s += kSWarps) {
        const int r0 = (s & 1) * 32, c = (s >> 1) * 8;
        const int r = rowA + r0 + lane, c0 = rowB + c;
        if (!(c0 < n && c0 + 7 >= rowA + r0)) continue;
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = sm[(r0 + lane) * kSPitch + c + j];
        if (e.L.nplanes > 0) epi_segment_max(a, e, r, c0, v, tr, sq);
        else epi_segment(a, e, r, c0, v, tr, sq);
    }
    if (a.last) {
        // warps w and w + 2 have the column groups of one 32 x 64 block
        __shared__ double red[kSWarps][2];
        for (int o = 16; o > 0; o >>= 1) {
            tr += __shfl_xor_sync(0xffffffffu, tr, o);
            sq += __shfl_xor_sync(0xffffffffu, sq, o);
        }
        if (lane == 0) {
            red[warp][0] = tr;
            red[warp][1] = sq;
        }
        __syncthreads();
        if (tid < 2 && rowA + 32 * tid < n)
            store_partial(a, tl.inst, tl.chain, (rowA >> 5) + tid, rowB >> 6, red[tid][0] + red[tid + 2][0],
                          red[tid][1] + red[tid + 2][1]);
    }
}

cudaError_t launch_layer_simt(const LayerArgs& a, cudaStream_t s) {
    const cudaError_t e = launch_after(layer_simt_kernel, dim3(4 * a.ntiles), dim3(kSThreads), 0, s, a);
    count_launch();
    return e;
}

}  // namespace ftsp2
