// Epilogue of one layer of the centred recursion, shared by the tensor-core
// and the CUDA-core layer kernels.  For an owned element (r, c), r <= c, with
// the constants of DevLayer:
//   xh = mul (Z_k^2)_{rc} + bp (Z_k)_{rc},   A' = A + d (Z_k)_{rc} + d2 xh,
//   Z_{k+1} = p xh + q A
// (centred Eq. mlsp2: Z_{k+1} = a_k Z_k^2 + (b_k + 2 a_k tau_k) Z_k,
// A' = A + d_k Z_k; centred Skip-SP2 with one stored layer and one
// accumulator: the square of the combination, then the next combination)
// then either the next layer's operands are written at (r, c) and (c, r), or,
// at the last layer, D = G + f0 I (Appendix A output, flipped as I - (A + X)
// when Eq. flip was used) is written and the FP64 partial sums of G are formed.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "ftsp2_internal.h"

namespace ftsp2 {

// Is tile `t` active at global layer g?  Returns the instance's local layer k.
__device__ __forceinline__ bool tile_active_g(const LayerArgs& a, const Tile& t, int g, int& k) {
    const ftsp2_rescale_rec& rec = a.rec[t.inst];
    if (rec.status != FTSP2_OK || rec.model < 0) return false;
    const int start = (a.iw[t.inst].start_layer >> (16 * t.chain)) & 0xffff;
    k = g - start;
    return k >= 0;
}
// ... at this launch's (first) layer
__device__ __forceinline__ bool tile_active(const LayerArgs& a, const Tile& t, int& k) {
    return tile_active_g(a, t, a.gl, k);
}

// 16-byte asynchronous global -> shared copies through the load/store path
// (cp.async, L2 only).  The store warps of the tensor-core kernel use them so
// that their loads do not queue behind the operand tiles in the TMA unit.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void store_partial(const LayerArgs& a, int inst, int chain, int rb, int cb, double tr,
                                              double sq) {
    double2* const p = reinterpret_cast<double2*>(a.partials) +
                       ((size_t)inst * a.nchains + chain) * partial_blocks(a.P) + partial_index(rb, cb);
    *p = make_double2(tr, sq);
}

struct EpiCtx {
    int n, P, chain, kind, flip, last;
    float mul;            // multiplier of the product: a_k
    size_t slab;          // b * P * P
    int64_t doff;         // D offset
    DevLayer L;
    double cdiag;         // f0 (or 1 - f0 when flipped) added on the diagonal of D
};

// CUDA-core epilogues: row r, columns c0 .. c0 + 7 (c0 % 8 == 0) with the
// products v, one row per lane of a 32-row block.  The next layer's operands
// are the full FP32 matrix: the direct row as two 16-byte vectors when all of
// it lies in the triangle and the order, the mirror (c, r) one element per
// lane, a contiguous run of row c across the warp.
__device__ __forceinline__ void store_operands8(const LayerArgs& a, const EpiCtx& e, int r, int c0, const float* z) {
    float* const op = reinterpret_cast<float*>(a.opw[e.chain]) + e.slab;
    float* const row = op + (size_t)r * e.P + c0;
    if (r <= c0 && c0 + 7 < e.n) {
        reinterpret_cast<float4*>(row)[0] = make_float4(z[0], z[1], z[2], z[3]);
        reinterpret_cast<float4*>(row)[1] = make_float4(z[4], z[5], z[6], z[7]);
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (c0 + j < e.n && r <= c0 + j) row[j] = z[j];
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (c0 + j < e.n && r < c0 + j) op[(size_t)(c0 + j) * e.P + r] = z[j];
}

// Last layer: D from the centred output g (Fermi chain) and the (diagonal sum,
// weighted square sum) of g in FP64.
__device__ __forceinline__ void store_last8(const LayerArgs& a, const EpiCtx& e, int r, int c0, const float* g,
                                            double& tr, double& sq) {
    const bool dout = e.kind == CHAIN_FERMI && a.D;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int c = c0 + j;
        if (c < e.n && r <= c) {
            if (dout) {
                float dv;
                if (e.flip) dv = (r == c ? (float)e.cdiag : 0.f) - g[j];
                else dv = g[j] + (r == c ? (float)e.cdiag : 0.f);
                a.D[e.doff + (int64_t)r * e.n + c] = dv;
                if (c != r) a.D[e.doff + (int64_t)c * e.n + r] = dv;
            }
            const double gd = (double)g[j];
            if (r == c) {
                tr += gd;
                sq += gd * gd;
            } else {
                sq += 2.0 * gd * gd;
            }
        }
    }
}

// The 8 state values of row r, columns c0 .. c0 + 7 (two float4 runs 128 floats
// apart in the blocked layout).
__device__ __forceinline__ void load_state8(const float* S, float* x) {
    const float4 u = reinterpret_cast<const float4*>(S)[0], w = reinterpret_cast<const float4*>(S + 128)[0];
    x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w; x[4] = w.x; x[5] = w.y; x[6] = w.z; x[7] = w.w;
}
__device__ __forceinline__ void store_state8(float* S, const float* x) {
    reinterpret_cast<float4*>(S)[0] = make_float4(x[0], x[1], x[2], x[3]);
    reinterpret_cast<float4*>(S + 128)[0] = make_float4(x[4], x[5], x[6], x[7]);
}

__device__ __forceinline__ void epi_segment(const LayerArgs& a, const EpiCtx& e, int r, int c0, const float* v,
                                            double& tr, double& sq) {
    if (r >= e.n) return;
    const size_t so = e.slab + state_off(e.P, r, c0);
    float* const Zs = a.Z[e.chain] + so;
    float* const As = a.A[e.chain] + so;
    float z[8], ac[8], zn[8], an[8];
    load_state8(Zs, z);
    load_state8(As, ac);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float xh = fmaf(e.mul, v[j], e.L.bp * z[j]);
        an[j] = fmaf(e.L.d2, xh, fmaf(e.L.d, z[j], ac[j]));
        zn[j] = e.last ? fmaf(e.L.g, xh, an[j]) : fmaf(e.L.p, xh, e.L.q * ac[j]);
    }
    if (!e.last) {
        store_state8(Zs, zn);
        store_state8(As, an);
        store_operands8(a, e, r, c0, zn);
    } else {
        store_last8(a, e, r, c0, zn, tr, sq);
    }
}

// Max-SP2 layer k (FP32 mode, CUDA-core layers only).  State plane j of the
// chain holds the centred stored layer x^_j = X_j - chi_j I (chi_j the layer
// values along the trajectory of mu0, sigma_k the combination's value there);
// the operands of layer k are the centred combination
// U^_k = sum_{j<=k} theta_{k,j} x^_j, and with v = (U^_k^2)_{rc}:
//   x^_{k+1} = v + 2 sigma_k U^_k          (bp = 2 sigma_k, mul = 1)
// is stored as plane k + 1 and the operands of layer k + 1,
// U^_{k+1} = sum_{j<=k+1} theta_{k+1,j} x^_j, are written at (r, c) and (c, r);
// the last layer forms G = sum_{j<=L} gamma_j x^_j instead (D = G + f0 I).
// U^_k is re-formed here from the planes in the order its operands were
// formed, so it equals the operand value the product used.
__device__ __forceinline__ void epi_segment_max(const LayerArgs& a, const EpiCtx& e, int r, int c0, const float* v,
                                                double& tr, double& sq) {
    if (r >= e.n) return;
    float* const X = a.Z[e.chain] + e.slab + state_off(e.P, r, c0);
    const int k1 = e.L.nplanes;                    // k + 1 stored layers are read
    const float* th = a.coef + e.L.coef;           // theta_{k,0..k}
    const float* tn = th + k1;                     // theta_{k+1,0..k+1}
    const float* gm = tn + k1 + 1;                 // gamma_{0..L} (last layer)
    float ui[8], un[8];                            // un: U^_{k+1} so far, or G at the last layer
#pragma unroll
    for (int j = 0; j < 8; ++j) ui[j] = un[j] = 0.f;
#pragma unroll 4
    for (int p = 0; p < k1; ++p) {
        const float tk = th[p], tq = e.last ? gm[p] : tn[p];
        float x[8];
        load_state8(X + (size_t)p * a.plane_elems, x);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            ui[j] = fmaf(tk, x[j], ui[j]);
            un[j] = fmaf(tq, x[j], un[j]);
        }
    }
    float xn[8];
    const float tl = e.last ? gm[k1] : tn[k1];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        xn[j] = fmaf(e.mul, v[j], e.L.bp * ui[j]);
        un[j] = fmaf(tl, xn[j], un[j]);
    }
    if (!e.last) {
        store_state8(X + (size_t)k1 * a.plane_elems, xn);
        store_operands8(a, e, r, c0, un);
    } else {
        store_last8(a, e, r, c0, un, tr, sq);
    }
}

__device__ __forceinline__ void make_ctx(const LayerArgs& a, const Tile& t, int k, EpiCtx& e) {
    const ftsp2_instance in = a.inst[t.inst];
    const ftsp2_rescale_rec& rec = a.rec[t.inst];
    const DevModel& M = a.models[rec.model];
    e.n = in.n;
    e.P = a.P;
    e.chain = t.chain;
    e.kind = a.chain_kind[t.chain];
    e.flip = rec.flip;
    e.last = a.last;
    e.slab = (size_t)t.inst * a.P * a.P;
    e.doff = in.offset;
    e.L = a.layers[(e.kind == CHAIN_ENTROPY ? M.offS : M.off) + k];
    e.cdiag = rec.flip ? 1.0 - M.f0 : M.f0;
    e.mul = e.L.a;
}

}  // namespace ftsp2
