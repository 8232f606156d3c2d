// Spectral bounds tightened by a few Lanczos steps (FTSP2_LANCZOS).
//
// The Gershgorin interval of Appendix A over-estimates the spectrum of dense
// Hamiltonians by the row sums of |H_ij| (a dense 0.01 N(0,1) noise on an
// n = 4096 lattice, or a random rotation of a spectrum, widen it 5 to 12
// times).  W enters beta' = W beta (Eq. beta'), hence the beta0 a model needs,
// its layer count and the amplification of rounding.  Steps (per instance, all
// instances of a batch in the same launches):
//   start  v_1 = q / ||q||, q_i = 2 u_i - 1 with u_i the top 53 bits of
//          splitmix64(i) scaled to [0, 1) (Steele, Lea, Flood 2014);
//   k = min(n, kLzSteps) steps of the three-term recurrence, no
//          re-orthogonalisation:  w = H v_j - beta_{j-1} v_{j-1},
//          alpha_j = w . v_j,  w -= alpha_j v_j,  beta_j = ||w||,  v_{j+1} = w / beta_j,
//          stopping when beta_j <= 1e-12 (|alpha_1| + beta_1 + 1).  The products
//          H v_j read an FP32 copy of H and of v_j (written by the Gershgorin
//          pass and by the previous step) with FP32 row sums: this GPU's FP64
//          rate would bound an FP64 product, and the bounds need ~1e-6 relative
//          (they carry a 1 % margin); vectors, dot products and norms stay FP64;
//   bounds the extreme eigenvalues of the tridiagonal T_m (Sturm bisection) and
//          the residual bounds r = beta_m |s_m| of their Ritz vectors (inverse
//          iteration on T_m shifted just outside its spectrum):
//          lo = theta_min - r_min - delta, hi = theta_max + r_max + delta,
//          delta = 0.01 (theta_max - theta_min) + 1e-6 max(|theta_min|, |theta_max|),
//          intersected with Gershgorin (each end kept inside it).
// Two launch shapes: batches whose instances all have n <= kLzSmallN run every
// step of an instance inside one CTA (vectors in shared memory, one CTA per
// SM so that the rows each CTA re-reads at every step can stay in L2); larger
// instances run each step as a multi-block matrix-vector launch plus an update
// launch.  The FP32 copy of H is stored per instance as a P x P slab with row
// pitch P, so every row starts 16-byte aligned.
// Reductions are in fixed order (deterministic).  The interval is not a
// rigorous enclosure; its safety terms (residual bound and the 1 % margin) are
// checked against the eigenvalues of the workload families in the tests.
#include <algorithm>

#include "div_by.h"
#include "ftsp2_internal.h"

namespace ftsp2 {

constexpr int kLzThreads = 256;

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
    unsigned long long z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// fixed-order block sum of one double per thread (T threads)
template <int T = kLzThreads>
__device__ double block_sum(double v, double* sh) {
    const int t = threadIdx.x;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((t & 31) == 0) sh[t >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (t == 0) {
        for (int w = 0; w < T / 32; ++w) s += sh[w];
        sh[T / 32] = s;
    }
    __syncthreads();
    s = sh[T / 32];
    __syncthreads();
    return s;
}

__device__ __forceinline__ double* lz_vec(const LanczosArgs& a, int which, int b) {
    double* base = which == 0 ? a.V0 : (which == 1 ? a.V1 : a.W);
    return base + (size_t)b * a.P;
}

// v_1 from the counter-based generator; v_0 = 0; steps done = 0
__global__ void __launch_bounds__(kLzThreads) lanczos_start_kernel(LanczosArgs a) {
    grid_wait();
    grid_trigger();
    __shared__ double sh[kLzThreads / 32 + 1];
    const int b = blockIdx.x;
    const int n = a.inst[b].n;
    double* v1 = lz_vec(a, 0, b);
    double* v0 = lz_vec(a, 1, b);
    float* v32 = a.V32 + (size_t)b * a.P;
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += kLzThreads) {
        const double u = (double)(splitmix64((unsigned long long)i) >> 11) * 0x1.0p-53;
        const double q = 2.0 * u - 1.0;
        v1[i] = q;
        v0[i] = 0.0;
        s += q * q;
    }
    s = block_sum(s, sh);
    __shared__ double norm[2];
    if (threadIdx.x == 0) {
        norm[0] = sqrt(s);
        norm[1] = 1.0 / norm[0];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kLzThreads) {
        v1[i] = div_by(v1[i], norm[0], norm[1]);
        v32[i] = (float)v1[i];
    }
    if (threadIdx.x == 0) a.state[b] = 0;
}

__device__ __forceinline__ bool lz_active(const LanczosArgs& a, int b, int j, int n) {
    return j < n && !(a.state[b] & kLzStopped);
}

// w = H v_j - beta_{j-1} v_{j-1}; per block (kLzRows rows, one warp each) the
// partial sum of w . v_j
__global__ void __launch_bounds__(kLzRows * 32) lanczos_matvec_kernel(LanczosArgs a, int j) {
    grid_wait();
    grid_trigger();
    const int b = blockIdx.y;
    const int n = a.inst[b].n;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = blockIdx.x * kLzRows + warp;
    __shared__ double sp[kLzRows];
    if (blockIdx.x * kLzRows >= n || !lz_active(a, b, j, n)) return;
    const double* vc = lz_vec(a, j & 1, b);
    const double* vp = lz_vec(a, (j + 1) & 1, b);
    const float* v32 = a.V32 + (size_t)b * a.P;
    double* w = lz_vec(a, 2, b);
    const double bprev = j > 0 ? a.ab[((size_t)b * kLzSteps + (j - 1)) * 2 + 1] : 0.0;
    double part = 0.0;
    if (row < n) {
        const float* Hr = a.H32 + ((size_t)b * a.P + row) * a.P;
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
        int c = lane;
        for (; c + 96 < n; c += 128) {
            s0 = fmaf(__ldg(Hr + c), v32[c], s0);
            s1 = fmaf(__ldg(Hr + c + 32), v32[c + 32], s1);
            s2 = fmaf(__ldg(Hr + c + 64), v32[c + 64], s2);
            s3 = fmaf(__ldg(Hr + c + 96), v32[c + 96], s3);
        }
        for (; c < n; c += 32) s0 = fmaf(__ldg(Hr + c), v32[c], s0);
        float sf = (s0 + s1) + (s2 + s3);
        for (int o = 16; o > 0; o >>= 1) sf += __shfl_xor_sync(0xffffffffu, sf, o);
        const double wr = (double)sf - bprev * vp[row];
        if (lane == 0) w[row] = wr;
        part = wr * vc[row];
    }
    if (lane == 0) sp[warp] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int r = 0; r < kLzRows; ++r) t += sp[r];
        a.part[(size_t)b * a.RB + blockIdx.x] = t;
    }
}

// alpha_j, w -= alpha_j v_j, beta_j = ||w||, v_{j+1} = w / beta_j (into the
// buffer of v_{j-1}); one block per instance
__global__ void __launch_bounds__(kLzThreads) lanczos_update_kernel(LanczosArgs a, int j) {
    grid_wait();
    grid_trigger();
    __shared__ double sh[kLzThreads / 32 + 1];
    const int b = blockIdx.x;
    const int n = a.inst[b].n;
    if (!lz_active(a, b, j, n)) return;
    const int nblk = (n + kLzRows - 1) / kLzRows;
    double s = 0.0;
    for (int i = threadIdx.x; i < nblk; i += kLzThreads) s += a.part[(size_t)b * a.RB + i];
    const double alpha = block_sum(s, sh);
    const double* vc = lz_vec(a, j & 1, b);
    double* vn = lz_vec(a, (j + 1) & 1, b);
    double* w = lz_vec(a, 2, b);
    s = 0.0;
    for (int i = threadIdx.x; i < n; i += kLzThreads) {
        const double wi = w[i] - alpha * vc[i];
        w[i] = wi;
        s += wi * wi;
    }
    // the square root and the reciprocal once, in one thread: by every thread they
    // and the divisions below were 2.5 of the 11 us of a step at n = 1728
    s = block_sum(s, sh);
    __shared__ double norm[2];
    __shared__ bool done;
    if (threadIdx.x == 0) {
        const double beta = sqrt(s);
        double* ab = a.ab + (size_t)b * kLzSteps * 2;
        const double a1 = j == 0 ? alpha : ab[0];
        const double b1 = j == 0 ? beta : ab[1];
        const bool stop = beta <= 1e-12 * (fabs(a1) + b1 + 1.0);
        ab[2 * j] = alpha;
        ab[2 * j + 1] = beta;
        a.state[b] = (j + 1) | (stop ? kLzStopped : 0);
        norm[0] = beta;
        norm[1] = 1.0 / beta;
        done = stop;
    }
    __syncthreads();
    if (done) return;
    const double beta = norm[0], rbeta = norm[1];
    float* v32 = a.V32 + (size_t)b * a.P;
    for (int i = threadIdx.x; i < n; i += kLzThreads) {
        const double v = div_by(w[i], beta, rbeta);
        vn[i] = v;
        v32[i] = (float)v;
    }
}

// Small instances (every n <= kLzSmallN): one CTA runs all steps of one
// instance at a time, with the Lanczos vectors in shared memory and the first
// rows of H (as many as the dynamic shared memory holds) cached there too; the
// CTAs take the instances from a queue, largest order first (longest
// processing time first: a fixed round-robin split left the CTA with the most
// large instances running about twice the mean).  The launch asks for enough shared memory that
// one CTA runs per SM, so the rows of H that the resident CTAs re-read at every
// step (one instance each, at most kLzSmallN^2 floats) stay in L2 instead of
// streaming the whole batch from HBM 24 times.  Arithmetic as in the
// multi-block kernels: FP32 products and row sums, FP64 vectors, dot
// products and norms, reductions in a fixed order.  The vectors' FP64 work is on
// eight of the 32 warps, square roots and reciprocals in one thread: a warp
// instruction takes 16 clocks of the FP64 pipe, and by every warp the square root,
// the divisions and the sums were a tenth of the kernel (ragged batch of 512:
// 2.62 ms, 2.40 now; the rest is reading the rows that are not cached).
constexpr int kLzSmallN = 1024;
constexpr int kLzSmallThreads = 1024;
constexpr int kLzSmallCacheBytes = 192 * 1024;
constexpr int kLzVecThreads = 256;               // threads of the vectors' FP64 work

// The queue of the small-instance kernel, in the partial-sum buffer (which
// only the multi-block path uses; nb RB doubles hold nb + 1 ints): queue[0]
// the next item (zeroed here), queue[1 + k] the instance of item k, by
// decreasing order n and then increasing index (the rank of b is the number
// of instances that come before it).  One thread per instance; O(nb^2)
// comparisons, a few microseconds up to kLzSortMax instances; larger batches
// keep their own order (the queue still balances the CTAs).
constexpr int kLzSortMax = 8192;
__device__ __forceinline__ int* lz_queue(const LanczosArgs& a) { return reinterpret_cast<int*>(a.part); }

__global__ void lanczos_queue_kernel(LanczosArgs a) {
    grid_wait();
    grid_trigger();
    int* const queue = lz_queue(a);
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b == 0) queue[0] = 0;
    if (b >= a.nb) return;
    int rank = b;
    if (a.nb <= kLzSortMax) {
        const int nself = a.inst[b].n;
        rank = 0;
        for (int q = 0; q < a.nb; ++q) {
            const int nq = a.inst[q].n;
            rank += (nq > nself || (nq == nself && q < b)) ? 1 : 0;
        }
    }
    queue[1 + rank] = b;
}

// Sum over the first kLzVecThreads threads in fixed order, the same in each; all of
// them call.  sh: one double a warp, not in use (two alternate between calls).
__device__ __forceinline__ double vec_sum(double v, double* sh) {
    constexpr int NV = kLzVecThreads / 32;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    asm volatile("bar.sync 1, %0;" ::"n"(kLzVecThreads) : "memory");
    v = sh[threadIdx.x % NV];
    for (int o = NV / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(kLzSmallThreads, 1) lanczos_small_kernel(LanczosArgs a) {
    grid_wait();
    __shared__ double vprev[kLzSmallN], vcur[kLzSmallN], w[kLzSmallN];
    __shared__ __align__(16) float v32[kLzSmallN];
    __shared__ double sh[2][kLzVecThreads / 32], norm[2];
    __shared__ bool done;
    __shared__ int item;
    extern __shared__ float4 hcache4[];             // rows 0 .. rc - 1 of H (FP32), pitch pc
    float* const hcache = reinterpret_cast<float*>(hcache4);
    constexpr int NW = kLzSmallThreads / 32;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    for (;;) {
        // every thread has read `item` of the previous instance: the loop body
        // ends with a barrier
        if (t == 0) item = atomicAdd(lz_queue(a), 1);
        __syncthreads();
        const int k = item;
        if (k >= a.nb) break;
        const int b = lz_queue(a)[1 + k];
        const int n = a.inst[b].n;
        const float* Hb = a.H32 + (size_t)b * a.P * a.P;
        const int pc = (n + 3) & ~3;                 // cached row pitch (16-byte rows)
        const int rc = min(n, (int)(kLzSmallCacheBytes / (4 * pc)));
        for (int i = t; i < rc * pc; i += kLzSmallThreads) {
            const int r = i / pc, c = i - r * pc;
            hcache[i] = c < n ? Hb[(size_t)r * a.P + c] : 0.f;
        }
        // v_1 from the counter-based generator, v_0 = 0
        if (t < kLzVecThreads) {
            double s = 0.0;
            for (int i = t; i < n; i += kLzVecThreads) {
                const double q = 2.0 * ((double)(splitmix64((unsigned long long)i) >> 11) * 0x1.0p-53) - 1.0;
                vcur[i] = q;
                vprev[i] = 0.0;
                s += q * q;
            }
            s = vec_sum(s, sh[1]);
            if (t == 0) {
                norm[0] = sqrt(s);
                norm[1] = 1.0 / norm[0];
            }
            asm volatile("bar.sync 1, %0;" ::"n"(kLzVecThreads) : "memory");
            for (int i = t; i < n; i += kLzVecThreads) {
                vcur[i] = div_by(vcur[i], norm[0], norm[1]);
                v32[i] = (float)vcur[i];
            }
        }
        __syncthreads();
        double* ab = a.ab + (size_t)b * kLzSteps * 2;
        const int steps = min(n, kLzSteps);
        const int n4 = n >> 2;                       // whole float4 columns; the rest per lane
        double a1 = 0.0, b1 = 0.0, bprev = 0.0;
        int m = 0;
        bool stop = false;
        for (int j = 0; j < steps && !stop; ++j) {
            // w = H v_j - beta_{j-1} v_{j-1}: two rows per warp at a time,
            // 16-byte loads (rows of H are 16-byte aligned in both copies)
            const float4* v4 = reinterpret_cast<const float4*>(v32);
            for (int row = warp; row < n; row += 2 * NW) {
                const int row2 = row + NW;
                const bool two = row2 < n;
                const float* Ra = row < rc ? hcache + (size_t)row * pc : Hb + (size_t)row * a.P;
                const float* Rb = two ? (row2 < rc ? hcache + (size_t)row2 * pc : Hb + (size_t)row2 * a.P) : Ra;
                const float4* A4 = reinterpret_cast<const float4*>(Ra);
                const float4* B4 = reinterpret_cast<const float4*>(Rb);
                float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f, t0 = 0.f, t1 = 0.f, t2 = 0.f, t3 = 0.f;
#pragma unroll 4
                for (int q = lane; q < n4; q += 32) {
                    const float4 x = A4[q], y = B4[q], v = v4[q];
                    s0 = fmaf(x.x, v.x, s0);
                    s1 = fmaf(x.y, v.y, s1);
                    s2 = fmaf(x.z, v.z, s2);
                    s3 = fmaf(x.w, v.w, s3);
                    t0 = fmaf(y.x, v.x, t0);
                    t1 = fmaf(y.y, v.y, t1);
                    t2 = fmaf(y.z, v.z, t2);
                    t3 = fmaf(y.w, v.w, t3);
                }
                const int c = 4 * n4 + lane;
                if (c < n) {
                    s0 = fmaf(Ra[c], v32[c], s0);
                    t0 = fmaf(Rb[c], v32[c], t0);
                }
                float sa = (s0 + s1) + (s2 + s3), sb = (t0 + t1) + (t2 + t3);
                for (int o = 16; o > 0; o >>= 1) {
                    sa += __shfl_xor_sync(0xffffffffu, sa, o);
                    sb += __shfl_xor_sync(0xffffffffu, sb, o);
                }
                if (lane == 0) {
                    w[row] = (double)sa - bprev * vprev[row];
                    if (two) w[row2] = (double)sb - bprev * vprev[row2];
                }
            }
            __syncthreads();
            if (t < kLzVecThreads) {
                double p = 0.0;
                for (int i = t; i < n; i += kLzVecThreads) p += w[i] * vcur[i];
                const double alpha = vec_sum(p, sh[0]);
                p = 0.0;
                for (int i = t; i < n; i += kLzVecThreads) {
                    const double wi = w[i] - alpha * vcur[i];
                    w[i] = wi;
                    p += wi * wi;
                }
                p = vec_sum(p, sh[1]);
                if (t == 0) {
                    const double beta = sqrt(p);
                    if (j == 0) {
                        a1 = alpha;
                        b1 = beta;
                    }
                    ab[2 * j] = alpha;
                    ab[2 * j + 1] = beta;
                    norm[0] = beta;
                    norm[1] = 1.0 / beta;
                    done = beta <= 1e-12 * (fabs(a1) + b1 + 1.0);
                }
                asm volatile("bar.sync 1, %0;" ::"n"(kLzVecThreads) : "memory");
                if (!done) {
                    const double beta = norm[0], rbeta = norm[1];
                    for (int i = t; i < n; i += kLzVecThreads) {
                        const double v = div_by(w[i], beta, rbeta);
                        vprev[i] = vcur[i];
                        vcur[i] = v;
                        v32[i] = (float)v;
                    }
                }
            }
            __syncthreads();
            m = j + 1;
            stop = done;
            bprev = norm[0];
        }
        if (t == 0) a.state[b] = m | (stop ? kLzStopped : 0);
        __syncthreads();
    }
}

// Number of eigenvalues below x of the m x m tridiagonal with diagonal al and
// squared off-diagonal b2 (entries of magnitude <= 2): the sign changes of the
// characteristic polynomials of its leading blocks, p_i = (al_{i-1} - x) p_{i-1}
// - b2_{i-2} p_{i-2} (Sturm).  A zero counts as a sign change.  No divisions:
// two dependent FP64 operations a step (a division takes some twenty, and they
// form one chain).
__device__ __forceinline__ int sturm_count(const double* al, const double* b2, int m, double x) {
    int cnt = 0;
    double pp = 1.0, p = al[0] - x;
    bool neg = !(p > 0.0);                       // sign of p_i, a zero counted opposite to p_{i-1}
    cnt += neg;
    for (int i = 1; i < m; ++i) {
        const double t = fma(al[i] - x, p, -b2[i - 1] * pp);
        pp = p;
        p = t;
        // keep the pair away from underflow (nearly decoupled, nearly equal entries)
        if (((__double2hiint(p) >> 20) & 0x7ff) < 500 && ((__double2hiint(pp) >> 20) & 0x7ff) < 500) {
            p *= 0x1p+400;
            pp *= 0x1p+400;
        }
        const bool n2 = p == 0.0 ? !neg : p < 0.0;
        cnt += n2 != neg;
        neg = n2;
    }
    return cnt;
}

// |last entry| of the unit eigenvector for the eigenvalue theta at the edge of
// the spectrum: inverse iteration with the shift sigma just outside, where
// T - sigma I is definite and the tridiagonal elimination needs no pivoting.
// The factors are formed once (reciprocal pivots), each solve then takes one
// FMA chain down and one up.
__device__ __forceinline__ double edge_vector_last(const double* al, const double* be, int m, double sigma) {
    double x[kLzSteps], r[kLzSteps];             // iterate; 1 / pivot
#pragma unroll
    for (int i = 0; i < kLzSteps; ++i) {
        x[i] = 1.0;
        r[i] = 0.0;
        if (i < m) {
            const double l = i > 0 ? be[i - 1] * r[i > 0 ? i - 1 : 0] : 0.0;
            r[i] = 1.0 / (i > 0 ? (al[i] - sigma) - l * be[i - 1] : al[i] - sigma);
        }
    }
    for (int it = 0; it < 3; ++it) {
        // solve (T - sigma I) y = x, y into x
#pragma unroll
        for (int i = 1; i < kLzSteps; ++i)
            if (i < m) x[i] -= (be[i - 1] * r[i - 1]) * x[i - 1];
        double nrm = 0.0, up = 0.0;              // up = be_i y_{i+1}
#pragma unroll
        for (int i = kLzSteps - 1; i >= 0; --i)
            if (i < m) {
                x[i] = (x[i] - up) * r[i];
                nrm += x[i] * x[i];
                if (i > 0) up = be[i - 1] * x[i];
            }
        const double inv = 1.0 / sqrt(nrm);
#pragma unroll
        for (int i = 0; i < kLzSteps; ++i) x[i] *= inv;
    }
    double last = 0.0;
#pragma unroll
    for (int i = 0; i < kLzSteps; ++i)
        if (i == m - 1) last = fabs(x[i]);
    return last;
}

// Two warps per instance: warp 0 the lower edge of the spectrum of T_m, warp 1
// the upper one.  The edge eigenvalue by multisection: the 32 lanes count the
// eigenvalues below 32 points of the bracket, which shrinks 33-fold per round;
// 8 rounds leave the edge within 33^-8 < 1e-12 of the bracket (the Gershgorin
// interval of T), far below the 1 % margin, and inside the 1e-10 shift of the
// residual bound's inverse iteration.  Bound by the latency of dependent FP64
// operations; one instance took 379 us with one warp, divisions in the Sturm
// counts and the factors formed anew in each solve, 84 us now.
__global__ void __launch_bounds__(64) lanczos_bounds_kernel(LanczosArgs a) {
    grid_wait();
    grid_trigger();
    __shared__ double al[kLzSteps], be[kLzSteps], sal[kLzSteps], sb2[kLzSteps];
    __shared__ double edge[2], res[2];
    const int lane = threadIdx.x & 31, upper = threadIdx.x >> 5;
    const int b = blockIdx.x;
    const int m = a.state[b] & (kLzStopped - 1);
    if (m < 1) return;
    const double* ab = a.ab + (size_t)b * kLzSteps * 2;
    if (threadIdx.x < m) {
        al[threadIdx.x] = ab[2 * threadIdx.x];
        be[threadIdx.x] = ab[2 * threadIdx.x + 1];
    }
    __syncthreads();
    // Gershgorin interval of T (lane i: row i)
    double lo = 1e300, hi = -1e300;
    bool finite = true;
    if (lane < m) {
        finite = isfinite(al[lane]) && isfinite(be[lane]);
        const double r = (lane > 0 ? fabs(be[lane - 1]) : 0.0) + (lane + 1 < m ? fabs(be[lane]) : 0.0);
        lo = al[lane] - r;
        hi = al[lane] + r;
    }
    if (!__all_sync(0xffffffffu, finite)) return;   // the Gershgorin bounds stay (and flag the input)
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    // in units of the interval, from its lower end: T' = (T - lo) 2^-e
    const int ex = hi > lo ? ilogb(hi - lo) : 0;
    if (threadIdx.x < m) {
        const double f = scalbn(be[threadIdx.x], -ex);
        sal[threadIdx.x] = scalbn(al[threadIdx.x] - lo, -ex);
        sb2[threadIdx.x] = f * f;
    }
    __syncthreads();
    double l = 0.0, h = scalbn(hi - lo, -ex);
    const int target = upper ? m : 1;
    if (h > 0.0)
        for (int it = 0; it < 8; ++it) {
            const double x = l + (h - l) * ((double)(lane + 1) * (1.0 / 33.0));
            const bool hit = sturm_count(sal, sb2, m, x) >= target;
            const unsigned mask = __ballot_sync(0xffffffffu, hit);
            const int k = mask ? __ffs(mask) - 1 : 32;       // the first point with enough eigenvalues below
            const double xk = __shfl_sync(0xffffffffu, x, k & 31);
            const double xk1 = __shfl_sync(0xffffffffu, x, k > 0 ? k - 1 : 0);
            if (k > 0) l = xk1;
            if (k < 32) h = xk;
        }
    if (lane == 0) edge[upper] = lo + scalbn(h, ex);
    __syncthreads();
    const double tmin = edge[0], tmax = edge[1];
    const double scale = fmax(fabs(tmin), fabs(tmax)) + (tmax - tmin) + 1e-300;
    if (lane == 0) {
        const double blast = be[m - 1];
        double r = 0.0;
        if (m > 1 && blast > 0.0)
            r = blast * edge_vector_last(al, be, m, upper ? tmax + 1e-10 * scale : tmin - 1e-10 * scale);
        else if (m == 1) r = blast;
        res[upper] = r;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    // 1 % of the Ritz spread, plus 1e-6 of the Ritz magnitude for the FP32 products
    const double delta = 0.01 * (tmax - tmin) + 1e-6 * fmax(fabs(tmin), fabs(tmax));
    const double elo = tmin - res[0] - delta, ehi = tmax + res[1] + delta;
    const double glo = dunkey(a.iw[b].kmin), ghi = dunkey(a.iw[b].kmax);
    if (!(isfinite(elo) && isfinite(ehi) && isfinite(glo) && isfinite(ghi))) return;
    // intersected with the Gershgorin interval, each end kept inside it
    a.iw[b].kmin = dkey(fmax(glo, fmin(elo, ghi)));
    a.iw[b].kmax = dkey(fmin(ghi, fmax(ehi, glo)));
}

static size_t lz_align(size_t x) { return (x + 1023) / 1024 * 1024; }

size_t lanczos_ws_bytes(int nb, int P) {
    const size_t vec = lz_align(sizeof(double) * (size_t)nb * P);
    const int RB = (P + kLzRows - 1) / kLzRows;
    return 3 * vec + lz_align(sizeof(float) * (size_t)nb * P) + lz_align(sizeof(double) * (size_t)nb * kLzSteps * 2) +
           lz_align(sizeof(double) * (size_t)nb * RB) + lz_align(sizeof(int) * (size_t)nb);
}

void lanczos_bind(LanczosArgs& a, uint8_t* ws, int nb, int P) {
    const size_t vec = lz_align(sizeof(double) * (size_t)nb * P);
    a.nb = nb;
    a.P = P;
    a.RB = (P + kLzRows - 1) / kLzRows;
    size_t off = 0;
    a.V0 = reinterpret_cast<double*>(ws + off);
    off += vec;
    a.V1 = reinterpret_cast<double*>(ws + off);
    off += vec;
    a.W = reinterpret_cast<double*>(ws + off);
    off += vec;
    a.V32 = reinterpret_cast<float*>(ws + off);
    off += lz_align(sizeof(float) * (size_t)nb * P);
    a.ab = reinterpret_cast<double*>(ws + off);
    off += lz_align(sizeof(double) * (size_t)nb * kLzSteps * 2);
    a.part = reinterpret_cast<double*>(ws + off);
    off += lz_align(sizeof(double) * (size_t)nb * a.RB);
    a.state = reinterpret_cast<int*>(ws + off);
}

void launch_lanczos(const LanczosArgs& a, int max_n, int sms, cudaStream_t s) {
    if (max_n <= kLzSmallN) {
        static bool attr = false;
        if (!attr) {
            cudaFuncSetAttribute(lanczos_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kLzSmallCacheBytes);
            attr = true;
        }
        launch_after(lanczos_queue_kernel, dim3((a.nb + 255) / 256), dim3(256), 0, s, a);
        launch_after(lanczos_small_kernel, dim3(std::min(a.nb, std::max(1, sms))), dim3(kLzSmallThreads),
                     kLzSmallCacheBytes, s, a);
        launch_after(lanczos_bounds_kernel, dim3(a.nb), dim3(64), 0, s, a);
        count_launch(3);
        return;
    }
    launch_after(lanczos_start_kernel, dim3(a.nb), dim3(kLzThreads), 0, s, a);
    count_launch();
    const int steps = max_n < kLzSteps ? max_n : kLzSteps;
    const dim3 mgrid((max_n + kLzRows - 1) / kLzRows, a.nb);
    for (int j = 0; j < steps; ++j) {
        launch_after(lanczos_matvec_kernel, mgrid, dim3(kLzRows * 32), 0, s, a, j);
        launch_after(lanczos_update_kernel, dim3(a.nb), dim3(kLzThreads), 0, s, a, j);
        count_launch(2);
    }
    launch_after(lanczos_bounds_kernel, dim3(a.nb), dim3(64), 0, s, a);
    count_launch();
}

}  // namespace ftsp2
