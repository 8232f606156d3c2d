// (a7) Training kernels (Sec. II C): per-sample forward and reverse sweep of the
// scalar recursion (Eq. mlsp2, Skip-SP2 with one stored layer and one
// accumulator, or Max-SP2; each also under the entropy expansion of Eqs.
// entropy expansion / entropy expansion-s), and the FP64 reductions of one
// Levenberg-Marquardt iteration.
//
// Layout: the augmented Jacobian M = [J | r] is stored parameter-major,
// M[j * ns + s] (column j of J contiguous over samples), j = 0..np-1 for
// the table entries (a_0, b_0, c_0, d_0, a_1, ...), j = np for the residual.
// The Gram matrix G = M^T M holds J^T J, J^T r and r^T r; it is reduced over
// fixed sample chunks and then over chunks in a fixed order (deterministic).
#include "ftsp2_internal.h"

namespace ftsp2 {

constexpr int kTrainMaxL = kMaxLayers;

__device__ __forceinline__ double target_value(int target, double x, double beta0, double mu0) {
    const double t = beta0 * (x - mu0);
    if (target == FTSP2_TARGET_ENTROPY) {
        const double at = fabs(t);
        const double e = exp(-at);
        return log1p(e) + at * e / (1.0 + e);
    }
    // increasing logistic 1/(1 + exp(-t)), evaluated without overflow
    if (t >= 0.0) return 1.0 / (1.0 + exp(-t));
    const double e = exp(t);
    return e / (1.0 + e);
}

template <bool WITH_J>
__global__ void __launch_bounds__(128) fwd_kernel(int target, double beta0, double mu0, int L, double alpha,
                                                  const __grid_constant__ ThetaParam thp,
                                                  const double* __restrict__ X, int ns,
                                                  double* __restrict__ R, double* __restrict__ M) {
    const double* th = thp.v;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ns) return;
    const double x = X[s];
    double xs[kTrainMaxL + 1];
    double xi = target == FTSP2_TARGET_ENTROPY ? alpha * (x - mu0) + mu0 : x;
    double A = 0.0;
    for (int i = 0; i < L; ++i) {
        xs[i] = xi;
        const double a = th[4 * i], b = th[4 * i + 1], c = th[4 * i + 2],
                     d = th[4 * i + 3];
        A = fma(d, xi, A);
        xi = fma(fma(a, xi, b), xi, c);
    }
    const double F = A + xi;
    double out = F, fac = 1.0;
    if (target == FTSP2_TARGET_ENTROPY) {
        const double k4 = 4.0 * 0.69314718055994530942;
        out = k4 * F * (1.0 - F);
        fac = k4 * (1.0 - 2.0 * F);
    }
    const double r = out - target_value(target, x, beta0, mu0);
    R[s] = r;
    if (!WITH_J) return;
    const int np = 4 * L;
    M[(size_t)np * ns + s] = r;
    double g = 1.0;
    for (int i = L - 1; i >= 0; --i) {
        const double a = th[4 * i], b = th[4 * i + 1], d = th[4 * i + 3];
        const double x_i = xs[i];
        M[(size_t)(4 * i + 0) * ns + s] = fac * g * x_i * x_i;
        M[(size_t)(4 * i + 1) * ns + s] = fac * g * x_i;
        M[(size_t)(4 * i + 2) * ns + s] = fac * g;
        M[(size_t)(4 * i + 3) * ns + s] = fac * x_i;
        g = fma(g, fma(2.0 * a, x_i, b), d);
    }
}

// Skip-SP2 with one stored layer and one accumulator (Sec. II A 3): th holds
// L rows (delta, alpha, beta, gamma) and the output row (A_0, gamma_L);
// u_i = delta_i + alpha_i x_i + beta_i A_i, A_{i+1} = A_i + gamma_i x_i,
// x_{i+1} = u_i^2, F = A_L + gamma_L x_L.  Reverse sweep with gx = dF/dx_i,
// gA = dF/dA_i: w = 2 u_i gx_{i+1} gives dF/d(delta, alpha, beta)_i =
// w (1, x_i, A_i), dF/dgamma_i = gA_{i+1} x_i, gx_i = w alpha_i + gA_{i+1}
// gamma_i, gA_i = w beta_i + gA_{i+1}; dF/dA_0 = gA_0, dF/dgamma_L = x_L.
// Columns j < 4L + 2 in that flattened order, the residual in column 4L + 2.
template <bool WITH_J>
__global__ void __launch_bounds__(128) fwd_skip_kernel(int target, double beta0, double mu0, int L, double alpha,
                                                       const __grid_constant__ ThetaParam thp,
                                                       const double* __restrict__ X, int ns,
                                                       double* __restrict__ R, double* __restrict__ M) {
    const double* th = thp.v;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ns) return;
    const double x = X[s];
    double xs[kTrainMaxL], As[kTrainMaxL], us[kTrainMaxL];
    double xi = target == FTSP2_TARGET_ENTROPY ? alpha * (x - mu0) + mu0 : x;
    double A = th[4 * L];
    for (int i = 0; i < L; ++i) {
        xs[i] = xi;
        As[i] = A;
        const double u = fma(th[4 * i + 2], A, fma(th[4 * i + 1], xi, th[4 * i]));
        us[i] = u;
        A = fma(th[4 * i + 3], xi, A);
        xi = u * u;
    }
    const double F = fma(th[4 * L + 1], xi, A);
    double out = F, fac = 1.0;
    if (target == FTSP2_TARGET_ENTROPY) {
        const double k4 = 4.0 * 0.69314718055994530942;
        out = k4 * F * (1.0 - F);
        fac = k4 * (1.0 - 2.0 * F);
    }
    const double r = out - target_value(target, x, beta0, mu0);
    R[s] = r;
    if (!WITH_J) return;
    const int np = 4 * L + 2;
    M[(size_t)np * ns + s] = r;
    M[(size_t)(4 * L + 1) * ns + s] = fac * xi;
    double gx = th[4 * L + 1], gA = 1.0;
    for (int i = L - 1; i >= 0; --i) {
        const double w = 2.0 * us[i] * gx;
        M[(size_t)(4 * i + 0) * ns + s] = fac * w;
        M[(size_t)(4 * i + 1) * ns + s] = fac * w * xs[i];
        M[(size_t)(4 * i + 2) * ns + s] = fac * w * As[i];
        M[(size_t)(4 * i + 3) * ns + s] = fac * gA * xs[i];
        const double gx_i = fma(w, th[4 * i + 1], gA * th[4 * i + 3]);
        gA = fma(w, th[4 * i + 2], gA);
        gx = gx_i;
    }
    M[(size_t)(4 * L) * ns + s] = fac * gA;
}

// Max-SP2 (Sec. II A 2, Eq. maxsp2) on the flat table th: for i < L the block
// (delta_i, gamma_i, theta_{i,0..i}) at off_i = i (i + 5) / 2, then (c, gamma_L);
// u_i = delta_i + sum_{j<=i} theta_{i,j} x_j, x_{i+1} = u_i^2,
// F = c + sum_{j<=L} gamma_j x_j.  Reverse sweep with g_j = dF/dx_j (from
// gamma_j; g_{i+1} is final once the layers after i are done):
// w = 2 u_i g_{i+1}, dF/d delta_i = w, dF/d theta_{i,j} = w x_j,
// g_j += w theta_{i,j}; dF/d gamma_j = x_j, dF/dc = 1.  Columns in the flat
// order, the residual after them.
constexpr int kTrainMaxMaxL = kMaxMaxLayers;

template <bool WITH_J>
__global__ void __launch_bounds__(128) fwd_max_kernel(int target, double beta0, double mu0, int L, double alpha,
                                                      const __grid_constant__ ThetaParam thp,
                                                      const double* __restrict__ X, int ns,
                                                      double* __restrict__ R, double* __restrict__ M) {
    const double* th = thp.v;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ns) return;
    const double x = X[s];
    double xs[kTrainMaxMaxL + 1], us[kTrainMaxMaxL], g[kTrainMaxMaxL + 1];
    xs[0] = target == FTSP2_TARGET_ENTROPY ? alpha * (x - mu0) + mu0 : x;
    const int oc = L * (L + 5) / 2;            // offset of (c, gamma_L)
    double F = th[oc];
    for (int i = 0; i < L; ++i) {
        const int o = i * (i + 5) / 2;
        double u = th[o];
        for (int j = 0; j <= i; ++j) u = fma(th[o + 2 + j], xs[j], u);
        us[i] = u;
        xs[i + 1] = u * u;
        F = fma(th[o + 1], xs[i], F);
    }
    F = fma(th[oc + 1], xs[L], F);
    double out = F, fac = 1.0;
    if (target == FTSP2_TARGET_ENTROPY) {
        const double k4 = 4.0 * 0.69314718055994530942;
        out = k4 * F * (1.0 - F);
        fac = k4 * (1.0 - 2.0 * F);
    }
    const double r = out - target_value(target, x, beta0, mu0);
    R[s] = r;
    if (!WITH_J) return;
    const int np = oc + 2;
    M[(size_t)np * ns + s] = r;
    M[(size_t)oc * ns + s] = fac;
    M[(size_t)(oc + 1) * ns + s] = fac * xs[L];
    for (int j = 0; j < L; ++j) g[j] = th[j * (j + 5) / 2 + 1];
    g[L] = th[oc + 1];
    for (int i = L - 1; i >= 0; --i) {
        const int o = i * (i + 5) / 2;
        const double w = 2.0 * us[i] * g[i + 1];
        M[(size_t)o * ns + s] = fac * w;
        M[(size_t)(o + 1) * ns + s] = fac * xs[i];
        for (int j = 0; j <= i; ++j) {
            M[(size_t)(o + 2 + j) * ns + s] = fac * w * xs[j];
            g[j] = fma(w, th[o + 2 + j], g[j]);
        }
    }
}

cudaError_t launch_train_fwd_jac(int target, double beta0, double mu0, int L, double alpha, const ThetaParam& th,
                                 const double* dX, int ns, double* dR, double* dM, cudaStream_t s, int family) {
    if (family == FTSP2_FAMILY_MAX)
        fwd_max_kernel<true><<<(ns + 127) / 128, 128, 0, s>>>(target, beta0, mu0, L, alpha, th, dX, ns, dR, dM);
    else if (family == FTSP2_FAMILY_SKIP)
        fwd_skip_kernel<true><<<(ns + 127) / 128, 128, 0, s>>>(target, beta0, mu0, L, alpha, th, dX, ns, dR, dM);
    else fwd_kernel<true><<<(ns + 127) / 128, 128, 0, s>>>(target, beta0, mu0, L, alpha, th, dX, ns, dR, dM);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_train_residual(int target, double beta0, double mu0, int L, double alpha, const ThetaParam& th,
                                  const double* dX, int ns, double* dR, cudaStream_t s, int family) {
    if (family == FTSP2_FAMILY_MAX)
        fwd_max_kernel<false><<<(ns + 127) / 128, 128, 0, s>>>(target, beta0, mu0, L, alpha, th, dX, ns, dR,
                                                               nullptr);
    else if (family == FTSP2_FAMILY_SKIP)
        fwd_skip_kernel<false><<<(ns + 127) / 128, 128, 0, s>>>(target, beta0, mu0, L, alpha, th, dX, ns, dR,
                                                                nullptr);
    else fwd_kernel<false><<<(ns + 127) / 128, 128, 0, s>>>(target, beta0, mu0, L, alpha, th, dX, ns, dR, nullptr);
    count_launch();
    return cudaGetLastError();
}

// Gram matrix of the columns of M (m = np + 1 columns of ns samples): the
// samples in nchunks chunks, each entry of a chunk one FMA per sample in
// increasing order; gram_reduce sums the chunks in order.
//
// Bound by the FP64 pipe (two FMAs per clock and SM, a 64th of the FP32 rate),
// so the entries that are computed and the balance over the SMs decide.  A
// thread owns a 2 x 2 block of entries of the upper triangle (the blocks
// numbered row by row), a CTA of 64 threads 64 consecutive blocks of one chunk,
// with the samples' rows of M staged in shared memory (8-byte cp.async, two
// slices of S samples): at m = 65 the blocks hold 2244 entries for the 2145 of
// the triangle (32 x 32 tiles: 6144), in 576 CTAs, 3.8 per SM.  m = 65, 1e5
// samples: 1.60 ms with the tiles, 0.73 ms with single-buffered slices,
// 0.45 ms now (the FP64 pipe alone: 0.38).
constexpr int kGramThreads = 64;

// row pitch of the staged samples: even (16-byte pairs), half of it odd
static int gram_pitch(int m) {
    const int h = (m + 1) / 2;
    return 2 * (h + 1 - (h & 1));
}

template <int S>
__global__ void __launch_bounds__(kGramThreads) gram_partial_kernel(const double* __restrict__ M, int ns, int m,
                                                                    int chunk, int pitch, double* __restrict__ part) {
    extern __shared__ __align__(16) double gram_rows[];        // [2][S][pitch]
    const int s0 = blockIdx.y * chunk, s1 = min(ns, s0 + chunk);
    const int nb = (m + 1) / 2;
    // block (i, j), i <= j, of this thread
    int i = 0, j = blockIdx.x * kGramThreads + threadIdx.x;
    while (i < nb && j >= nb - i) {
        j -= nb - i;
        ++i;
    }
    const bool own = i < nb;
    j = own ? j + i : 0;
    if (!own) i = 0;
    // slice of samples sb .. sb + S - 1, zeros past the chunk and past the columns
    auto load = [&](int sb, int buf) {
        const uint32_t dst = smem_u32(gram_rows + buf * S * pitch);
        for (int e = threadIdx.x; e < S * 2 * nb; e += kGramThreads) {
            const int col = e / S, smp = e % S;
            const bool in = sb + smp < s1 && col < m;
            const double* src = in ? M + (size_t)col * ns + sb + smp : M;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst + 8u * (smp * pitch + col)), "l"(src),
                         "r"(in ? 8 : 0)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    double c00 = 0.0, c01 = 0.0, c10 = 0.0, c11 = 0.0;
    int buf = 0;
    if (s0 < s1) load(s0, 0);
    for (int sb = s0; sb < s1; sb += S) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                       // the slice is in, the other one read
        if (sb + S < s1) load(sb + S, buf ^ 1);
        if (own) {
            const double* const rows = gram_rows + buf * S * pitch;
#pragma unroll
            for (int k = 0; k < S; ++k) {
                const double2 x = *reinterpret_cast<const double2*>(rows + k * pitch + 2 * i);
                const double2 y = *reinterpret_cast<const double2*>(rows + k * pitch + 2 * j);
                c00 = fma(x.x, y.x, c00);
                c01 = fma(x.x, y.y, c01);
                c10 = fma(x.y, y.x, c10);
                c11 = fma(x.y, y.y, c11);
            }
        }
        buf ^= 1;
    }
    if (!own) return;
    double* const P = part + (size_t)blockIdx.y * m * m + (size_t)(2 * i) * m + 2 * j;
    const bool r1 = 2 * i + 1 < m, q1 = 2 * j + 1 < m;
    P[0] = c00;
    if (q1) P[1] = c01;
    if (r1 && i < j) P[m] = c10;
    if (r1 && q1) P[m + 1] = c11;
}

__global__ void gram_reduce_kernel(const double* __restrict__ part, int m, int nchunks, double* __restrict__ G) {
    const size_t mm = (size_t)m * m;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < mm; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / m), j = (int)(e % m);
        const double* p = part + (size_t)min(i, j) * m + max(i, j);        // the upper triangle was written
        double s = 0.0;
#pragma unroll 16
        for (int c = 0; c < nchunks; ++c) s += p[c * mm];
        G[e] = s;
    }
}

cudaError_t launch_train_gram(const double* dM, int ns, int np, double* dG, double* dScratch, int nchunks,
                              cudaStream_t s) {
    const int m = np + 1;
    const int nb = (m + 1) / 2, blocks = nb * (nb + 1) / 2;
    const int chunk = (ns + nchunks - 1) / nchunks;
    const int pitch = gram_pitch(m);
    const dim3 grid((blocks + kGramThreads - 1) / kGramThreads, nchunks);
    // two slices within the 48 KB a launch has without asking for more
    if (pitch <= 130)
        gram_partial_kernel<16><<<grid, kGramThreads, 2 * 16 * pitch * sizeof(double), s>>>(dM, ns, m, chunk, pitch,
                                                                                            dScratch);
    else
        gram_partial_kernel<8><<<grid, kGramThreads, 2 * 8 * pitch * sizeof(double), s>>>(dM, ns, m, chunk, pitch,
                                                                                          dScratch);
    gram_reduce_kernel<<<(m * m + 63) / 64, 64, 0, s>>>(dScratch, m, nchunks, dG);
    count_launch(2);
    return cudaGetLastError();
}

// out[j] = sum_s M[j][s] * w_s with w_s = (2/h) ((rh_s - r_s)/h - sum_j' J[j'][s] v[j'])
// (geodesic-acceleration right-hand side J^T r_vv), or with plain w = v-sum
// when rh == nullptr (J v).  One block per 256-sample chunk, then an ordered
// reduction over chunks.
// The second product takes its rows of M in slices of 16 samples (4 for wide
// tables) through shared memory (8-byte cp.async, two slices) instead of each
// thread along a column; the partial sums are staged the same way for the
// reduction, a chain of 391 dependent FP64 additions.  L = 16, 1e5 samples: 43 ->
// 37 us and 28 -> 18 us; the 2 x 64 FP64 products of a sample take 22.
template <int S>
__global__ void __launch_bounds__(256) accel_partial_kernel(const double* __restrict__ M, int ns, int np,
                                                            const double* __restrict__ v, const double* __restrict__ rh,
                                                            double h, double* __restrict__ part, int pitch) {
    extern __shared__ __align__(16) double acc_rows[];         // [2][S][pitch]
    __shared__ double w[256];
    const int base = blockIdx.x * 256, cnt = min(256, ns - base);
    const int s = base + threadIdx.x;
    auto load = [&](int k0, int buf) {
        const uint32_t dst = smem_u32(acc_rows + buf * S * pitch);
        for (int e = threadIdx.x; e < S * np; e += 256) {
            const int col = e / S, smp = e % S;
            if (k0 + smp < cnt)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + 8u * (smp * pitch + col)),
                             "l"(M + (size_t)col * ns + base + k0 + smp)
                             : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    double ws = 0.0;
    if (s < ns) {
        double jv = 0.0;
#pragma unroll 8
        for (int j = 0; j < np; ++j) jv = fma(M[(size_t)j * ns + s], v[j], jv);
        const double r = M[(size_t)np * ns + s];
        ws = (2.0 / h) * ((rh[s] - r) / h - jv);
    }
    w[threadIdx.x] = ws;
    load(0, 0);
    // columns of this thread: threadIdx.x, + 256, ...
    constexpr int kMaxCols = 2;
    double acc[kMaxCols];
#pragma unroll
    for (int q = 0; q < kMaxCols; ++q) acc[q] = 0.0;
    int buf = 0;
    for (int k0 = 0; k0 < cnt; k0 += S) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                       // the slice is in (and w), the other one read
        if (k0 + S < cnt) load(k0 + S, buf ^ 1);
        const double* const rows = acc_rows + buf * S * pitch;
        const int ke = min(S, cnt - k0);
#pragma unroll
        for (int q = 0; q < kMaxCols; ++q) {
            const int j = threadIdx.x + 256 * q;
            if (j >= np) break;
            for (int k = 0; k < ke; ++k) acc[q] = fma(rows[k * pitch + j], w[k0 + k], acc[q]);
        }
        buf ^= 1;
    }
#pragma unroll
    for (int q = 0; q < kMaxCols; ++q) {
        const int j = threadIdx.x + 256 * q;
        if (j < np) part[(size_t)blockIdx.x * np + j] = acc[q];
    }
}

constexpr int kAccelJ = 8, kAccelC = 512;

__global__ void __launch_bounds__(256) accel_reduce_kernel(const double* __restrict__ part, int nblk, int np,
                                                           double* __restrict__ out) {
    __shared__ double sm[kAccelC][kAccelJ];
    const int j0 = blockIdx.x * kAccelJ, jj = threadIdx.x % kAccelJ;
    double s = 0.0;
    for (int c0 = 0; c0 < nblk; c0 += kAccelC) {
        const int cn = min(kAccelC, nblk - c0);
        __syncthreads();
#pragma unroll 4
        for (int c = threadIdx.x / kAccelJ; c < cn; c += 256 / kAccelJ)
            if (j0 + jj < np) sm[c][jj] = part[(size_t)(c0 + c) * np + j0 + jj];
        __syncthreads();
        if (threadIdx.x < kAccelJ)
#pragma unroll 16
            for (int c = 0; c < cn; ++c) s += sm[c][jj];
    }
    if (threadIdx.x < kAccelJ && j0 + jj < np) out[j0 + jj] = s;
}

cudaError_t launch_train_accel(const double* dM, const double* dV, const double* dRh, double h, int ns, int np,
                               double* dPart, double* dOut, cudaStream_t s) {
    const int nblk = (ns + 255) / 256;
    const int pitch = np | 1;
    if (np > 512) return cudaErrorInvalidValue;              // two columns a thread; tables have at most 258
    // two slices and the 2 KB of w within the 48 KB a launch has without asking for more
    if (pitch <= 184)
        accel_partial_kernel<16><<<nblk, 256, 2 * 16 * pitch * sizeof(double), s>>>(dM, ns, np, dV, dRh, h, dPart,
                                                                                    pitch);
    else
        accel_partial_kernel<4><<<nblk, 256, 2 * 4 * pitch * sizeof(double), s>>>(dM, ns, np, dV, dRh, h, dPart,
                                                                                  pitch);
    accel_reduce_kernel<<<(np + kAccelJ - 1) / kAccelJ, 256, 0, s>>>(dPart, nblk, np, dOut);
    count_launch(2);
    return cudaGetLastError();
}

// max |r_s| over samples: per-block maxima, then one block.
__global__ void absmax_kernel(const double* __restrict__ r, int ns, double* __restrict__ part) {
    __shared__ double sm[256];
    double m = 0.0;
    for (int s = blockIdx.x * 256 + threadIdx.x; s < ns; s += gridDim.x * 256) m = fmax(m, fabs(r[s]));
    sm[threadIdx.x] = m;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sm[threadIdx.x] = fmax(sm[threadIdx.x], sm[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sm[0];
}

cudaError_t launch_train_absmax(const double* dR, int ns, double* dPart, double* dOut, cudaStream_t s) {
    absmax_kernel<<<64, 256, 0, s>>>(dR, ns, dPart);
    absmax_kernel<<<1, 256, 0, s>>>(dPart, 64, dOut);
    count_launch(2);
    return cudaGetLastError();
}

}  // namespace ftsp2
