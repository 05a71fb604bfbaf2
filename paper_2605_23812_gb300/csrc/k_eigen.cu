// k_eigen.cu -- the eigenvector ensemble of Sec. 3.3.2 (Eq. eigenvm1) on the device:
//   B = U Sigma U^T, U^T M_f U = I,  E = U_N Sigma_N^{1/2} sqrt(N - 1).
// On the uniform control cells M_f = dx dy I cancels, so E = V_N Lambda_N^{1/2} sqrt(N - 1) with
// (V, Lambda) the Euclidean eigenpairs of the one-component covariance B_s (Eq. covarianceB with
// c_xy = infinity) restricted to the control cells; both forcing components share B_s, so every
// eigenvector of B_s gives one fx and one fy member.
//
// B_s x = sigma^2 gather( K_y scatter(x) K_x ) with the 1-D Gaussian kernels K_x (nrx x nrx) and
// K_y (nry x nry) of the control rectangle: B_s is never formed.  Its leading eigenpairs come from
// Lanczos with full reorthogonalisation (two classical Gram-Schmidt passes per step).  Of the
// tridiagonal projection only the kept pairs are computed, one block each (k_tridiag_pairs); where
// two kept eigenvalues are too close for vectors computed apart, the whole projection is
// diagonalised by parallel cyclic Jacobi in one block.  The Ritz vectors are Q S.  All of this runs
// once per ensemble, before any forward run.
#include <algorithm>
#include <vector>

#include "envar_internal.cuh"

namespace envar {

// K[i][j] = exp(-((i - j) h)^2 / a^2)
__global__ void k_gauss_kernel(int n, double h, double a, double *__restrict__ K)
{
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= (long long)n * n) return;
    const int i = (int)(q / n), j = (int)(q % n);
    const double d = (i - j) * h;
    K[q] = exp(-d * d / (a * a));
}

// C[M x N] = A[M x K] B[K x N], row-major FP64, 16 x 16 shared-memory tiles.
__global__ void k_gemm_nn(int M, int N, int K, const double *__restrict__ A, const double *__restrict__ B,
                          double *__restrict__ C)
{
    __shared__ double sa[16][17], sb[16][17];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int row = blockIdx.y * 16 + ty, col = blockIdx.x * 16 + tx;
    double acc = 0.0;
    for (int k0 = 0; k0 < K; k0 += 16) {
        sa[ty][tx] = (row < M && k0 + tx < K) ? A[(long long)row * K + k0 + tx] : 0.0;
        sb[ty][tx] = (k0 + ty < K && col < N) ? B[(long long)(k0 + ty) * N + col] : 0.0;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; ++k) acc = fma(sa[ty][k], sb[k][tx], acc);
        __syncthreads();
    }
    if (row < M && col < N) C[(long long)row * N + col] = acc;
}

static void gemm_nn(int M, int N, int K, const double *A, const double *B, double *C, cudaStream_t st)
{
    dim3 blk(16, 16), grd(cdiv(N, 16), cdiv(M, 16));
    k_gemm_nn<<<grd, blk, 0, st>>>(M, N, K, A, B, C);
    count_launches(1);
}

// R[cidx[q]] = x[q], and imap = the compact index of a control cell of the rectangle (-1 elsewhere,
// set before).
__global__ void k_scatter_cc(int ncc, const int *__restrict__ cidx, const double *__restrict__ x,
                             double *__restrict__ R, int *__restrict__ imap)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < ncc) { R[cidx[q]] = x[q]; imap[cidx[q]] = q; }
}

// The kernels of a Lanczos step follow one another at 2 to 3 us each, so each is launched while its
// predecessor still runs (programmatic dependent launch) and waits for its completion, and thereby for all
// before it, ahead of its first access to memory: 7.3 ms -> 5.3 ms for 32 members at 256 x 128.
__device__ __forceinline__ void after_predecessor()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <class... P, class... A>
static void launch_after(void (*k)(P...), dim3 grid, int block, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t lc = {};
    lc.gridDim = grid;
    lc.blockDim = dim3(block);
    lc.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    cudaLaunchKernelEx(&lc, k, static_cast<P>(args)...);
    count_launches(1);
}

// The two products of one Lanczos step, C = A B (row-major FP64, M x K by K x N).  Both are small
// (104 x 32 with inner dimension 32 and 104 at 256 x 128), so time is the latency of one block's
// chain, not the flops: an 8 x 8 tile per block gives 52 blocks there, four threads share an output
// and take every fourth k, and 128 k of both operands are staged at once, eight loads in flight per
// thread.
// With imap the product goes to the compact vector, out[imap[e]] = scale C[e].
__global__ void __launch_bounds__(256) k_gemm_step(int M, int N, int K, const double *__restrict__ A,
                                                   const double *__restrict__ B, const int *__restrict__ imap,
                                                   double scale, double *__restrict__ out)
{
    after_predecessor();
    constexpr int KC = 128;
    __shared__ double sa[8][KC + 1], sb[KC][9], part[4][64];
    const int t = threadIdx.x, o = t & 63, s = t >> 6, r = o >> 3, c = o & 7;
    const int row0 = blockIdx.y * 8, col0 = blockIdx.x * 8;
    double acc = 0.0;
    for (int k0 = 0; k0 < K; k0 += KC) {
#pragma unroll
        for (int u = 0; u < 8 * KC / 256; ++u) {
            const int e = t + 256 * u;
            const int ar = e / KC, ak = e % KC, bk = e / 8, bc = e % 8;
            sa[ar][ak] = (row0 + ar < M && k0 + ak < K) ? A[(long long)(row0 + ar) * K + k0 + ak] : 0.0;
            sb[bk][bc] = (k0 + bk < K && col0 + bc < N) ? B[(long long)(k0 + bk) * N + col0 + bc] : 0.0;
        }
        __syncthreads();
        const int kn = min(KC, K - k0);
#pragma unroll 4
        for (int k = s; k < kn; k += 4) acc = fma(sa[r][k], sb[k][c], acc);
        __syncthreads();
    }
    part[s][o] = acc;
    __syncthreads();
    if (s == 0 && row0 + r < M && col0 + c < N) {
        const double v = (part[0][o] + part[1][o]) + (part[2][o] + part[3][o]);
        const int e = (row0 + r) * N + col0 + c;
        if (!imap) out[e] = v;
        else if (imap[e] >= 0) out[imap[e]] = scale * v;
    }
}

static void gemm_step(int M, int N, int K, const double *A, const double *B, const int *imap, double scale, double *out,
                      cudaStream_t st)
{
    launch_after(k_gemm_step, dim3(cdiv(N, 8), cdiv(M, 8)), 256, st, M, N, K, A, B, imap, scale, out);
}

// c[k] = Q_k . w for the rows k = 0 .. of Q ([rows][n]), one block each.
__global__ void k_dots(int n, const double *__restrict__ Q, const double *__restrict__ w, double *__restrict__ c)
{
    after_predecessor();
    const double *a = Q + (long long)blockIdx.x * n;
    double acc = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc = fma(a[i], w[i], acc);
    acc = block_reduce(acc, false);
    if (threadIdx.x == 0) c[blockIdx.x] = acc;
}

// w -= sum_k c[k] Q_k; part (if given) receives each block's sum of w^2.  One thread per cell walks
// the nq rows of Q one load behind another (26 us at 2873 cells and 72 rows: 12 blocks, latency); 32
// cells per block with eight threads per cell, each taking every eighth row, is 90 blocks of a chain of
// nine (6.9 us, launch included).
__global__ void __launch_bounds__(256) k_subtract(int n, int nq, const double *__restrict__ Q,
                                                  const double *__restrict__ c, double *__restrict__ w,
                                                  double *__restrict__ part)
{
    after_predecessor();
    __shared__ double sums[8][33];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    double v = 0.0;
    if (i < n) {
#pragma unroll 4
        for (int k = g; k < nq; k += 8) v = fma(c[k], Q[(long long)k * n + i], v);
    }
    sums[g][lane] = v;
    __syncthreads();
    if (g > 0) return;
    const double s = ((sums[0][lane] + sums[1][lane]) + (sums[2][lane] + sums[3][lane])) +
                     ((sums[4][lane] + sums[5][lane]) + (sums[6][lane] + sums[7][lane]));
    double r = 0.0;
    if (i < n) {
        r = w[i] - s;
        w[i] = r;
    }
    if (part) {
        r = warp_sum(r * r);
        if (lane == 0) part[blockIdx.x] = r;
    }
}

// beta = |w| from the blocks' sums; q_{j+1} = w / beta, also scattered into R for the next product;
// T[j][j] = c1[j] + c2[j]; T[j][j+1] = T[j+1][j] = beta.
__global__ void __launch_bounds__(256) k_lanczos_close(int n, int j, int m, int np, const double *__restrict__ part,
                                                       const double *__restrict__ c1, const double *__restrict__ c2,
                                                       const double *__restrict__ w, const int *__restrict__ cidx,
                                                       double *__restrict__ qnext, double *__restrict__ R,
                                                       double *__restrict__ T, double *__restrict__ beta_out)
{
    after_predecessor();
    double ww = 0.0;
    for (int b = threadIdx.x; b < np; b += blockDim.x) ww += part[b];
    const double beta = sqrt(block_reduce(ww, false));
    const double inv = (beta > 0.0) ? 1.0 / beta : 0.0;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const double q = w[i] * inv;
        qnext[i] = q;
        R[cidx[i]] = q;
    }
    if (i == 0) {
        T[(long long)j * m + j] = c1[j] + c2[j];
        if (j + 1 < m) {
            T[(long long)j * m + j + 1] = beta;
            T[(long long)(j + 1) * m + j] = beta;
        }
        beta_out[j] = beta;
    }
}

// The leading pairs of the symmetric tridiagonal T (order m, diagonal T[i][i] with row length mmax,
// off-diagonal beta[i]), one block per pair: lam[r] the r-th largest eigenvalue, Z[r][] its unit
// vector, bound[r] = beta[m-1] |Z[r][m-1]|, the residual of the Ritz pair.
//
// Eigenvalue: Givens' Sturm count with 128 points per pass, so the interval shrinks by 129 and eight
// passes reach rounding.  The determinants' recurrence p_i = (d_i - x) p_{i-1} - e_i^2 p_{i-2} is two
// dependent multiply-adds per row; its quotient form holds a division per row, five times the chain.
// The entries are scaled by a power of two to norm <= 2 and the pair (p_i, p_{i-1}) is rescaled every
// four rows, so nothing over- or underflows; e^2 is kept >= 2^-110 (2^-55 of the norm).
//
// Vector: D+ and D- of the factorisations from the top and from the bottom are the quotients of those
// pairs (two threads run the recurrences, all threads divide), and the vector grows from the row
// where |D+ + D- - (d - lam)| is smallest (Fernando's double factorisation), upwards and downwards at once.
//
// Time is the serial chain (eight counts and one factorisation: 0.23 ms at order 144); Jacobi on the whole
// projection in one block took 108 ms over orders 72 and 144, each of its rounds a pass over the matrix behind
// three barriers.  The ensemble of 32 members at 256 x 128, this and the shorter steps: 120.0 ms -> 7.3 ms.
__global__ void __launch_bounds__(128) k_tridiag_pairs(int m, int mmax, const double *__restrict__ T,
                                                       const double *__restrict__ beta, double *__restrict__ lam,
                                                       double *__restrict__ bound, double *__restrict__ Z)
{
    extern __shared__ double sh[];
    double *d = sh, *e = d + m, *e2 = e + m, *ap = e2 + m, *aq = ap + m, *bp = aq + m, *bq = bp + m;
    __shared__ double s_unit;
    __shared__ int s_tw;
    const int t = threadIdx.x, r = blockIdx.x;
    double lo = 0.0, hi = 0.0, big = 0.0;
    for (int i = t; i < m; i += 128) {
        const double off = (i > 0 ? beta[i - 1] : 0.0) + (i + 1 < m ? beta[i] : 0.0), di = T[(long long)i * mmax + i];
        d[i] = di;
        e[i] = (i > 0) ? beta[i - 1] : 0.0;                  // couples rows i - 1 and i
        big = fmax(big, fabs(di) + off);
    }
    big = block_reduce(big, true);
    if (t == 0) s_unit = (big > 0.0) ? ldexp(1.0, ilogb(big)) : 1.0;
    __syncthreads();
    const double unit = s_unit, inv = 1.0 / unit;
    for (int i = t; i < m; i += 128) {
        d[i] *= inv;
        e[i] *= inv;
        e2[i] = fmax(e[i] * e[i], 0x1p-110);
    }
    __syncthreads();
    auto rescale = [](double &p, double &q) {
        const int ex = max((max(__double2hiint(p) & 0x7fffffff, __double2hiint(q) & 0x7fffffff)) >> 20, 1);
        const double f = __hiloint2double((2046 - min(ex, 2045)) << 20, 0);
        p *= f;
        q *= f;
    };
    lo = -2.0; hi = 2.0;                                     // |T| <= 2 after the scaling
    for (int pass = 0; pass < 9 && hi - lo > 0x1p-54; ++pass) {
        const double step = (hi - lo) / 129.0, x = lo + step * (t + 1);
        double q = 1.0, p = d[0] - x;
        int neg = __double2hiint(p) < 0;                     // eigenvalues below x = sign changes of the sequence
        int i = 1;
        for (; i + 4 <= m; i += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const double n = fma(d[i + u] - x, p, -e2[i + u] * q);
                neg += (__double2hiint(n) ^ __double2hiint(p)) < 0;
                q = p;
                p = n;
            }
            rescale(p, q);
        }
        for (; i < m; ++i) {
            const double n = fma(d[i] - x, p, -e2[i] * q);
            neg += (__double2hiint(n) ^ __double2hiint(p)) < 0;
            q = p;
            p = n;
        }
        const int below = __syncthreads_count(neg <= m - 1 - r);   // points at or below the wanted eigenvalue
        hi = (below < 128) ? lo + step * (below + 1) : hi;
        lo = lo + step * below;
    }
    const double x = 0.5 * (lo + hi);
    // factorisations from both ends: the pairs whose quotients are D+ (a) and D- (b)
    if (t == 0 || t == 32) {
        const bool up = t != 0;
        double *sp = up ? bp : ap, *sq = up ? bq : aq;
        double q = 1.0, p = 1.0;
        for (int k = 0; k < m; ++k) {
            const int i = up ? m - 1 - k : k;
            const double off = up ? (k > 0 ? e2[i + 1] : 0.0) : (k > 0 ? e2[i] : 0.0);
            double n = (k > 0) ? fma(d[i] - x, p, -off * q) : d[i] - x;
            if (fabs(n) < 0x1p-60 * fabs(p)) n = 0x1p-60 * fabs(p);   // a pivot of rounding size
            sp[i] = n;
            sq[i] = p;
            q = p;
            p = n;
            rescale(p, q);
        }
    }
    __syncthreads();
    double best = HUGE_VAL;
    int at = 0;
    for (int i = t; i < m; i += 128) {
        const double dp = ap[i] / aq[i], dm = bp[i] / bq[i];
        const double g = fabs(dp + dm - (d[i] - x));
        if (g < best) { best = g; at = i; }
        ap[i] = -(i + 1 < m ? e[i + 1] : 0.0) / dp;          // z_i = ap_i z_{i+1} above the twist
        bp[i] = -e[i] / dm;                                  // z_i = bp_i z_{i-1} below it
    }
    const double mine = (best < HUGE_VAL) ? -best / (1.0 + best) : -1.0;   // the reduction's maximum starts at -1
    const double least = block_reduce(mine, true);
    if (t == 0) s_tw = m;
    __syncthreads();
    if (mine == least) atomicMin(&s_tw, at);
    __syncthreads();
    const int tw = min(s_tw, m - 1);
    if (t == 0) {
        double z = 1.0;
        aq[tw] = 1.0;
        for (int i = tw - 1; i >= 0; --i) { z *= ap[i]; aq[i] = z; }
    } else if (t == 32) {
        double z = 1.0;
        for (int i = tw + 1; i < m; ++i) { z *= bp[i]; aq[i] = z; }
    }
    __syncthreads();
    double nn = 0.0;
    for (int i = t; i < m; i += 128) nn = fma(aq[i], aq[i], nn);
    nn = 1.0 / sqrt(block_reduce(nn, false));
    for (int i = t; i < m; i += 128) Z[(long long)r * m + i] = nn * aq[i];
    if (t == 0) {
        lam[r] = x * unit;
        bound[r] = fabs(beta[m - 1] * (nn * aq[m - 1]));
    }
}

// W = Z - (Z Z^T - I) Z / 2: vectors computed apart deviate from orthogonality by rounding over the gap
// of their eigenvalues; the first-order symmetric orthogonalisation leaves the square of that.  Block r
// makes row r.
__global__ void __launch_bounds__(256) k_orthogonalise(int m, int k, const double *__restrict__ Z, double *__restrict__ W)
{
    extern __shared__ double g[];                            // row r of Z Z^T - I
    const int r = blockIdx.x, lane = threadIdx.x & 31;
    for (int s = threadIdx.x >> 5; s < k; s += 8) {
        double a = 0.0;
        for (int i = lane; i < m; i += 32) a = fma(Z[(long long)r * m + i], Z[(long long)s * m + i], a);
        a = warp_sum(a);
        if (lane == 0) g[s] = a - (s == r ? 1.0 : 0.0);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += 256) {
        double a = 0.0;
        for (int s = 0; s < k; ++s) a = fma(g[s], Z[(long long)s * m + i], a);
        W[(long long)r * m + i] = Z[(long long)r * m + i] - 0.5 * a;
    }
}

__global__ void k_normalize(int n, double *__restrict__ q)
{
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc += q[i] * q[i];
    acc = block_reduce(acc, false);
    const double inv = 1.0 / sqrt(acc);
    for (int i = threadIdx.x; i < n; i += blockDim.x) q[i] *= inv;
}

// Parallel cyclic Jacobi on the symmetric m x m matrix A (m even; row-major, in place) with the
// circle ordering: in round r of a sweep, element m-1 meets r and element (r + k) meets (r - k),
// both mod m-1, so the m/2 rotations of a round act on disjoint index pairs.  V accumulates the
// rotations (A_in = V diag(A_out) V^T).  Stops when the off-diagonal Frobenius norm falls below
// tol times the full norm, or after max_sweeps sweeps; *sweeps_out receives the sweeps used.
__global__ void __launch_bounds__(1024) k_jacobi(int m, double *__restrict__ A, double *__restrict__ V, double tol,
                                                 int max_sweeps, int *sweeps_out)
{
    extern __shared__ double sh[];   // c[m/2], s[m/2], then pairs p[m/2], q[m/2] as ints
    double *cs = sh, *sn = sh + m / 2;
    int *pp = reinterpret_cast<int *>(sn + m / 2), *qq = pp + m / 2;
    const int tid = threadIdx.x, nt = blockDim.x, h = m / 2;
    for (long long e = tid; e < (long long)m * m; e += nt) V[e] = ((e / m) == (e % m)) ? 1.0 : 0.0;
    __syncthreads();
    int sweep = 0;
    for (; sweep < max_sweeps; ++sweep) {
        double off = 0.0, all = 0.0;
        for (long long e = tid; e < (long long)m * m; e += nt) {
            const double a = A[e];
            all += a * a;
            if ((e / m) != (e % m)) off += a * a;
        }
        off = block_reduce(off, false);
        all = block_reduce(all, false);
        if (off <= tol * tol * all) break;
        for (int r = 0; r < m - 1; ++r) {
            for (int k = tid; k < h; k += nt) {
                int p, q;
                if (k == 0) { p = r; q = m - 1; }
                else { p = (r + k) % (m - 1); q = (r - k + (m - 1)) % (m - 1); }
                if (p > q) { const int t = p; p = q; q = t; }
                const double apq = A[(long long)p * m + q];
                double c = 1.0, s = 0.0;
                if (apq != 0.0) {
                    const double tau = (A[(long long)q * m + q] - A[(long long)p * m + p]) / (2.0 * apq);
                    const double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
                    c = 1.0 / sqrt(1.0 + t * t);
                    s = t * c;
                }
                cs[k] = c; sn[k] = s; pp[k] = p; qq[k] = q;
            }
            __syncthreads();
            // rows: A <- J^T A
            for (long long e = tid; e < (long long)h * m; e += nt) {
                const int k = (int)(e / m), j = (int)(e % m);
                const int p = pp[k], q = qq[k];
                const double c = cs[k], s = sn[k];
                const double ap = A[(long long)p * m + j], aq = A[(long long)q * m + j];
                A[(long long)p * m + j] = c * ap - s * aq;
                A[(long long)q * m + j] = s * ap + c * aq;
            }
            __syncthreads();
            // columns: A <- A J, V <- V J
            for (long long e = tid; e < (long long)h * m; e += nt) {
                const int k = (int)(e / m), i = (int)(e % m);
                const int p = pp[k], q = qq[k];
                const double c = cs[k], s = sn[k];
                const double ap = A[(long long)i * m + p], aq = A[(long long)i * m + q];
                A[(long long)i * m + p] = c * ap - s * aq;
                A[(long long)i * m + q] = s * ap + c * aq;
                const double vp = V[(long long)i * m + p], vq = V[(long long)i * m + q];
                V[(long long)i * m + p] = c * vp - s * vq;
                V[(long long)i * m + q] = s * vp + c * vq;
            }
            __syncthreads();
        }
    }
    if (tid == 0) *sweeps_out = sweep;
}

// Indices of the k largest diagonal entries of A (m x m), in decreasing order (one thread; m small).
__global__ void k_top_diag(int m, int k, const double *__restrict__ A, int *__restrict__ idx, double *__restrict__ lam)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    for (int r = 0; r < k; ++r) {
        int best = -1;
        for (int i = 0; i < m; ++i) {
            bool used = false;
            for (int t = 0; t < r; ++t) used |= (idx[t] == i);
            if (used) continue;
            if (best < 0 || A[(long long)i * m + i] > A[(long long)best * m + best]) best = i;
        }
        idx[r] = best;
        lam[r] = A[(long long)best * m + best];
    }
}

// Sk[r][j] = S[j][idx[r]]: the eigenvector coefficients of the k kept Ritz pairs, as rows.
__global__ void k_gather_ritz(int m, int k, const double *__restrict__ S, const int *__restrict__ idx,
                              double *__restrict__ Sk)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m * k) return;
    const int r = e / m, j = e % m;
    Sk[e] = S[(long long)j * m + idx[r]];
}

// Ritz vector r (row r of v = Sk Q): normalised, sign so that its largest-magnitude entry is
// positive, scaled by sqrt(lambda_r (N-1)); written as members 2r (fx) and 2r+1 (fy) of E
// (n_ctrl x N column-major, zero elsewhere), when those members exist, or, with y_only, as the fy
// member r.  One block per r.
__global__ void k_ritz_members(int n, int N, int y_only, const double *__restrict__ lam, const double *__restrict__ v,
                               double *__restrict__ E)
{
    const int r = blockIdx.x;
    const double *vr = v + (long long)r * n;
    double nrm = 0.0, amax = -1.0;
    int imax = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double a = vr[i];
        nrm += a * a;
        if (fabs(a) > amax) { amax = fabs(a); imax = i; }
    }
    nrm = block_reduce(nrm, false);
    // arg-max |v| (ties: lowest index) through the shared-memory reduction of block_reduce's layout
    __shared__ double s_val[1024];
    __shared__ int s_idx[1024];
    s_val[threadIdx.x] = amax;
    s_idx[threadIdx.x] = imax;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            const double a = s_val[threadIdx.x + o];
            const int ia = s_idx[threadIdx.x + o];
            if (a > s_val[threadIdx.x] || (a == s_val[threadIdx.x] && ia < s_idx[threadIdx.x])) {
                s_val[threadIdx.x] = a;
                s_idx[threadIdx.x] = ia;
            }
        }
        __syncthreads();
    }
    const double sgn = (vr[s_idx[0]] < 0.0) ? -1.0 : 1.0;
    const double scale = sgn * sqrt(fmax(lam[r], 0.0) * (double)(N - 1)) / sqrt(nrm);
    const long long nctrl = 2LL * n;
    for (int comp = y_only ? 1 : 0; comp < 2; ++comp) {
        const int k = y_only ? r : 2 * r + comp;
        if (k >= N) break;
        double *Ek = E + (long long)k * nctrl;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            Ek[(long long)comp * n + i] = scale * vr[i];
            Ek[(long long)(1 - comp) * n + i] = 0.0;
        }
    }
}

// Residual of the k kept Ritz pairs after m Lanczos steps: |B v_r - theta_r v_r| =
// beta_m |S[m-1][idx_r]| (exact in exact arithmetic; with full reorthogonalisation a faithful
// estimate).
__global__ void k_ritz_bounds(int m, int k, const double *__restrict__ S, const int *__restrict__ idx,
                              const double *__restrict__ beta, double *__restrict__ bound)
{
    for (int r = threadIdx.x; r < k; r += blockDim.x) bound[r] = fabs(beta[m - 1] * S[(long long)(m - 1) * m + idx[r]]);
}

// copy the leading m x m block of T (stored with row length mmax) to A (row length m)
__global__ void k_copy_block(int m, int mmax, const double *__restrict__ T, double *__restrict__ A)
{
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e < (long long)m * m) A[e] = T[(e / m) * mmax + (e % m)];
}

size_t eigen_work_doubles(int nrx, int nry, int ncc, int mmax, int k)
{
    return (size_t)nrx * nrx + (size_t)nry * nry + 2 * (size_t)nrx * nry + (size_t)(mmax + 1) * ncc + ncc +
           2 * (size_t)(mmax + 2) + 3 * (size_t)mmax * mmax + mmax + 2 * (size_t)k + (size_t)k * ncc +
           2 * (size_t)k * mmax + (size_t)k + ((size_t)nrx * nry + 1) / 2 + cdiv(ncc, 32) + 8;
}

// Leading k eigenpairs of B_s by Lanczos; writes the N members of E (compact, column-major).  The
// Lanczos basis grows from m0 steps, doubling up to mmax (<= ncc), until every kept Ritz pair's
// residual bound is below tol times the largest eigenvalue.  work: eigen_work_doubles(..., mmax, k)
// doubles.  Host outputs (nullable): the k eigenvalues, the steps used, the largest bound.
int eigen_ensemble(int nrx, int nry, double dx, double dy, double a, double sigma, int ncc, const int *cidx, int N,
                   int y_only, int m0, int mmax, double tol, unsigned long long seed, double *work, double *E,
                   double *lam_host, int *steps_host, double *bound_host, cudaStream_t st)
{
    const int k = y_only ? N : (N + 1) / 2;
    mmax -= mmax % 2;
    m0 = std::min(m0 - m0 % 2, mmax);
    if (m0 < 2 || k > m0) return -1;
    double *p = work;
    double *Kx = p; p += (size_t)nrx * nrx;
    double *Ky = p; p += (size_t)nry * nry;
    double *R = p; p += (size_t)nrx * nry;
    double *T1 = p; p += (size_t)nrx * nry;
    double *Q = p; p += (size_t)(mmax + 1) * ncc;
    double *w = p; p += ncc;
    double *c1 = p; p += mmax + 2;
    double *c2 = p; p += mmax + 2;
    double *T = p; p += (size_t)mmax * mmax;
    double *A = p; p += (size_t)mmax * mmax;
    double *V = p; p += (size_t)mmax * mmax;
    double *beta = p; p += mmax;
    double *lam = p; p += k;
    double *bound = p; p += k;
    double *vr = p; p += (size_t)k * ncc;
    double *Sk = p; p += (size_t)k * mmax;
    double *Z = p; p += (size_t)k * mmax;
    const int np = cdiv(ncc, 32);
    double *part = p; p += np;
    int *idx = reinterpret_cast<int *>(p); p += k;
    int *imap = reinterpret_cast<int *>(p); p += ((size_t)nrx * nry + 1) / 2;
    int *sweeps = reinterpret_cast<int *>(p);

    k_gauss_kernel<<<cdiv(nrx * nrx, 256), 256, 0, st>>>(nrx, dx, a, Kx);
    k_gauss_kernel<<<cdiv(nry * nry, 256), 256, 0, st>>>(nry, dy, a, Ky);
    count_launches(2);
    cudaMemsetAsync(T, 0, sizeof(double) * (size_t)mmax * mmax, st);
    launch_normals(seed, 7ULL, 0LL, ncc, Q, st);   // seeded start vector
    k_normalize<<<1, 1024, 0, st>>>(ncc, Q);
    count_launches(1);
    const int gb = cdiv(ncc, 256);
    cudaMemsetAsync(R, 0, sizeof(double) * (size_t)nrx * nry, st);
    cudaMemsetAsync(imap, 0xff, sizeof(int) * (size_t)nrx * nry, st);
    k_scatter_cc<<<gb, 256, 0, st>>>(ncc, cidx, Q, R, imap);
    count_launches(1);
    int done = 0, m = m0;
    std::vector<double> hl(2 * (size_t)k);                   // eigenvalues and bounds of the kept pairs
    double worst = 0.0;
    for (;;) {
        for (int j = done; j < m; ++j) {
            // w = B_s q_j (R holds q_j on the rectangle)
            gemm_step(nry, nrx, nry, Ky, R, nullptr, 1.0, T1, st);
            gemm_step(nry, nrx, nrx, T1, Kx, imap, sigma * sigma, w, st);
            // two Gram-Schmidt passes against q_0 .. q_j, then |w|^2 by blocks
            launch_after(k_dots, dim3(j + 1), 256, st, ncc, Q, w, c1);
            launch_after(k_subtract, dim3(np), 256, st, ncc, j + 1, Q, c1, w, nullptr);
            launch_after(k_dots, dim3(j + 1), 256, st, ncc, Q, w, c2);
            launch_after(k_subtract, dim3(np), 256, st, ncc, j + 1, Q, c2, w, part);
            launch_after(k_lanczos_close, dim3(gb), 256, st, ncc, j, mmax, np, part, c1, c2, w, cidx, Q + (size_t)(j + 1) * ncc, R, T, beta);
        }
        done = m;
        const size_t smem = sizeof(double) * 7 * m;
        k_tridiag_pairs<<<k, 128, smem, st>>>(m, mmax, T, beta, lam, bound, Z);
        k_orthogonalise<<<k, 256, sizeof(double) * k, st>>>(m, k, Z, Sk);
        count_launches(2);
        cudaMemcpyAsync(hl.data(), lam, sizeof(double) * 2 * k, cudaMemcpyDeviceToHost, st);
        cudaStreamSynchronize(st);
        // vectors computed apart mix by rounding / gap; below 1e-7 of the largest eigenvalue the projection is
        // diagonalised as a whole (exactly degenerate pairs too: a square control set)
        bool close = false;
        for (int r = 1; r < k; ++r) close |= !(hl[r - 1] - hl[r] >= 1e-7 * hl[0]);
        if (close) {
            k_copy_block<<<cdiv(m * m, 256), 256, 0, st>>>(m, mmax, T, A);
            k_jacobi<<<1, 1024, (sizeof(double) + sizeof(int)) * m, st>>>(m, A, V, 1e-15, 60, sweeps);
            k_top_diag<<<1, 32, 0, st>>>(m, k, A, idx, lam);
            k_ritz_bounds<<<1, 256, 0, st>>>(m, k, V, idx, beta, bound);
            k_gather_ritz<<<cdiv(m * k, 256), 256, 0, st>>>(m, k, V, idx, Sk);
            count_launches(5);
            cudaMemcpyAsync(hl.data(), lam, sizeof(double) * 2 * k, cudaMemcpyDeviceToHost, st);
            cudaStreamSynchronize(st);
        }
        worst = 0.0;
        for (int r = 0; r < k; ++r) worst = std::max(worst, hl[k + r] / std::max(hl[0], 1e-300));
        if (worst <= tol || m >= mmax) break;
        m = std::min(2 * m, mmax);
    }
    gemm_nn(k, ncc, m, Sk, Q, vr, st);
    k_ritz_members<<<k, 1024, 0, st>>>(ncc, N, y_only, lam, vr, E);
    count_launches(1);
    if (lam_host) cudaMemcpyAsync(lam_host, lam, sizeof(double) * k, cudaMemcpyDeviceToHost, st);
    if (steps_host) *steps_host = m;
    if (bound_host) *bound_host = worst;
    return 0;
}

} // namespace envar
