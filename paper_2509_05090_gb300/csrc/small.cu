// Bandwidth- and latency-bound kernels of the CTMRG step: C3v projection and
// double layer (Sec. II.A, App. A, Fig. 1b), environment initialisation,
// warm start of the reduced corner, corner re-symmetrisation and
// normalisation (Fig. 3a), edge normalisation, the corner-spectrum
// convergence test, and the final bond-energy contraction (Eq. 1, Eq. 4).
// All FP64.
#include <math.h>

#include <atomic>
#include <cooperative_groups.h>
#include <mutex>

#include "ctm_internal.h"
#include "fp64_chain.h"

namespace {

__device__ __forceinline__ double block_sum(double v, double *red)
{
    // block-wide reduction (any block size up to 1024; red: >= 32 doubles): warp
    // sums, then warp 0 reduces the per-warp sums with shuffles -- short FP64 chains
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double s = (lane < nw) ? red[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) red[32] = s;
    }
    __syncthreads();
    return red[32];
}

// a0: A_sym = (1/6) sum over the six permutations of the virtual legs, then
// unit Frobenius norm.  One CTA; the tensor is at most a few thousand entries.
__global__ void c3v_project_kernel(int d, int D, const double *Ain, double *Aout, int symmetrize)
{
    extern __shared__ double sA[];
    __shared__ double red[33];
    const int D3 = D * D * D, tot = d * D3;
    for (int t = threadIdx.x; t < tot; t += blockDim.x) {
        int s = t / D3, r = t % D3;
        int i = r / (D * D), j = (r / D) % D, k = r % D;
        const double *As = Ain + (size_t)s * D3;
        double v;
        if (symmetrize)
            v = (As[(i * D + j) * D + k] + As[(i * D + k) * D + j] + As[(j * D + i) * D + k] +
                 As[(j * D + k) * D + i] + As[(k * D + i) * D + j] + As[(k * D + j) * D + i]) / 6.0;
        else
            v = As[r];
        sA[t] = v;
    }
    __syncthreads();
    double ss = 0.0;
    for (int t = threadIdx.x; t < tot; t += blockDim.x) ss += sA[t] * sA[t];
    ss = block_sum(ss, red);
    double f = (symmetrize && ss > 0.0) ? 1.0 / sqrt(ss) : 1.0;
    for (int t = threadIdx.x; t < tot; t += blockDim.x) Aout[t] = sA[t] * f;
}

// a1: a[(ii')][(jj')][(kk')] = sum_s K[s,i,j,k] B[s,i',j',k'].
__global__ void double_layer_kernel(int d, int D, const double *K, const double *B, double *a)
{
    const int D2 = D * D, D3 = D * D * D;
    const long long tot = (long long)D2 * D2 * D2;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x) {
        int u = (int)(t / (D2 * D2)), v = (int)((t / D2) % D2), w = (int)(t % D2);
        int i = u / D, i2 = u % D, j = v / D, j2 = v % D, k = w / D, k2 = w % D;
        double s = 0.0;
        for (int p = 0; p < d; ++p)
            s = fma(K[(size_t)p * D3 + (i * D + j) * D + k], B[(size_t)p * D3 + (i2 * D + j2) * D + k2], s);
        a[t] = s;
    }
}

// Open layers for the bond-energy contraction: b[(s,t)][u][v][w] = A[s]... (x) A[t]...
__global__ void open_layers_kernel(int d, int D, const double *A, double *b)
{
    const int D2 = D * D, D3 = D * D * D;
    const long long per = (long long)D2 * D2 * D2;
    const long long tot = per * d * d;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
         t += (long long)gridDim.x * blockDim.x) {
        int p = (int)(t / per);
        long long r = t - p * per;
        int s = p / d, q = p % d;
        int u = (int)(r / (D2 * D2)), v = (int)((r / D2) % D2), w = (int)(r % D2);
        int i = u / D, i2 = u % D, j = v / D, j2 = v % D, k = w / D, k2 = w % D;
        b[t] = A[(size_t)s * D3 + (i * D + j) * D + k] * A[(size_t)q * D3 + (i2 * D + j2) * D + k2];
    }
}

// Initial environment: C = I, T[a][u][b] = delta_ab t_u, t_u = sum_{v,w} a[u][(vv)][(ww)],
// Q = first chi columns of I_n.
__global__ void init_env_kernel(int chi, int D, const double *a, double *C, double *T, double *Q)
{
    const int D2 = D * D;
    const long long n = (long long)chi * D2;
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long t = tid; t < (long long)chi * chi; t += stride) C[t] = ((t / chi) == (t % chi)) ? 1.0 : 0.0;
    for (long long t = tid; t < n * chi; t += stride) Q[t] = ((t / chi) == (t % chi)) ? 1.0 : 0.0;
    for (long long t = tid; t < (long long)chi * D2 * chi; t += stride) {
        int al = (int)(t / ((long long)D2 * chi));
        int u = (int)((t / chi) % D2);
        int be = (int)(t % chi);
        double v = 0.0;
        if (al == be)
            for (int p = 0; p < D; ++p)
                for (int q = 0; q < D; ++q) v += a[((size_t)u * D2 + p * D + p) * D2 + q * D + q];
        T[t] = v;
    }
}

// Reduced-corner warm start: Qs = Q diag(sgn C_jj), sgn(0) = +1.
__global__ void warm_start_kernel(long long n, int chi, const double *Q, const double *C, double *Qs)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n * chi;
         t += (long long)gridDim.x * blockDim.x) {
        int j = (int)(t % chi);
        double v = Q[t];
        Qs[t] = (C[(size_t)j * chi + j] < 0.0) ? -v : v;
    }
}

// Y = M Q S where Q is the first chi columns of I_n (M n x n row-major).
__global__ void select_columns_kernel(long long n, int chi, const double *M, const double *C, double *Y)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n * chi;
         t += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(t % chi);
        const double v = M[(t / chi) * n + j];
        Y[t] = (C[(size_t)j * chi + j] < 0.0) ? -v : v;
    }
}

// a5 tail: C' = (Cr + Cr^T)/2, then unit Frobenius norm, over several blocks (the FP64 work of one SM would
// bind): partial sums of squares, then every block derives the factor from the
// partials with one warp and scales its share.
__global__ void corner_sym_sumsq_kernel(int chi, const double *Cr, double *partials)
{
    __shared__ double red[33];
    double ss = 0.0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < chi * chi; t += gridDim.x * blockDim.x) {
        const int i = t / chi, j = t - i * chi;
        const double v = 0.5 * (Cr[t] + Cr[(size_t)j * chi + i]);
        ss = fma(v, v, ss);
    }
    ss = block_sum(ss, red);
    if (threadIdx.x == 0) partials[blockIdx.x] = ss;
}
__global__ void corner_sym_scale_kernel(int chi, const double *Cr, const double *partials, int np, double *Cn)
{
    __shared__ double f;
    if (threadIdx.x < 32) {
        double s = 0.0;
        for (int i = threadIdx.x; i < np; i += 32) s += partials[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) f = s > 0.0 ? 1.0 / sqrt(s) : 1.0;
    }
    __syncthreads();
    const double h = 0.5 * f;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < chi * chi; t += gridDim.x * blockDim.x) {
        const int i = t / chi, j = t - i * chi;
        Cn[t] = (Cr[t] + Cr[(size_t)j * chi + i]) * h;
    }
}

// Frobenius normalisation of a large array: per-block partial sums of squares...
__global__ void sumsq_partial_kernel(long long count, const double *x, double *partials)
{
    __shared__ double red[33];
    double s = 0.0;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
         t += (long long)gridDim.x * blockDim.x)
        s = fma(x[t], x[t], s);
    s = block_sum(s, red);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

// ... then every block re-sums the partials in the same order and scales its share.
__global__ void scale_by_partials_kernel(long long count, double *x, const double *partials, int np)
{
    __shared__ double f;
    if (threadIdx.x < 32) {   // one warp sums the partials: short chains, then shuffles
        double s = 0.0;
        for (int i = threadIdx.x; i < np; i += 32) s += partials[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) f = s > 0.0 ? 1.0 / sqrt(s) : 1.0;
    }
    __syncthreads();
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
         t += (long long)gridDim.x * blockDim.x)
        x[t] *= f;
}

// a7: corner spectrum and delta, in three launches.
// (1) Householder tridiagonalisation of the symmetric corner -> diagonal d and squared
//     off-diagonal e^2 (global work buffer): one CTA with the corner in shared memory
//     below TRI_CLUSTER_MIN, a thread-block cluster holding it by rows from there;
// (2) one warp per eigenvalue: multisection on [-|C|_F, |C|_F], each
//     lane evaluating the Sturm count at one of 32 points per round
//     (5 bits per round instead of 1).  The count is the number of sign
//     changes of p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2}, kept in range by
//     exact power-of-two rescaling -- no division on the dependent chain;
// (3) one CTA: |lambda| sorted descending by rank, unit 2-norm, delta.
constexpr int TRI_THREADS = 256;
constexpr size_t SPEC_SM_ALONE_BYTES = 220 * 1024;   // within the 224 KB opt-in of spectrum_prepare
constexpr int TRI_FULL_MAX = 160;   // the full corner in shared memory up to here, its lower triangle beyond
constexpr int TRI_SMEM_MAX = 224;   // the lower triangle of a 224 x 224 corner: 197 KB of shared memory
constexpr int SPEC_MAX_CHI = 512;   // beyond TRI_SMEM_MAX the lower triangle lives in the work buffer (L2)
// From here up the reduction runs over a thread-block cluster where the device schedules one
// (its per-column cost hardly depends on chi, so it overtakes the one-CTA kernels early;
// the benchmark's chi = 72 and the batch's instances keep the one-CTA kernel)
constexpr int TRI_CLUSTER_MIN = 97;

// offset (doubles) of the global lower triangle in the spectrum's work buffer, after
// d, e^2 (2 chi) and the eigenvalues (chi)
__host__ __device__ inline size_t tri_global_off(int chi) { return (size_t)3 * chi + 8; }

// One CTA, chi <= TRI_FULL_MAX.  Bound by FP64 issue (one warp instruction per 64 cycles and
// sub-partition: m^2 multiply-adds for the mat-vec and as many for the update, lower
// triangle only) and by the serial chain per column, which is kept to one reduction and one
// pair of Householder scalars:
//   y = A x (x: the column below the diagonal), s2 = x^T y;  with v = x - alpha e_0 and
//   p = beta A v = beta (y - alpha A e_0) the inner product p^T v is
//   beta (s2 - 2 alpha y_0 + alpha^2 A_00), so nothing waits for a second reduction;
//   with K = beta/2 p^T v and g = p - 2 K v the update is A_ij -= v_i p_j + g_i v_j.
// Per column three barriers: A (y is complete, and the scalar warp's alpha and beta), B (p, v
// and K), C (the next x).  The last warp works one column ahead: after B it updates the next
// column itself (the workers leave it out), hands it over at C without waiting, and forms
// |x|^2, alpha and beta while the others update and multiply.  A column already reduced has
// beta = 0, alpha = x_0 and an update of zero.  chi = 72: 391 -> 211 us alone.
constexpr int TRI_WARPS = 9;   // eight workers, two per sub-partition (four lanes per row, eight per row pair), one scalar warp
__host__ __device__ inline int tri_pitch(int chi) { return chi + ((20 - chi % 16) % 16); }   // = 4 mod 16: conflict-free rows and columns
__host__ __device__ inline size_t tri_full_smem_bytes(int chi)
{
    return sizeof(double) * ((size_t)chi * tri_pitch(chi) + 5 * (size_t)chi);
}
__device__ __forceinline__ void cta_sync() { asm volatile("bar.sync 0;" ::: "memory"); }
__device__ __forceinline__ void next_x_sync(int threads) { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); }
__device__ __forceinline__ void next_x_arrive(int threads)
{
    __threadfence_block();
    asm volatile("bar.arrive 1, %0;" ::"r"(threads) : "memory");
}

// alpha and beta of column x (m entries) for the kernels below: s1 = sum_{i >= 1} x_i^2
__device__ __forceinline__ void tri_scalars(double s1, double x0, double *alpha, double *beta)
{
    if (s1 == 0.0) {   // already reduced
        *alpha = x0;
        *beta = 0.0;
        return;
    }
    const HouseholderScalars h = householder_scalars(fma(x0, x0, s1), fabs(x0));
    *alpha = (x0 >= 0.0) ? -h.nrm : h.nrm;
    *beta = h.beta;
}

__global__ void __launch_bounds__(32 * TRI_WARPS) tridiag_kernel(int chi, const double *C, double *work)
{
    extern __shared__ double sm[];
    __shared__ double sh_alpha, sh_beta, sh_K;
    const int ld = tri_pitch(chi);
    double *A = sm;                                // chi x ld, lower triangle
    double *xb = A + (size_t)chi * ld;             // 2 x chi: the column, by parity
    double *y = xb + 2 * chi, *p = y + chi, *v = p + chi;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nthr = blockDim.x, nwork = nthr - 32;
    for (int t = tid; t < chi * chi; t += nthr) {
        const int i = t / chi, j = t % chi;
        if (j <= i) A[i * ld + j] = 0.5 * (C[t] + C[(size_t)j * chi + i]);
    }
    __syncthreads();
    if (tid >= nwork) {
        // ------------------------------------------------ scalar warp
        // column 0, then per reduced column the next one
        for (int i = lane; i + 1 < chi; i += 32) xb[i] = A[(i + 1) * ld];
        if (lane == 0) work[0] = A[0];
        __syncwarp();
        next_x_arrive(nthr);
        for (int kc = 0; kc + 1 < chi; ++kc) {
            const double *x = xb + (kc & 1) * chi;
            const int m = chi - kc - 1;
            double s1 = 0.0;
            for (int i = 1 + lane; i < m; i += 32) s1 = fma(x[i], x[i], s1);
            s1 = warp_sum(s1);
            double alpha, beta;
            tri_scalars(s1, x[0], &alpha, &beta);
            if (lane == 0) {
                sh_alpha = alpha;
                sh_beta = beta;
                work[chi + kc] = alpha * alpha;
            }
            if (kc + 2 >= chi) break;
            cta_sync();   // A
            cta_sync();   // B
            const int b0 = kc + 1;
            const double K2 = 2.0 * sh_K, p0 = p[0], v0 = v[0];
            double *xn = xb + ((kc + 1) & 1) * chi;
            for (int i = lane; i < m; i += 32) {
                const double vi = v[i], a = A[(b0 + i) * ld + b0];
                const double w = fma(-fma(-K2, vi, p[i]), v0, fma(-vi, p0, a));
                if (i == 0) work[b0] = w;
                else xn[i - 1] = w;
            }
            __syncwarp();
            next_x_arrive(nthr);
        }
        if (lane == 0) work[2 * chi - 1] = 0.0;
        return;
    }
    next_x_sync(nthr);
    for (int kc = 0; kc + 2 < chi; ++kc) {
        const double *x = xb + (kc & 1) * chi;
        const int b0 = kc + 1, m = chi - b0;
        double *B = A + b0 * ld + b0;   // the trailing block's lower triangle
        {
            // four elements at a time, loaded before they are used: one worker warp per
            // sub-partition cannot hide shared memory's latency
            const int c = tid & 3;
            for (int i0 = 0; i0 < m; i0 += nwork / 4) {
                const int i = i0 + (tid >> 2);
                double s0 = 0.0, s1 = 0.0;
                if (i0 + (warp << 3) < m) {
                    const int ii = i < m ? i : m - 1;
                    auto at = [&](int j) { return j <= ii ? B[ii * ld + j] : B[j * ld + ii]; };
                    int j = c;
                    for (; j + 12 < m; j += 16) {
                        const double a0 = at(j), a1 = at(j + 4), a2 = at(j + 8), a3 = at(j + 12);
                        const double x0 = x[j], x1 = x[j + 4], x2 = x[j + 8], x3 = x[j + 12];
                        s0 = fma(a0, x0, s0);
                        s1 = fma(a1, x1, s1);
                        s0 = fma(a2, x2, s0);
                        s1 = fma(a3, x3, s1);
                    }
                    for (; j < m; j += 4) s0 = fma(at(j), x[j], s0);
                }
                s0 += s1;
                s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
                s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
                if (i < m && c == 0) y[i] = s0;
            }
        }
        cta_sync();   // A
        {
            const double alpha = sh_alpha, beta = sh_beta;
            if (warp == 0) {
                double s2 = 0.0;
                for (int i = lane; i < m; i += 32) s2 = fma(x[i], y[i], s2);
                const double q = alpha * fma(alpha, B[0], -2.0 * y[0]), hb = 0.5 * beta * beta;
                s2 = warp_sum(s2);
                if (lane == 0) sh_K = hb * (s2 + q);
            } else {
                for (int i = tid - 32; i < m; i += nwork - 32) {
                    p[i] = beta * fma(-alpha, B[i * ld], y[i]);
                    v[i] = i == 0 ? x[0] - alpha : x[i];
                }
            }
        }
        cta_sync();   // B
        {
            // rows 1 .. m-1, columns 1 .. row: rows a and mm-1-a make one list of mm+1 elements
            const double K2 = 2.0 * sh_K;
            const int mm = m - 1, c = tid & 7;
            double *S = B + ld + 1;
            for (int a = tid >> 3; a < (mm + 1) / 2; a += nwork / 8) {
                const int r2 = mm - 1 - a, len = r2 == a ? a + 1 : mm + 1;
                const double va = v[a + 1], ga = fma(-K2, va, p[a + 1]);
                const double vr = v[r2 + 1], gr = fma(-K2, vr, p[r2 + 1]);
                auto place = [&](int e) { return e <= a ? a * ld + e : r2 * ld + e - a - 1; };
                auto upd = [&](int e, double t, double pj, double vj) {
                    return e <= a ? fma(-ga, vj, fma(-va, pj, t)) : fma(-gr, vj, fma(-vr, pj, t));
                };
                int e = c;
                for (; e + 8 < len; e += 16) {
                    const int f = e + 8, j = e <= a ? e : e - a - 1, h = f <= a ? f : f - a - 1;
                    double *t = S + place(e), *u = S + place(f);
                    const double t0 = *t, u0 = *u, pj = p[j + 1], vj = v[j + 1], ph = p[h + 1], vh = v[h + 1];
                    const double wa = e <= a ? va : vr, wg = e <= a ? ga : gr, za = f <= a ? va : vr, zg = f <= a ? ga : gr;
                    *t = fma(-wg, vj, fma(-wa, pj, t0));
                    *u = fma(-zg, vh, fma(-za, ph, u0));
                }
                if (e < len) {
                    const int j = e <= a ? e : e - a - 1;
                    double *t = S + place(e);
                    *t = upd(e, *t, p[j + 1], v[j + 1]);
                }
            }
        }
        next_x_sync(nthr);   // C
    }
    if (tid == 0 && chi >= 2) work[chi - 1] = A[(chi - 1) * ld + chi - 1];
}

// The same reduction with only the lower triangle stored (packed rows; the mat-vec reads
// the upper part through the symmetry), for corners too large for the full matrix:
// chi > TRI_FULL_MAX.  GA: the triangle lives in the work buffer (global memory, L2
// resident: 1 MB at chi = 512) instead of shared memory, for chi > TRI_SMEM_MAX; the
// steps are the same, and __syncthreads orders the block's global accesses as it does
// its shared ones.
__device__ __forceinline__ int lo_off(int i, int j) { return i * (i + 1) / 2 + j; }   // i >= j

template <bool GA>
__global__ void __launch_bounds__(TRI_THREADS) tridiag_packed_kernel(int chi, const double *C, double *work)
{
    extern __shared__ double sm[];
    __shared__ double red[33];
    __shared__ double sh_beta, sh_alpha;
    double *A = GA ? work + tri_global_off(chi) : sm;         // chi (chi + 1) / 2
    double *v = GA ? sm : A + (size_t)chi * (chi + 1) / 2;    // chi
    double *p = v + chi;                                      // chi
    const int tid = threadIdx.x;
    for (int t = tid; t < chi * chi; t += blockDim.x) {
        const int i = t / chi, j = t % chi;
        if (j <= i) A[lo_off(i, j)] = 0.5 * (C[t] + C[(size_t)j * chi + i]);
    }
    __syncthreads();
    for (int kc = 0; kc + 2 < chi; ++kc) {
        const int b0 = kc + 1, m = chi - b0;
        double part = 0.0;
        for (int i = tid; i < m; i += blockDim.x) {
            const double x = A[lo_off(b0 + i, kc)];
            v[i] = x;
            if (i > 0) part += x * x;
        }
        const double tail = block_sum(part, red);
        if (tail == 0.0) continue;
        const double x0 = v[0];
        if (tid == (int)blockDim.x - 1) {
            const double nrm = sqrt(tail + x0 * x0);
            const double alpha = (x0 >= 0.0) ? -nrm : nrm;
            sh_alpha = alpha;
            sh_beta = 1.0 / (nrm * (nrm + fabs(x0)));
        }
        for (int i = tid; i < m; i += blockDim.x) {
            const int r = b0 + i;
            const double *row = A + lo_off(r, b0);   // A[r][b0 + j] for j <= i
            double s0 = 0.0, s1 = 0.0;
            int j = 0;
            for (; j + 1 <= i; j += 2) {
                s0 = fma(row[j], v[j], s0);
                s1 = fma(row[j + 1], v[j + 1], s1);
            }
            if (j <= i) s0 = fma(row[j], v[j], s0);
            for (j = i + 1; j < m; ++j) s1 = fma(A[lo_off(b0 + j, r)], v[j], s1);   // A[r][b0+j] = A[b0+j][r]
            p[i] = s0 + s1;
        }
        __syncthreads();
        const double beta = sh_beta, alpha = sh_alpha;
        for (int i = tid; i < m; i += blockDim.x) p[i] = beta * fma(-alpha, A[lo_off(b0 + i, b0)], p[i]);
        if (tid == 0) v[0] = x0 - alpha;
        __syncthreads();
        double pv = 0.0;
        for (int i = tid; i < m; i += blockDim.x) pv += p[i] * v[i];
        pv = block_sum(pv, red);
        const double Kf = 0.5 * beta * pv;
        for (int i = tid; i < m; i += blockDim.x) p[i] -= Kf * v[i];   // p <- w
        __syncthreads();
        for (int t = tid; t < m * m; t += blockDim.x) {
            const int i = t / m, j = t % m;
            if (j <= i) A[lo_off(b0 + i, b0 + j)] -= v[i] * p[j] + p[i] * v[j];
        }
        if (tid == 0) A[lo_off(b0, kc)] = alpha;
        __syncthreads();
    }
    for (int i = tid; i < chi; i += blockDim.x) {
        work[i] = A[lo_off(i, i)];
        double e = (i + 1 < chi) ? A[lo_off(i + 1, i)] : 0.0;
        work[chi + i] = e * e;
    }
}

// The reduction spread over a thread-block cluster, for chi >= TRI_CLUSTER_MIN: the
// symmetric corner is distributed by rows (row i, all chi entries, on CTA i % CS), so
// each CTA's mat-vec and rank-2 update touch only its own shared memory.  The steps are the
// one-CTA kernel's, with one cluster barrier per column: every CTA forms y_i = (A x)_i for
// its rows and writes them into every CTA's y buffer (distributed shared memory), and the
// owner of row kc + 1 writes that row's trailing part, as it is before the update, into
// every CTA's row buffer.  After the barrier every CTA derives K, p, v, the next column x
// (the broadcast row, updated) and its alpha and beta from the same bits, and updates its
// rows.  The two buffers alternate by column parity, so a broadcast never overwrites one
// still being read (a CTA writes parity kc again only after the barrier of column kc + 1,
// which every CTA reaches after finishing column kc).  Cluster barriers are hardware
// barriers: nothing spins.  Bound by the chain of that barrier, one reduction over chi
// entries and the mat-vec; chi = 128: 654 -> 347 us, chi = 480: 6.52 -> 3.56 ms.
constexpr int TRI_CL_THREADS = 544;   // the largest block tri_cluster_threads gives
constexpr int TRI_CL_SMEM_MAX = 226 * 1024;   // dynamic, below the 227 KB opt-in less the static part

// one warp per local row (4 to 16 warps) and the scalar warp
__host__ __device__ inline int tri_cluster_threads(int chi, int cs)
{
    const int w = (chi + cs - 1) / cs;
    return 32 * ((w < 4 ? 4 : w > 16 ? 16 : w) + 1);
}

__host__ __device__ inline size_t tri_cluster_smem_bytes(int chi, int cs)
{
    return sizeof(double) * ((size_t)((chi + cs - 1) / cs) * chi + 8 * (size_t)chi);
}

template <int CS>
__global__ void __launch_bounds__(TRI_CL_THREADS, 1) tridiag_cluster_kernel(int chi, const double *C, double *work)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ double sm[];
    __shared__ double sh_alpha, sh_beta, sh_K;
    const int rank = (int)cl.block_rank();
    const int nthr = blockDim.x, nwork = nthr - 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = nwork >> 5;
    const int nloc = (chi - rank + CS - 1) / CS;   // rows rank, rank + CS, ...
    const int nmax = (chi + CS - 1) / CS;
    double *A = sm;                           // nmax x chi, full rows
    double *yb = A + (size_t)nmax * chi;      // 2 x chi: y, by parity
    double *rb = yb + 2 * (size_t)chi;        // 2 x chi: the next pivot row, by parity
    double *xb = rb + 2 * (size_t)chi;        // 2 x chi: the column x, by parity
    double *p = xb + 2 * (size_t)chi, *v = p + chi;
    for (int t = tid; t < nloc * chi; t += nthr) {
        const int l = t / chi, j = t % chi, i = rank + CS * l;
        A[t] = 0.5 * (C[(size_t)i * chi + j] + C[(size_t)j * chi + i]);
    }
    for (int j = tid; j < chi; j += nthr) {
        const double a = 0.5 * (C[j] + C[(size_t)j * chi]);
        if (j == 0) {
            if (rank == 0) work[0] = a;
        } else {
            xb[j - 1] = a;
        }
    }
    cl.sync();   // every CTA of the cluster is running before the first remote store
    if (tid >= nwork) {
        // ------------------------------------------------ scalar warp (as in tridiag_kernel)
        for (int kc = 0; kc + 1 < chi; ++kc) {
            const double *x = xb + (size_t)(kc & 1) * chi;
            const int b0 = kc + 1, m = chi - b0;
            double s1 = 0.0, s1b = 0.0;
            for (int i = 1 + lane; i < m; i += 64) {
                s1 = fma(x[i], x[i], s1);
                if (i + 32 < m) s1b = fma(x[i + 32], x[i + 32], s1b);
            }
            s1 = warp_sum(s1 + s1b);
            double alpha, beta;
            tri_scalars(s1, x[0], &alpha, &beta);
            if (lane == 0) {
                sh_alpha = alpha;
                sh_beta = beta;
                if (rank == 0) work[chi + kc] = alpha * alpha;
            }
            if (kc + 2 >= chi) break;
            cl.sync();
            cta_sync();   // B
            const double *r = rb + (size_t)(kc & 1) * chi;
            double *xn = xb + (size_t)((kc + 1) & 1) * chi;
            const double v0 = v[0], p0 = p[0], g0 = fma(-2.0 * sh_K, v0, p0);
            for (int j = lane; j < m; j += 32) {
                const double w = fma(-g0, v[j], fma(-v0, p[j], r[j]));
                if (j > 0) xn[j - 1] = w;
                else if (rank == 0) work[b0] = w;
            }
            __syncwarp();
            next_x_arrive(nthr);
        }
        if (rank == 0 && lane == 0) work[2 * chi - 1] = 0.0;
    } else {
        for (int kc = 0; kc + 2 < chi; ++kc) {
            const int b0 = kc + 1, m = chi - b0;
            const double *x = xb + (size_t)(kc & 1) * chi;
            double *y = yb + (size_t)(kc & 1) * chi, *r = rb + (size_t)(kc & 1) * chi;
            int lf = b0 - rank;                    // first local row with i >= b0
            lf = lf > 0 ? (lf + CS - 1) / CS : 0;
            if (b0 % CS == rank) {
                const double *row = A + (size_t)(b0 / CS) * chi + b0;
                for (int t = tid; t < m * CS; t += nwork) {
                    const int q = t / m, j = t % m;
                    cl.map_shared_rank(r, q)[j] = row[j];
                }
            }
            // half a warp per row: the mat-vec's sums are short, so fewer lanes mean fewer
            // FP64 additions to combine them
            for (int l0 = lf + 2 * warp; l0 < nloc; l0 += 2 * nwarps) {
                const int l = l0 + (lane >> 4), c = lane & 15, i = rank + CS * l;
                double s0 = 0.0, s1 = 0.0;
                if (l < nloc) {
                    const double *row = A + (size_t)l * chi + b0;
                    for (int j = c; j < m; j += 32) {
                        s0 = fma(row[j], x[j], s0);
                        if (j + 16 < m) s1 = fma(row[j + 16], x[j + 16], s1);
                    }
                }
                s0 += s1;
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
                if (l < nloc && c < CS) cl.map_shared_rank(y, c)[i - b0] = s0;
            }
            cl.sync();
            const double alpha = sh_alpha, beta = sh_beta;
            if (warp == 0) {
                double s2 = 0.0, s3 = 0.0;
                for (int i = lane; i < m; i += 64) {
                    s2 = fma(x[i], y[i], s2);
                    if (i + 32 < m) s3 = fma(x[i + 32], y[i + 32], s3);
                }
                const double q = alpha * fma(alpha, r[0], -2.0 * y[0]), hb = 0.5 * beta * beta;
                s2 = warp_sum(s2 + s3);
                if (lane == 0) sh_K = hb * (s2 + q);
            } else {
                for (int i = tid - 32; i < m; i += nwork - 32) {
                    p[i] = beta * fma(-alpha, r[i], y[i]);   // A_i0 = A_0i = r_i
                    v[i] = i == 0 ? x[0] - alpha : x[i];
                }
            }
            cta_sync();   // B
            const double K2 = 2.0 * sh_K;
            for (int l = lf + warp; l < nloc; l += nwarps) {
                const int ii = rank + CS * l - b0;
                if (ii == 0) continue;   // the pivot row: finished by the scalar warps
                const double vi = v[ii], gi = fma(-K2, vi, p[ii]);
                double *row = A + (size_t)l * chi + b0;
                for (int j = 1 + lane; j < m; j += 32) row[j] = fma(-gi, v[j], fma(-vi, p[j], row[j]));
            }
            next_x_sync(nthr);   // C: the rows are final and the next x is there
        }
        if (tid == 0 && (chi - 1) % CS == rank) work[chi - 1] = A[(size_t)((chi - 1) / CS) * chi + chi - 1];
    }
    cl.sync();   // no CTA leaves while another may still write into its shared memory
}

// Number of eigenvalues of the tridiagonal (d, e2), scaled to unit size, below x: the sign
// changes of p_i = (d_i - x) p_{i-1} - e2_{i-1} p_{i-2}.  One FP64 FMA per step on the
// dependent chain; signs are counted, and the range is checked every fourth step, with
// integer instructions on the bit pattern.  No e2 is zero (bisect_kernel puts a floor under
// them), so p = 0 counts as positive and the next p has the sign opposite to the previous
// one's: one change, as it should be.  *p_out 2^(300 *k_out) is the last p.
__device__ __forceinline__ int sturm_count(int n, const double *d, const double *e2, double x, double *p_out,
                                           int *k_out)
{
    double pm = 1.0, p = d[0] - x;
    unsigned hp = (unsigned)__double2hiint(p);
    int cnt = (int)(hp >> 31), k = 0;
    auto step = [&](int i) {
        const double pn = fma(d[i] - x, p, -e2[i - 1] * pm);
        const unsigned hn = (unsigned)__double2hiint(pn);
        cnt += (int)((hn ^ hp) >> 31);
        pm = p;
        p = pn;
        hp = hn;
    };
    int i = 1;
    for (; i + 3 < n; i += 4) {
        step(i);
        step(i + 1);
        step(i + 2);
        step(i + 3);
        const int ex = (int)(hp >> 20) & 0x7FF;
        if (ex > 1023 + 300) {
            p *= 0x1p-300;
            pm *= 0x1p-300;
            ++k;
        } else if (ex < 1023 - 300) {
            p *= 0x1p+300;
            pm *= 0x1p+300;
            --k;
        }
    }
    for (; i < n; ++i) step(i);
    *p_out = p;
    *k_out = k;
    return cnt;
}

// The same count in FP32 (four cycles per dependent operation instead of ~64), rescaled
// every fourth step by the exact power of two of the larger of |p| and |pm|.  Its rounding
// moves an eigenvalue by a few 2^-24 of the matrix's size; the caller checks it.
__device__ __forceinline__ int sturm_count_f32(int n, const float *d, const float *e2, float x)
{
    float pm = 1.0f, p = d[0] - x;
    int cnt = (int)(__float_as_uint(p) >> 31);
    for (int i = 1; i < n; ++i) {
        const float pn = fmaf(d[i] - x, p, -e2[i - 1] * pm);
        cnt += (int)((__float_as_uint(pn) ^ __float_as_uint(p)) >> 31);
        pm = p;
        p = pn;
        if ((i & 3) == 0) {
            const unsigned ex = __float_as_uint(fmaxf(fabsf(p), fabsf(pm))) & 0x7F800000u;
            const float sc = __uint_as_float((254u << 23) - min(max(ex, 1u << 23), 253u << 23));
            p *= sc;
            pm *= sc;
        }
    }
    return cnt;
}

// One warp per eigenvalue (the ei-th smallest), one eigenvalue per CTA, so the Sturm chains
// spread over chi SMs.  Each round counts at 32 points.  Four FP32 rounds bracket the
// eigenvalue to ~2^-19 of the matrix's size; that bracket, widened by 2^-19 on both sides,
// enters FP64 only if the FP64 counts at its ends confirm it (else the whole range does).
// In FP64 the points cluster geometrically (factors of four) around the secant through the
// bracket's last p values, so a round on a well separated eigenvalue shrinks its bracket by
// ~2^15 to 2^24 instead of 2^5; a round that shrank it by less than 2^4 is followed by an
// evenly spaced one, so a cluster costs at most twice the rounds of plain multisection.
// Bound by the FMA chain of a count: 11 FP64 rounds at ~130 cycles a step before, about
// three or four at ~75 and four short ones now; chi = 72: 155 -> 38 us (90 on a corner
// graded over twelve decades), chi = 480: 1068 -> 357 us.
constexpr double BISECT_WIDTH = 4e-16;   // final bracket, of the Frobenius norm
__global__ void bisect_kernel(int chi, const double *work, double *lam)
{
    extern __shared__ double sm[];
    double *d = sm, *e2 = sm + chi;                              // 2 chi
    float *df = reinterpret_cast<float *>(e2 + chi), *e2f = df + chi;   // 2 chi FP32
    const int lane = threadIdx.x & 31;
    const int ei = blockIdx.x;
    // every eigenvalue lies in [-|T|_F, |T|_F] (the Frobenius norm bounds the spectral
    // radius; it is the corner's, unchanged by the orthogonal reduction)
    double f2 = 0.0;
    for (int i = lane; i < chi; i += 32) f2 = fma(work[i], work[i], f2) + 2.0 * work[chi + i];
    f2 = warp_sum(f2);
    const int fx = (__double2hiint(f2) >> 20) & 0x7FF;
    if (fx < 2 || fx > 2044) {   // zero (or far below the range), or not finite
        if (lane == 0) lam[ei] = fx < 2 ? 0.0 : __longlong_as_double(0x7FF8000000000000LL);
        return;
    }
    const int k = (fx - 1023) >> 1;   // |T|_F = sqrt(f2) in [2^k, 2^(k+1))
    const double sc = __hiloint2double((1023 - k) << 20, 0);
    for (int i = lane; i < chi; i += 32) {
        const double di = work[i] * sc, ei2 = fmax(work[chi + i] * sc * sc, 0x1p-200);
        d[i] = di;
        e2[i] = ei2;
        df[i] = (float)di;
        e2f[i] = fmaxf((float)ei2, 0x1p-60f);
    }
    __syncwarp();
    const double top = 2.0;   // > |T|_F of the scaled matrix
    double lo = -top, hi = top;
    {
        float flo = -2.0f, fhi = 2.0f;
        for (int round = 0; round < 4; ++round) {
            const float x = flo + (fhi - flo) * (float)(lane + 1) * (1.0f / 33.0f);
            const unsigned below = __ballot_sync(0xffffffffu, sturm_count_f32(chi, df, e2f, x) <= ei);
            const int L = __popc(below);
            const float xl = __shfl_sync(0xffffffffu, x, L > 0 ? L - 1 : 0);
            const float xh = __shfl_sync(0xffffffffu, x, L < 32 ? L : 31);
            flo = L > 0 ? xl : flo;
            fhi = L < 32 ? xh : fhi;
        }
        lo = (double)flo - 0x1p-19;
        hi = (double)fhi + 0x1p-19;
    }
    const double width = BISECT_WIDTH * sc * sqrt(f2);
    bool ends = true;       // this pass checks the bracket's own ends
    bool even = true;       // evenly spaced points
    double r = 0.0;         // secant estimate, when !even
    for (int round = 0; round < 40 && hi - lo > width; ++round) {
        double x;
        if (ends) {
            x = lo + (hi - lo) * ((double)lane * (1.0 / 31.0));
        } else if (even) {
            x = lo + (hi - lo) * ((double)(lane + 1) * (1.0 / 33.0));
        } else {
            // lanes 0 .. 15: r - (r - lo) 4^-(lane + 1/2); lanes 16 .. 31 likewise towards hi
            const int q = lane < 16 ? lane : 31 - lane;
            const double off = __hiloint2double((1022 - 2 * q) << 20, 0);   // 2^-(2 q + 1)
            x = lane < 16 ? r - (r - lo) * off : r + (hi - r) * off;
        }
        double pl;
        int pk;
        const int cnt = sturm_count(chi, d, e2, x, &pl, &pk);
        const unsigned below = __ballot_sync(0xffffffffu, cnt <= ei);   // a prefix of lanes
        const int L = __popc(below);
        if (ends) {
            ends = false;
            if (L == 0 || L == 32) {   // the FP32 bracket missed: the whole range
                lo = -top;
                hi = top;
                continue;
            }
        }
        const int a = L > 0 ? L - 1 : 0, b = L < 32 ? L : 31;
        const double xl = __shfl_sync(0xffffffffu, x, a), xh = __shfl_sync(0xffffffffu, x, b);
        const double nlo = L > 0 ? xl : lo, nhi = L < 32 ? xh : hi;
        const bool poor = !even && nhi - nlo > 0.0625 * (hi - lo);
        // secant through the bracket's ends, in FP32 on a common exponent
        const double fl = __shfl_sync(0xffffffffu, pl, a), fh = __shfl_sync(0xffffffffu, pl, b);
        const int kl = __shfl_sync(0xffffffffu, pk, a), kh = __shfl_sync(0xffffffffu, pk, b);
        const int xa = (__double2hiint(fl) >> 20) & 0x7FF, xe = (__double2hiint(fh) >> 20) & 0x7FF;
        lo = nlo;
        hi = nhi;
        even = poor || L == 0 || L == 32 || kl != kh || xa == 0 || xe == 0 || xa - xe > 60 || xe - xa > 60;
        if (!even) {
            const float ga = (float)__hiloint2double((__double2hiint(fl) & 0x000FFFFF) | 0x3FF00000, __double2loint(fl));
            const float gb = (float)__hiloint2double(
                (__double2hiint(fh) & 0x000FFFFF) | ((1023 + xe - xa) << 20), __double2loint(fh));
            r = lo + (hi - lo) * (double)(ga / (ga + gb));
            even = !(r > lo && r < hi);
        }
    }
    if (lane == 0) lam[ei] = 0.5 * (lo + hi) * __hiloint2double((1023 + k) << 20, 0);
}

// stride 2: the chi x stride eigenvalues come in equal pairs (a Hermitian corner through
// its real embedding); every second one of the sorted magnitudes is kept.
__global__ void spectrum_finish_kernel(int chi, int stride, const double *lam_in, double *s_new, const double *s_old,
                                       double *delta)
{
    __shared__ double red[33];
    __shared__ double lam[SPEC_MAX_CHI], srt[SPEC_MAX_CHI];
    const int tid = threadIdx.x, nall = chi * stride;
    for (int i = tid; i < nall; i += blockDim.x) lam[i] = fabs(lam_in[i]);
    __syncthreads();
    // magnitudes compare as integers (the FP64 pipe's compares would bind: 139 -> 19 us at
    // chi = 480)
    const unsigned long long *key = reinterpret_cast<const unsigned long long *>(lam);
    for (int i = tid; i < nall; i += blockDim.x) {
        const unsigned long long ai = key[i];
        int rank = 0;
        for (int j = 0; j < nall; ++j) rank += key[j] + (j < i ? 1 : 0) > ai;
        srt[rank] = lam[i];
    }
    __syncthreads();
    double ss = 0.0;
    for (int i = tid; i < chi; i += blockDim.x) ss += srt[i * stride] * srt[i * stride];
    ss = block_sum(ss, red);
    const double f = ss > 0.0 ? 1.0 / sqrt(ss) : 0.0;
    for (int i = tid; i < chi; i += blockDim.x) lam[i] = srt[i * stride] * f;
    __syncthreads();
    for (int i = tid; i < chi; i += blockDim.x) srt[i] = lam[i];
    __syncthreads();
    double dd = 0.0;
    for (int i = tid; i < chi; i += blockDim.x) {
        double x = srt[i] - s_old[i];
        dd += x * x;
    }
    dd = block_sum(dd, red);
    for (int i = tid; i < chi; i += blockDim.x) s_new[i] = srt[i];
    if (tid == 0) *delta = sqrt(dd);
}

__global__ void spectrum_init_kernel(int chi, double *s)
{
    for (int i = threadIdx.x; i < chi; i += blockDim.x) s[i] = 1.0 / sqrt((double)chi);
}

// Eq. (1): rho[(sA sB)][(tA tB)] = raw[(sB tB)][(sA tA)] / trace; e_a = tr(rho h_a);
// E_site = (1/2) sum_a e_a.  out: e_x, e_y, e_z, E_site, then rho (d^4).
__global__ void bond_energy_kernel(int d, const double *raw, const double *h, double *out)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int dd = d * d;
    double z = 0.0;
    for (int sA = 0; sA < d; ++sA)
        for (int sB = 0; sB < d; ++sB) z += raw[(sB * d + sB) * dd + (sA * d + sA)];
    double *rho = out + 4;
    for (int sA = 0; sA < d; ++sA)
        for (int sB = 0; sB < d; ++sB)
            for (int tA = 0; tA < d; ++tA)
                for (int tB = 0; tB < d; ++tB)
                    rho[(sA * d + sB) * dd + tA * d + tB] = raw[(sB * d + tB) * dd + (sA * d + tA)] / z;
    double es = 0.0;
    for (int a = 0; a < 3; ++a) {
        double e = 0.0;
        for (int r = 0; r < dd; ++r)
            for (int c = 0; c < dd; ++c) e += rho[r * dd + c] * h[(size_t)a * dd * dd + c * dd + r];
        out[a] = e;
        es += e;
    }
    out[3] = 0.5 * es;
}

__global__ void check_finite_kernel(long long count, const double *x, int *flag)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < count;
         t += (long long)gridDim.x * blockDim.x)
        if (!isfinite(x[t])) *flag = 1;
}

int grid_for(long long count, int per_sm = 8)
{
    long long b = (count + 255) / 256;
    long long cap = (long long)per_sm * device_sm_count();
    if (b > cap) b = cap;
    return b < 1 ? 1 : (int)b;
}

}  // namespace

cudaError_t launch_c3v_project_normalize(int d, int D, const double *Ain, double *Aout, int symmetrize,
                                         cudaStream_t st)
{
    size_t smem = sizeof(double) * (size_t)d * D * D * D;
    if (smem > 200 * 1024) return cudaErrorInvalidValue;
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(c3v_project_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    CTM_COUNT_LAUNCH(1);
    c3v_project_kernel<<<1, 256, smem, st>>>(d, D, Ain, Aout, symmetrize);
    return cudaGetLastError();
}

cudaError_t launch_double_layer(int d, int D, const double *K, const double *B, double *a, cudaStream_t st)
{
    long long tot = (long long)D * D * D * D * D * D;
    CTM_COUNT_LAUNCH(1);
    double_layer_kernel<<<grid_for(tot), 256, 0, st>>>(d, D, K, B, a);
    return cudaGetLastError();
}

cudaError_t launch_open_layers(int d, int D, const double *A, double *b, cudaStream_t st)
{
    long long tot = (long long)D * D * D * D * D * D * d * d;
    CTM_COUNT_LAUNCH(1);
    open_layers_kernel<<<grid_for(tot), 256, 0, st>>>(d, D, A, b);
    return cudaGetLastError();
}

cudaError_t launch_init_env(int chi, int D, const double *a, double *C, double *T, double *Q, cudaStream_t st)
{
    long long tot = (long long)chi * D * D * chi;
    CTM_COUNT_LAUNCH(1);
    init_env_kernel<<<grid_for(tot), 256, 0, st>>>(chi, D, a, C, T, Q);
    return cudaGetLastError();
}

cudaError_t launch_warm_start(int n, int chi, const double *Q, const double *C, double *Qs, cudaStream_t st)
{
    CTM_COUNT_LAUNCH(1);
    warm_start_kernel<<<grid_for((long long)n * chi), 256, 0, st>>>(n, chi, Q, C, Qs);
    return cudaGetLastError();
}

cudaError_t launch_select_columns(int n, int chi, const double *M, const double *C, double *Y, cudaStream_t st)
{
    CTM_COUNT_LAUNCH(1);
    select_columns_kernel<<<grid_for((long long)n * chi), 256, 0, st>>>(n, chi, M, C, Y);
    return cudaGetLastError();
}

cudaError_t launch_corner_sym_normalize(int chi, const double *Cr, double *Cn, double *partials, cudaStream_t st)
{
    int nb = (chi * chi + 255) / 256;
    if (nb > CORNER_NORM_BLOCKS) nb = CORNER_NORM_BLOCKS;
    CTM_COUNT_LAUNCH(2);
    corner_sym_sumsq_kernel<<<nb, 256, 0, st>>>(chi, Cr, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    corner_sym_scale_kernel<<<nb, 256, 0, st>>>(chi, Cr, partials, nb, Cn);
    return cudaGetLastError();
}

cudaError_t launch_normalize(long long count, double *x, double *partials, int nblocks, cudaStream_t st)
{
    CTM_COUNT_LAUNCH(1);
    sumsq_partial_kernel<<<nblocks, 256, 0, st>>>(count, x, partials);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    CTM_COUNT_LAUNCH(1);
    scale_by_partials_kernel<<<nblocks, 256, 0, st>>>(count, x, partials, nblocks);
    return cudaGetLastError();
}

// Cluster size for the distributed reduction of a chi x chi corner (chi >= TRI_CLUSTER_MIN):
// 16 CTAs where the device schedules such clusters with this shared memory, else 8,
// else 0 (the single-CTA reduction from global memory).  Decided once per chi.
static std::mutex g_tri_mu;
static signed char g_tri_cs[SPEC_MAX_CHI + 1];   // 0: not decided, -1: none, else the size
static std::atomic<bool> g_tri_cluster_ok{false}; // the cluster kernels' attributes were accepted

template <int CS>
static int tri_cluster_fits(int chi)
{
    const size_t smem = tri_cluster_smem_bytes(chi, CS);
    if (smem > TRI_CL_SMEM_MAX) return 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(CS, 1, 1);
    cfg.blockDim = dim3(tri_cluster_threads(chi, CS), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, tridiag_cluster_kernel<CS>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nc > 0;
}

static int tri_cluster_size(int chi)
{
    if (chi < TRI_CLUSTER_MIN || chi > SPEC_MAX_CHI || !g_tri_cluster_ok) return 0;
    std::lock_guard<std::mutex> lk(g_tri_mu);
    if (!g_tri_cs[chi]) g_tri_cs[chi] = tri_cluster_fits<16>(chi) ? 16 : tri_cluster_fits<8>(chi) ? 8 : -1;
    return g_tri_cs[chi] > 0 ? g_tri_cs[chi] : 0;
}

static cudaError_t launch_tridiag_cluster(int cs, int chi, const double *C, double *work, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cs, 1, 1);
    cfg.blockDim = dim3(tri_cluster_threads(chi, cs), 1, 1);
    cfg.dynamicSmemBytes = tri_cluster_smem_bytes(chi, cs);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cs == 16 ? cudaLaunchKernelEx(&cfg, tridiag_cluster_kernel<16>, chi, C, work)
                    : cudaLaunchKernelEx(&cfg, tridiag_cluster_kernel<8>, chi, C, work);
}

size_t spectrum_work_doubles(int chi)
{
    return tri_global_off(chi) + (chi > TRI_SMEM_MAX ? (size_t)chi * (chi + 1) / 2 : 0);
}

// bisection of the tridiagonal in work (n = chi x stride eigenvalues), then the sorted,
// normalised magnitudes (every stride-th) and delta
static cudaError_t spectrum_tail(int chi, int stride, double *work, double *s_new, const double *s_old, double *delta,
                                 cudaStream_t st)
{
    const int n = chi * stride;
    CTM_COUNT_LAUNCH(2);
    bisect_kernel<<<n, 32, 3 * sizeof(double) * n, st>>>(n, work, work + 2 * n);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    spectrum_finish_kernel<<<1, 256, 0, st>>>(chi, stride, work + 2 * n, s_new, s_old, delta);
    return cudaGetLastError();
}

static cudaError_t launch_tridiag(int chi, const double *C, double *work, cudaStream_t st, bool reserve_sm);

cudaError_t launch_spectrum_pairs(int chi, const double *E, double *s_new, const double *s_old, double *delta,
                                  double *work, cudaStream_t st)
{
    if (2 * chi > SPEC_MAX_CHI || !work) return cudaErrorInvalidValue;
    cudaError_t e = launch_tridiag(2 * chi, E, work, st, false);
    if (e != cudaSuccess) return e;
    return spectrum_tail(chi, 2, work, s_new, s_old, delta, st);
}

cudaError_t launch_spectrum(int chi, const double *C, double *s_new, const double *s_old, double *delta,
                            double *work, cudaStream_t st, bool reserve_sm)
{
    if (chi > SPEC_MAX_CHI || !work) return cudaErrorInvalidValue;
    cudaError_t e = launch_tridiag(chi, C, work, st, reserve_sm);
    if (e != cudaSuccess) return e;
    return spectrum_tail(chi, 1, work, s_new, s_old, delta, st);
}

// step one of the spectrum: the tridiagonal (d, e^2) of the symmetric chi x chi matrix C in work
static cudaError_t launch_tridiag(int chi, const double *C, double *work, cudaStream_t st, bool reserve_sm)
{
    // reserve_sm: the tridiagonalisation runs beside a lone instance's step for ~0.4 ms on
    // one SM; asking for (nearly) all of the SM's shared memory keeps the step's CTAs off
    // that SM, whose CTAs it would otherwise slow (a grid-synchronous QR waits for its
    // slowest CTA): measured 0.892 -> 0.872 ms per step at D = 6, chi = 72.  (Not inside a
    // batch, where many spectra run at once.)
    const bool full = chi <= TRI_FULL_MAX, global = chi > TRI_SMEM_MAX;
    size_t smem = full ? tri_full_smem_bytes(chi)
                       : sizeof(double) * ((global ? 0 : (size_t)chi * (chi + 1) / 2) + 2 * (size_t)chi);
    if (reserve_sm && smem < SPEC_SM_ALONE_BYTES) smem = SPEC_SM_ALONE_BYTES;
    CTM_COUNT_LAUNCH(1);
    cudaError_t e = cudaSuccess;
    const int cs = tri_cluster_size(chi);
    if (cs) e = launch_tridiag_cluster(cs, chi, C, work, st);
    else if (full) tridiag_kernel<<<1, 32 * TRI_WARPS, smem, st>>>(chi, C, work);
    else if (!global) tridiag_packed_kernel<false><<<1, TRI_THREADS, smem, st>>>(chi, C, work);
    else tridiag_packed_kernel<true><<<1, TRI_THREADS, smem, st>>>(chi, C, work);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t launch_spectrum_from_tridiag(int chi, double *work, double *s_new, const double *s_old, double *delta,
                                        cudaStream_t st)
{
    if (chi > SPEC_MAX_CHI || !work) return cudaErrorInvalidValue;
    return spectrum_tail(chi, 1, work, s_new, s_old, delta, st);
}

cudaError_t launch_spectrum_init(int chi, double *s, cudaStream_t st)
{
    CTM_COUNT_LAUNCH(1);
    spectrum_init_kernel<<<1, 256, 0, st>>>(chi, s);
    return cudaGetLastError();
}

cudaError_t launch_bond_energy(int d, const double *rho_raw, const double *h, double *out, cudaStream_t st)
{
    CTM_COUNT_LAUNCH(1);
    bond_energy_kernel<<<1, 32, 0, st>>>(d, rho_raw, h, out);
    return cudaGetLastError();
}

cudaError_t launch_check_finite(long long count, const double *x, int *flag, cudaStream_t st)
{
    CTM_COUNT_LAUNCH(1);
    check_finite_kernel<<<grid_for(count), 256, 0, st>>>(count, x, flag);
    return cudaGetLastError();
}

cudaError_t spectrum_prepare()
{
    cudaError_t e = cudaFuncSetAttribute(tridiag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(tridiag_packed_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(tridiag_packed_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024);
    if (e != cudaSuccess) return e;
    // the cluster reduction is optional: where the device refuses these attributes the
    // single-CTA reduction from global memory serves
    const bool ok = cudaFuncSetAttribute(tridiag_cluster_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         TRI_CL_SMEM_MAX) == cudaSuccess &&
                    cudaFuncSetAttribute(tridiag_cluster_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         TRI_CL_SMEM_MAX) == cudaSuccess &&
                    cudaFuncSetAttribute(tridiag_cluster_kernel<16>, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                         1) == cudaSuccess;
    if (!ok) cudaGetLastError();
    g_tri_cluster_ok = ok;
    return cudaSuccess;
}
