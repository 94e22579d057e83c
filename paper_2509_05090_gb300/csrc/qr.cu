// Householder QR of the reduced corner Y (n x k, tall and skinny), Sec. II.B,
// Fig. 3(d): Y = Q R with Q serving as the isometric projector and the gauge
// fixed so that diag(R) >= 0.  Always FP64.
//
// One cooperative launch over G <= #SM CTAs.  CTA c keeps its block of rows of
// Y (and later of the reflectors) in shared memory for the whole factorisation, or,
// where one SM's share of the rows does not fit there beside the panel scratch (large
// k or n), in its part of a global slab that stays in L2 (qr_kernel<true>: the same
// steps on the same layout, on a grid that leaves two SMs free).
// Columns are taken in panels of up to QB (8).  For a panel starting at column j0
// every CTA forms, over its rows >= j0, the partial Gram rows
// G[i][kk] = a_{j0+i}^T a_kk (i < QB, kk >= j0+i) and the owners publish the
// panel's rows j0 .. j0+QB-1; the partial sums meet in global memory through
// FP64 atomics and one grid barrier.  Then every CTA derives the panel's
// reflectors redundantly, column by column, from those numbers alone: for
// column j = j0+i with x = the column below the diagonal, alpha = -sign(x_0)|x|,
// v = x - alpha e_0, tau = 2/v^T v and v^T a_kk = G[i][kk] - alpha a_jk.
// Because the reflector H_j is orthogonal, the Gram rows of the later panel
// columns after applying it are the same inner products minus the row-j
// contribution, G[i'][kk] -= R[j][j0+i'] R[j][kk], and the published rows are
// updated like the data.  A downdated squared norm that falls below 1/16 of its
// value at the panel start ends the panel there (so rounding errors are
// amplified at most 4x); the next panel then starts from freshly reduced sums,
// which makes the worst case the one-column-per-barrier algorithm.  Finally the
// CTA applies the panel's reflectors to its own rows and, in the same pass over
// its shared-memory block, forms the next panel's partial Gram rows.  So a
// panel of QB columns costs one grid barrier.  Q = H_0 ... H_{k-1} [I; 0] is then
// formed in compact-WY form inside the same launch: with the unnormalised
// reflectors v_j as the columns of V and S = V^T V, the triangular factor
// satisfies T^{-1} = striu(S) + diag(S)/2 (the "UT" form of the product of
// reflectors), so Q = E - V W with W = T V_top^T.  Every CTA adds its rows' share
// of S with FP64 atomics; after a grid barrier ceil(k/4) CTAs solve four columns
// of W each (blocked back-substitution with inverted 8 x 8 diagonal blocks); after
// a second barrier every CTA forms its rows of Q and applies the gauge (columns
// with R_jj < 0 negated, and the rows of R with them).  The grid size is tuned
// once per shape by timing a few rows-per-CTA choices.
//
// What bounds it: FP64 instructions, one per warp, 64 cycles and sub-partition, whether or not
// the next depends on it and whether or not its lanes are predicated off (measured).  So the
// panel's chain runs in one warp on the QB x QB blocks alone, with the other columns and the
// rows following it reflector by reflector in other sub-partitions; lanes per column are picked
// from that cost; partial sums are combined by halving; nothing FP64 sits under a predicate.
// n x k: 512 x 32 119 -> 66 us, 2592 x 72 307 -> 214 (panels 23k -> 13k cycles each, update and
// Gram passes 17k -> 8k), 8192 x 128 1027 -> 833, 5184 x 144 987 -> 802, 12000 x 240
// 2350 -> 1960.  From n k^2 = 5e7 on, S, W and Q, and
// with many columns the trailing update too, leave that pipe for the tensor cores (the blocked
// form near the end of this file): 8192 x 128 845 -> 643 us, 12000 x 480 12.9 -> 4.3 ms.
//
// The grid barrier is one monotonic counter in global memory; its spin is
// bounded (about a second) and on expiry sets an error flag that the host
// reports as CTM_ETIMEOUT instead of hanging.  A context's forced-timeout switch
// (a test of that path) makes the barrier wait for one arrival more than the grid
// has, with a short spin limit; every CTA then gives up at its first barrier and
// returns.
#include <cooperative_groups.h>
#include <cstdlib>
#include <type_traits>

#include "ctm_internal.h"
#include "fp64_chain.h"

namespace {

constexpr int QR_THREADS = 512;
constexpr int QR_DET_GMAX = 320;   // deterministic mode: partial-sum slots (CTAs) provided for
constexpr int QB = 8;                     // panel width (columns per grid barrier)
constexpr int QR_DOWNDATE_LOG2 = 4;               // smallest kept ratio of downdated / fresh norm^2: 2^-4
constexpr long long QR_SPIN_LIMIT = 20000000LL;   // x ~64 ns sleep: ~1.3 s

// Grid barrier number `epoch` (1, 2, ...): every CTA adds 1 to a monotonic
// counter with a release reduction (no value returned) and polls the counter
// with acquire loads until it reaches G * epoch.  No reset, no separate flag;
// the poll is bounded.
__device__ __forceinline__ bool grid_barrier(unsigned *count, unsigned G, unsigned epoch, int *err, unsigned extra,
                                             long long spin_limit)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
        const unsigned target = G * epoch + extra;
        long long it = 0;
        unsigned f;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(f) : "l"(count) : "memory");
            if ((int)(f - target) >= 0) break;
            if (++it > spin_limit) {
                atomicExch(err, 1);
                break;
            }
            if (it > 64) __nanosleep(32);
        }
    }
    __syncthreads();
    return *((volatile int *)err) == 0;
}

// sum_{c < G} p[c * stride] by a group of DET_LANES consecutive lanes: lane `part`
// adds c = part, part + DET_LANES, ... (independent loads, one round of L2 latency), and
// an xor butterfly adds the lanes' sums (every lane gets the same bits; the assignment
// is fixed, so the result is the same on every run): the deterministic mode's
// cross-CTA reduction.  All lanes of the group must call it.
constexpr int DET_LANES = 16;
__device__ __forceinline__ double det_sum(const double *p, size_t stride, int G, int part)
{
    double s = 0.0;
    for (int c = part; c < G; c += DET_LANES) s += __ldcg(p + (size_t)c * stride);
#pragma unroll
    for (int o = DET_LANES / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, DET_LANES);
    return s;
}

struct QrArgs {
    int n, k, G, rows_per;
    const double *Y;
    double *R;
    double *Q;        // n x k projector (written)
    double *V;        // first k rows of the reflectors (written, read by the W solve)
    double *S;        // k x k: V^T V, upper triangle (zeroed by the host, summed with atomics)
    double *W;        // k x k: T V_top^T (written by the solving CTAs)
    double *sbuf;     // 3 x QB x k rotating Gram-row accumulators
    double *rowbuf;   // 2 x QB x k published panel rows
    unsigned *bar;
    int *err;
    unsigned bar_extra;
    long long spin_limit;
    // deterministic mode (non-null): each CTA writes its partial sums to its own slot
    // and every reader adds the G slots in CTA order, instead of FP64 atomics
    double *gpart;    // 2 x G x QB x k: partial Gram rows, by panel parity
    double *spart;    // G x k x k: partial V^T V
    // row blocks too tall for shared memory: CTA c's block at yslab + c * rows_per * (k | 1)
    double *yslab;
    // one panel of the blocked factorisation (qr_kernel's FACT): row pitch of Y, R and V (n x k
    // here, all rows), and per column tau and the sign of R's diagonal
    int pitch;
    double *taus, *sgn;
};

// W = U^{-1} V_top^T with U = striu(S) + diag(S)/2 (unit diagonal where tau = 0).
// (V null: U^{-1} itself.)  The k right-hand sides are independent: CTA b of the QR grid solves columns
// [4b, 4b + 4) after the grid barrier that completes S.
// Rows are blocked by QR_WB = 8 from the bottom; every CTA first inverts the
// diagonal 8 x 8 blocks of U (all blocks at once, one thread per block column),
// then per row block sums the already solved rows below it (independent dot
// products split over QR_WL lanes) and applies the block inverse (8-term dots).
// So the dependent FP64 chains per block are short and the CTA syncs twice per
// block.  U (packed upper triangle), the block inverses and the CTA's W columns
// live in shared memory.
constexpr int QR_WB = 8;      // row block (and diagonal inverse) size
constexpr int QR_WC = 4;      // right-hand-side columns per CTA
constexpr int QR_WL = 8;      // lanes per dot product in the block update

__device__ __forceinline__ int up_off(int k, int i, int j) { return i * k - (i * (i - 1)) / 2 + (j - i); }

// Up to QR_WY_PACKED_MAX columns U is copied into shared memory (packed upper triangle);
// beyond, the solve reads it from S in global memory (L2) and shared memory holds only
// the block inverses and the CTA's W columns.
constexpr int QR_WY_PACKED_MAX = 160;
constexpr int QR_MAX_COLS = 512;   // the Q formation gives each column at least one thread
constexpr size_t QR_SMEM_MAX = 200 * 1024;
__host__ __device__ inline bool wy_packed(int k) { return k <= QR_WY_PACKED_MAX; }

size_t qr_wy_smem_bytes(int k)
{
    const int nb = (k + QR_WB - 1) / QR_WB;
    const size_t packed = wy_packed(k) ? (size_t)k * (k + 1) / 2 : 0;
    return sizeof(double) * (packed + (size_t)nb * QR_WB * QR_WB + (size_t)k * QR_WC + k);
}

template <bool PACKED>
__device__ void wy_solve_cta(int k, int cblk, const double *S, const double *V, const double *taus, double *W,
                             double *sm)
{
    const int nb = (k + QR_WB - 1) / QR_WB;
    double *Us = sm;                                               // PACKED: k (k+1) / 2
    double *Di = Us + (PACKED ? (size_t)k * (k + 1) / 2 : 0);      // nb x 8 x 8 block inverses
    double *Wc = Di + (size_t)nb * QR_WB * QR_WB;                  // k x QR_WC
    double *rd = Wc + (size_t)k * QR_WC;                           // k reciprocal diagonal
    const int c0 = cblk * QR_WC;
    const int ncol = min(QR_WC, k - c0);
    const int tid = threadIdx.x;
    // U[i][j] (j >= i): striu(S) + diag(S)/2, a unit diagonal where tau = 0
    auto uval = [&](int i, int j) -> double {
        if (PACKED) return Us[up_off(k, i, j)];
        if (j > i) return __ldcg(S + (size_t)i * k + j);
        return (taus[i] == 0.0) ? 1.0 : 0.5 * __ldcg(S + (size_t)i * k + i);
    };
    if (PACKED)
        for (int t = tid; t < k * k; t += blockDim.x) {
            const int i = t / k, j = t % k;
            if (j > i) Us[up_off(k, i, j)] = __ldcg(S + t);
            else if (j == i) Us[up_off(k, i, i)] = (taus[i] == 0.0) ? 1.0 : 0.5 * __ldcg(S + t);
        }
    for (int t = tid; t < k * QR_WC; t += blockDim.x) {
        const int i = t / QR_WC, cc = t % QR_WC;
        Wc[t] = V ? ((cc < ncol) ? __ldcg(V + (size_t)(c0 + cc) * k + i) : 0.0) : (i == c0 + cc ? 1.0 : 0.0);
    }
    __syncthreads();
    for (int i = tid; i < k; i += blockDim.x) rd[i] = 1.0 / uval(i, i);
    __syncthreads();
    // block inverses: thread (b, c) back-substitutes D_b x = e_c
    for (int t = tid; t < nb * QR_WB; t += blockDim.x) {
        const int bb = t / QR_WB, cl = t % QR_WB;
        const int i0 = bb * QR_WB, bs = min(QR_WB, k - i0);
        double *D = Di + bb * QR_WB * QR_WB;
        if (cl < bs) {
            double x[QR_WB];
#pragma unroll
            for (int r = QR_WB - 1; r >= 0; --r) {
                double v = 0.0;
                if (r <= cl) {
                    v = (r == cl) ? 1.0 : 0.0;
#pragma unroll
                    for (int j = r + 1; j < QR_WB; ++j)
                        if (j <= cl) v = fma(-uval(i0 + r, i0 + j), x[j], v);
                    v *= rd[i0 + r];
                }
                x[r] = v;
            }
#pragma unroll
            for (int r = 0; r < QR_WB; ++r) D[r * QR_WB + cl] = x[r];
        } else {
#pragma unroll
            for (int r = 0; r < QR_WB; ++r) D[r * QR_WB + cl] = 0.0;
        }
    }
    __syncthreads();
    for (int bb = nb - 1; bb >= 0; --bb) {
        const int i0 = bb * QR_WB, i1 = min(k, i0 + QR_WB);
        // rhs of the block: Wc[i][cc] -= sum_{j >= i1} U[i][j] Wc[j][cc]
        for (int t = tid; t < QR_WB * QR_WC * QR_WL; t += blockDim.x) {
            const int lane = t % QR_WL, pc = t / QR_WL;
            const int i = i0 + pc / QR_WC, cc = pc % QR_WC;
            double s0 = 0.0, s1 = 0.0;
            if (i < i1) {
                // u[j] = U[i][j] for j >= i (j > i here: the rows below the block)
                const double *u = PACKED ? Us + up_off(k, i, i) - i : S + (size_t)i * k;
                int j = i1 + lane;
                for (; j + QR_WL < k; j += 2 * QR_WL) {
                    s0 = fma(PACKED ? u[j] : __ldcg(u + j), Wc[j * QR_WC + cc], s0);
                    s1 = fma(PACKED ? u[j + QR_WL] : __ldcg(u + j + QR_WL), Wc[(j + QR_WL) * QR_WC + cc], s1);
                }
                if (j < k) s0 = fma(PACKED ? u[j] : __ldcg(u + j), Wc[j * QR_WC + cc], s0);
            }
            double sum = s0 + s1;
#pragma unroll
            for (int o = QR_WL / 2; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o, QR_WL);
            if (lane == 0 && i < i1) Wc[i * QR_WC + cc] -= sum;
        }
        __syncthreads();
        // apply the block inverse
        double wv = 0.0;
        const int r = tid / QR_WC, cc = tid % QR_WC;
        if (tid < QR_WB * QR_WC && i0 + r < i1) {
            const double *D = Di + bb * QR_WB * QR_WB + r * QR_WB;
#pragma unroll
            for (int j = 0; j < QR_WB; ++j)
                if (i0 + j < i1) wv = fma(D[j], Wc[(i0 + j) * QR_WC + cc], wv);
        }
        __syncthreads();
        if (tid < QR_WB * QR_WC && i0 + r < i1) Wc[(i0 + r) * QR_WC + cc] = wv;
        __syncthreads();
    }
    for (int t = tid; t < k * QR_WC; t += blockDim.x) {
        const int i = t / QR_WC, cc = t % QR_WC;
        if (cc < ncol) W[(size_t)i * k + c0 + cc] = Wc[t];
    }
}

// RP rows per thread and pass of the Q formation, W from L2 four rows at a time
template <int RP>
__device__ void q_rows(const QrArgs &a, const double *alps, const double *Ys, int ld, int r0, int nr)
{
    const int k = a.k, grp = blockDim.x / k, col = threadIdx.x % k, g = threadIdx.x / k;
    if (g >= grp) return;
    const double sgn = alps[col] < 0.0 ? -1.0 : 1.0;
    for (int rb = g * RP; rb < nr; rb += grp * RP) {
        const double *rows[RP];
        double acc[RP];
#pragma unroll
        for (int q = 0; q < RP; ++q) {
            acc[q] = 0.0;
            rows[q] = Ys + (size_t)min(rb + q, nr - 1) * ld;
        }
        int j = 0;
        for (; j + 3 < k; j += 4) {
            double w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = __ldcg(a.W + (size_t)(j + u) * k + col);
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int q = 0; q < RP; ++q) acc[q] = fma(rows[q][j + u], w[u], acc[q]);
        }
        for (; j < k; ++j) {
            const double w = __ldcg(a.W + (size_t)j * k + col);
#pragma unroll
            for (int q = 0; q < RP; ++q) acc[q] = fma(rows[q][j], w, acc[q]);
        }
#pragma unroll
        for (int q = 0; q < RP; ++q) {
            const int rg = r0 + rb + q;
            if (rb + q < nr) a.Q[(size_t)rg * k + col] = sgn * ((rg == col ? 1.0 : 0.0) - acc[q]);
        }
    }
}

// GY: the CTA's row block lives in a global slab (L2) instead of shared memory, for
// blocks too tall for it (large k or n); the algorithm and the access order are the same.
// FACT: one panel of the blocked factorisation below, columns of a wider matrix: R's block, the
// reflectors (each scaled by a power of two to v_0 in [1, 2)) and T = U^{-1} instead of Q.
template <bool GY, bool FACT = false>
__global__ void __launch_bounds__(QR_THREADS, 1) qr_kernel(QrArgs a)
{
    extern __shared__ double sm[];
    __shared__ double pan_sc[QB][3];    // a panel's reflectors: tau, v_0, alpha
    __shared__ double pan_pc[QB + 1][QB];   // [i][ip]: entry of v_i in the panel's row ip > i (row QB: unused)
    __shared__ double pan_rr[QB + 1][QB];   // [i][q]: R[j0 + i][j0 + q], q > i (row QB: unused)
    __shared__ int pan_stop;            // the panel ends before this reflector
    const int k = a.k;
    const int ld = k | 1;   // odd row pitch: a warp reading one column of 16 rows hits 16 distinct bank pairs
    const int c = blockIdx.x;
    const int r0 = c * a.rows_per;
    const int r1 = min(a.n, r0 + a.rows_per);
    const int nr = max(0, r1 - r0);
    const int tid = threadIdx.x;
    double *Ys = GY ? a.yslab + (size_t)c * a.rows_per * ld : sm;   // rows_per x ld
    double *taus = GY ? sm : Ys + (size_t)a.rows_per * ld;          // k
    double *v0s = taus + k;                         // k
    double *alps = v0s + k;                         // k
    double *Gs = alps + k;                          // QB x k: panel Gram rows
    double *Ps = Gs + QB * k;                       // QB x k: panel rows
    double *cfs = Ps + QB * k;                      // QB x k: tau_j v_j^T a_kk
    // (after the factorisation the region from Gs on holds the triangular solve's buffers)
    const bool det = a.gpart != nullptr;
    // atomics: three rotating accumulators; deterministic: this CTA's slot of panel parity blk
    auto acc_buf = [&](int blk) {
        return det ? a.gpart + ((size_t)(blk & 1) * a.G + c) * QB * k : a.sbuf + (size_t)(blk % 3) * QB * k;
    };
    auto pub_buf = [&](int blk) { return a.rowbuf + (size_t)(blk & 1) * QB * k; };

    const int pitch = FACT ? a.pitch : k;
    for (int t = tid; t < nr * k; t += blockDim.x)
        Ys[(t / k) * ld + t % k] = FACT ? a.Y[(size_t)(r0 + t / k) * pitch + t % k] : a.Y[(size_t)r0 * k + t];
    __syncthreads();

    // The sweep of gram_pass below over the columns kk >= j1: P lanes per column share its rows
    // from local row rs on, two at a time (two independent chains keep the FP64 pipe busy).
    auto sweep = [&](int j0, int nb, int j1, int nn, int rs, int P, double *acc, double *pub, auto full) {
        constexpr bool FULL = decltype(full)::value;
        const int ncols = k - j1, nrow = max(0, nr - rs);
        const int lg = 31 - __clz(P);
        auto row_of = [&](int r) { return Ys + (size_t)r * ld; };
        for (int base = 0; base < ncols * P; base += blockDim.x) {
            const int t = base + tid;
            const int kk = j1 + (t >> lg), part = t & (P - 1);
            double g[QB];
#pragma unroll
            for (int i = 0; i < QB; ++i) g[i] = 0.0;
            if (t < ncols * P) {
                const bool upd = (FULL || nb > 0) && kk >= j1 + nn;
                double cf[QB];
#pragma unroll
                for (int i = 0; i < QB; ++i) cf[i] = (upd && (FULL || i < nb)) ? cfs[i * k + kk] : 0.0;
                int r = rs + part;
                // pairs of rows; the columns of the next panel are updated already (cf = 0)
                for (; r + P < nr; r += 2 * P) {
                    double *ra = row_of(r), *rb = row_of(r + P);
                    double x = ra[kk], y = rb[kk];
                    if (upd) {
                        double v[QB], w[QB];
#pragma unroll
                        for (int i = 0; i < QB; ++i)
                            if (FULL || i < nb) {
                                v[i] = ra[j0 + i];
                                w[i] = rb[j0 + i];
                            }
#pragma unroll
                        for (int i = 0; i < QB; ++i)
                            if (FULL || i < nb) {
                                x = fma(-v[i], cf[i], x);
                                y = fma(-w[i], cf[i], y);
                            }
                        ra[kk] = x;
                        rb[kk] = y;
                    }
#pragma unroll
                    for (int i = 0; i < QB; ++i)
                        if (FULL || i < nn) g[i] = fma(ra[j1 + i], x, g[i]);
#pragma unroll
                    for (int i = 0; i < QB; ++i)
                        if (FULL || i < nn) g[i] = fma(rb[j1 + i], y, g[i]);
                    const int rg = r0 + r;
                    if (rg < j1 + nn) pub[(rg - j1) * k + kk] = x;
                    if (rg + P < j1 + nn) pub[(rg + P - j1) * k + kk] = y;
                }
                if (r < nr) {
                    double *ra = row_of(r);
                    double x = ra[kk];
                    if (upd) {
#pragma unroll
                        for (int i = 0; i < QB; ++i)
                            if (FULL || i < nb) x = fma(-ra[j0 + i], cf[i], x);
                        ra[kk] = x;
                    }
#pragma unroll
                    for (int i = 0; i < QB; ++i)
                        if (FULL || i < nn) g[i] = fma(ra[j1 + i], x, g[i]);
                    if (r0 + r < j1 + nn) pub[(r0 + r - j1) * k + kk] = x;
                }
            }
            // Combine the P lanes of a column by halving: at each of the first three levels a lane
            // keeps half of its sums and hands over the other half, 4 + 2 + 1 additions instead of
            // 8 per level; the sums then sit on different lanes and so do their atomics.
            int i0 = 0;
            if (P >= 2) {
                const bool up = part & 1;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const double o = __shfl_xor_sync(0xffffffffu, up ? g[i] : g[i + 4], 1);
                    g[i] = (up ? g[i + 4] : g[i]) + o;
                }
                i0 = up ? 4 : 0;
            }
            if (P >= 4) {
                const bool up = part & 2;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const double o = __shfl_xor_sync(0xffffffffu, up ? g[i] : g[i + 2], 2);
                    g[i] = (up ? g[i + 2] : g[i]) + o;
                }
                i0 += up ? 2 : 0;
            }
            if (P >= 8) {
                const bool up = part & 4;
                const double o = __shfl_xor_sync(0xffffffffu, up ? g[0] : g[1], 4);
                g[0] = (up ? g[1] : g[0]) + o;
                i0 += up ? 1 : 0;
            }
            if (P >= 16) g[0] += __shfl_xor_sync(0xffffffffu, g[0], 8);
            if (P >= 32) g[0] += __shfl_xor_sync(0xffffffffu, g[0], 16);
            const int held = P >= 8 ? 1 : QB >> lg;
#pragma unroll
            for (int i = 0; i < QB; ++i) {
                if (i >= held) break;
                const int ii = i0 + i;
                if (t >= ncols * P || (part >> 3) != 0 || ii >= nn) continue;
                // deterministic: every entry of the panel's rows in this CTA's slot, zero where the
                // CTA has no rows below the panel
                if (det) acc[ii * k + kk] = (nrow > 0 && j1 + ii <= kk) ? g[i] : 0.0;
                else if (nrow > 0 && j1 + ii <= kk) atomicAdd(&acc[ii * k + kk], g[i]);
            }
        }
    };

    // Apply the reflectors of the panel at j0 (width nb, coefficients cfs, vectors
    // in the panel columns) to this CTA's rows >= j1 and form the partial Gram
    // rows of the panel at j1 (width nn) over those rows; the owners of rows
    // j1 .. j1+nn-1 publish them.  Panel columns j1 .. j1+nn-1 are updated first
    // (one thread per element), then every column kk >= j1 is swept once: P lanes
    // split its rows, the update is a sum of nb independent terms and the nn Gram
    // sums are independent chains; partial sums meet through FP64 atomics.
    auto gram_pass = [&](int j0, int nb, int j1, int nn, double *acc, double *pub) {
        const int rs = max(r0, j1) - r0;   // first local row >= j1
        const int nrow = max(0, nr - rs);
        if (nb > 0) {
            for (int t = tid; t < nrow * nn; t += blockDim.x) {
                const int r = rs + t / nn, col = j1 + t % nn;
                double *row = Ys + (size_t)r * ld;
                double v[QB], cf[QB], x = row[col];
#pragma unroll
                for (int i = 0; i < QB; ++i) {
                    v[i] = i < nb ? row[j0 + i] : 0.0;
                    cf[i] = i < nb ? cfs[i * k + col] : 0.0;
                }
#pragma unroll
                for (int i = 0; i < QB; ++i)
                    if (i < nb) x = fma(-v[i], cf[i], x);
                row[col] = x;
            }
            __syncthreads();
        }
        const int ncols = k - j1;
        // Lanes per column, from what the busiest sub-partition issues: 2 QB multiply-adds per row
        // of a lane (update and Gram sums) and about log2(P) + 6 instructions to combine lanes;
        // measured per instruction: ~98 cycles with one warp on the sub-partition, 66 with more.
        // Rows in the slab come from L2, whose latency wants every warp.
        int P = 1;
        if (GY) {
            while (P < 32 && P * 2 * ncols <= (int)blockDim.x) P *= 2;
        } else {
            int best = 1 << 30;
            for (int lg = 0; lg <= 5 && (ncols << lg) <= 2 * (int)blockDim.x; ++lg) {
                const int w = ((ncols << lg) + 127) >> 7;
                const int cost = (w == 1 ? 3 : 2 * w) * (2 * QB * ((nrow + (1 << lg) - 1) >> lg) + (lg ? lg + 6 : 0));
                if (cost < best) {
                    best = cost;
                    P = 1 << lg;
                }
            }
        }
        // full panels (all but a restart's and the last one's) take straight-line code
        if (nb == QB && nn == QB) sweep(j0, QB, j1, QB, rs, P, acc, pub, std::true_type());
        else sweep(j0, nb, j1, nn, rs, P, acc, pub, std::false_type());
    };

    int j0 = 0, nn0 = min(QB, k), blk = 0;
    unsigned ep = 0;   // grid barriers passed
    gram_pass(0, 0, 0, nn0, acc_buf(0), pub_buf(0));
    while (j0 < k) {
        const double *acc = acc_buf(blk);
        const double *pub = pub_buf(blk);
        if (!grid_barrier(a.bar, a.G, ++ep, a.err, a.bar_extra, a.spin_limit)) return;
        if (det) {
            // the G partial sums of each entry added in a fixed order, the entries shared
            // out over the CTAs, into a.sbuf; one more barrier publishes them
            const double *slots = a.gpart + (size_t)(blk & 1) * a.G * QB * k;
            const int ne = nn0 * (k - j0), lane = tid & 31, part = tid % DET_LANES;
            // entries by groups of lanes; whole warps iterate together (the groups shuffle)
            for (int wb = c * blockDim.x + tid - lane; wb < ne * DET_LANES; wb += a.G * blockDim.x) {
                const int u = wb + lane;
                const int t = min(u / DET_LANES, ne - 1);
                const int i = t / (k - j0), kk = j0 + t % (k - j0);
                const double v = det_sum(slots + i * k + kk, (size_t)QB * k, a.G, part);
                if (part == 0 && u / DET_LANES < ne && kk >= j0 + i) a.sbuf[i * k + kk] = v;
            }
            if (!grid_barrier(a.bar, a.G, ++ep, a.err, a.bar_extra, a.spin_limit)) return;
        }
        for (int t = tid; t < nn0 * (k - j0); t += blockDim.x) {
            const int i = t / (k - j0), kk = j0 + t % (k - j0);
            double gv = 0.0;
            if (kk >= j0 + i) gv = det ? __ldcg(a.sbuf + i * k + kk) : ((volatile const double *)acc)[i * k + kk];
            Gs[i * k + kk] = gv;
            Ps[i * k + kk] = ((volatile const double *)pub)[i * k + kk];
        }
        if (c == 0 && !det) {
            double *z = a.sbuf + (size_t)((blk + 2) % 3) * QB * k;
            for (int t = tid; t < QB * k; t += blockDim.x) z[t] = 0.0;
        }
        if (tid == 0) pan_stop = -1;
        __syncthreads();
        // ------------------------------------------------ the panel's reflectors
        // Warp 0 derives them from the panel's QB x QB blocks of G and P alone, a column after
        // the other: alpha = -sign(x_0)|x|, v_0 = x_0 - alpha, tau = 1 / (|x| (|x| + |x_0|)),
        // then cf = tau v^T a and R's entries of the panel's later columns, and both blocks
        // downdated.  Lane (r, q) holds rows r and r + 4 of column q of each block.  As soon as
        // a reflector is published (shared memory, named barrier i + 1), the outer warps apply
        // it to their columns kk >= j0 + nn0 -- cf, R and the downdates of the column's QB
        // entries of G and P, in registers -- while warp 0 works on the next one.  The chain
        // per column is one pair of Householder scalars and about eight FP64 instructions; the
        // two-barrier pass over all columns it replaces took 23k cycles a panel at k = 72.
        const int warp = tid >> 5, lane = tid & 31;
        const int jo = j0 + nn0, nout = k - jo;       // outer columns
        const bool pairs = nout <= 64;                // two lanes per column: one G, one P
        const int cpw = pairs ? 16 : 32;
        // outer warps, and behind them the row warps, are the warps off warp 0's sub-partition
        constexpr int OTHERS = 3 * (QR_THREADS >> 5) / 4;
        const int rs = max(r0, jo) - r0, nrw = (max(0, nr - rs) + 31) / 32;   // rows below the panel
        const bool pipe_rows = !GY && nrw <= OTHERS / 2;
        const int now = min((nout + cpw - 1) / cpw, OTHERS - (pipe_rows ? nrw : 0));
        const int bar_n = 32 * (now + (pipe_rows ? nrw : 0) + 1);
        const int wi = (warp & 3) ? warp - 1 - (warp >> 2) : -1;   // index among those warps
        if (warp == 0) {
            const int r = lane >> 3, q = lane & 7;
            double P0 = 0.0, P1 = 0.0, G0 = 0.0, G1 = 0.0;
            if (q < nn0 && r < nn0) {
                P0 = Ps[r * k + j0 + q];
                G0 = Gs[r * k + j0 + q];
            }
            if (q < nn0 && r + 4 < nn0) {
                P1 = Ps[(r + 4) * k + j0 + q];
                G1 = Gs[(r + 4) * k + j0 + q];
            }
            int stop = nn0;
            // One copy of the loop body: unrolled, its instructions would come from beyond the
            // instruction cache once per panel (measured: the scalars 910 instead of 590 cycles).
            // Signs and ranges are tested on the bit patterns: an FP64 compare costs as much as
            // an FMA.  While rows 0 .. 3 are still wanted, the downdate of rows 4 .. 7 waits until
            // the next column's scalars are under way (pend).
            const double fresh = q < nn0 ? Gs[q * k + j0 + q] : 0.0;   // the norms at the panel's start
            bool pend = false;
            double cf = 0.0, rv = 0.0, pc1 = 0.0, rr1 = 0.0;
#pragma unroll 1
            for (int i = 0; i < nn0; ++i) {
                const int j = j0 + i, src = ((i & 3) << 3) | i;
                const double nrm2 = __shfl_sync(0xffffffffu, i < 4 ? G0 : G1, src);
                const double x0 = __shfl_sync(0xffffffffu, i < 4 ? P0 : P1, src);
                const long long nb2 = __double_as_longlong(nrm2);
                // cancellation (or NaN): the panel ends here and the next one starts from fresh sums
                const long long least = __double_as_longlong(__shfl_sync(0xffffffffu, fresh, i)) - ((long long)QR_DOWNDATE_LOG2 << 52);
                if (i > 0 && !(nb2 >= least && nb2 <= 0x7FF0000000000000LL && nb2 > 0)) {
                    stop = i;
                    break;
                }
                const double gi = __shfl_sync(0xffffffffu, i < 4 ? G0 : G1, ((i & 3) << 3) | q);
                const double pi = __shfl_sync(0xffffffffu, i < 4 ? P0 : P1, ((i & 3) << 3) | q);
                double tau = 0.0, alpha = 0.0, v0 = 0.0;
                if (nb2 > 0) {
                    const HouseholderScalars h = householder_scalars(nrm2, fabs(x0));
                    alpha = __hiloint2double(__double2hiint(h.nrm) | (~__double2hiint(x0) & (int)0x80000000),
                                             __double2loint(h.nrm));
                    v0 = x0 - alpha;
                    tau = h.beta;
                }
                if (pend) {
                    G1 = fma(-rr1, rv, G1);
                    P1 = fma(-pc1, cf, P1);
                    pend = false;
                }
                cf = tau * fma(-alpha, pi, gi);
                rv = fma(-v0, cf, pi);
                // every lane stores (equal values meet at equal addresses): no divergent branches
                pan_sc[i][0] = tau;
                pan_sc[i][1] = v0;
                pan_sc[i][2] = alpha;
                pan_pc[q == i ? i : QB][r] = P0;
                pan_pc[q == i ? i : QB][r + 4] = P1;
                pan_rr[i][q] = rv;
                *(q > i && q < nn0 ? cfs + i * k + j0 + q : &pan_rr[QB][0]) = cf;
                if (bar_n > 32) {
                    __syncwarp();
                    asm volatile("bar.arrive %0, %1;" ::"r"(i + 1), "r"(bar_n) : "memory");
                }
                pc1 = __shfl_sync(0xffffffffu, P1, (r << 3) | i);
                rr1 = __shfl_sync(0xffffffffu, rv, r + 4);
                if (i < 3) {
                    const double pc = __shfl_sync(0xffffffffu, P0, (r << 3) | i), rr = __shfl_sync(0xffffffffu, rv, r);
                    G0 = fma(-rr, rv, G0);
                    P0 = fma(-pc, cf, P0);
                    pend = true;
                } else {
                    G1 = fma(-rr1, rv, G1);
                    P1 = fma(-pc1, cf, P1);
                }
                if (lane == 0) {
                    taus[j] = tau;
                    v0s[j] = v0;
                    alps[j] = alpha;
                }
                if (c == 0) {
                    for (int kk = lane; kk < j0; kk += 32) a.R[(size_t)j * pitch + kk] = 0.0;
                    if (r == 0 && q < nn0) a.R[(size_t)j * pitch + j0 + q] = q < i ? 0.0 : (q == i ? alpha : rv);
                }
            }
            if (lane == 0) pan_stop = stop;
            if (stop < nn0 && bar_n > 32) {
                __syncwarp();
                asm volatile("bar.arrive %0, %1;" ::"r"(stop + 1), "r"(bar_n) : "memory");
            }
        } else if (wi >= now && wi < now + nrw && pipe_rows) {
            // rows below the panel: v_i's entries take the in-panel updates, one thread per row
            const int rl = rs + (wi - now) * 32 + lane;
            double *row = Ys + (size_t)min(rl, nr - 1) * ld + j0;
            double v[QB];
#pragma unroll
            for (int i = 0; i < QB; ++i) v[i] = i < nn0 ? row[i] : 0.0;
            int done = nn0;
#pragma unroll
            for (int i = 0; i < QB; ++i) {
                if (i >= nn0) break;
                asm volatile("bar.sync %0, %1;" ::"r"(i + 1), "r"(bar_n) : "memory");
                if (*(volatile int *)&pan_stop == i) {
                    done = i;
                    break;
                }
#pragma unroll
                for (int ip = i + 1; ip < QB; ++ip)
                    if (ip < nn0) v[ip] = fma(-v[i], cfs[i * k + j0 + ip], v[ip]);
            }
            if (rl < nr) {
#pragma unroll
                for (int i = 1; i < QB; ++i)
                    if (i < done) row[i] = v[i];
            }
        } else if (wi >= 0 && wi < now) {
            // columns kk, then (more than the warps hold) a second sweep with nothing to wait for
            for (int sweep = 0, base = wi * cpw; base < nout; ++sweep, base += now * cpw) {
                const int kk = jo + base + (pairs ? lane >> 1 : lane);
                const bool in = kk < k, isg = pairs && (lane & 1);
                double p[QB], g[QB];   // pairs: p holds this lane's entries (of G or of P)
#pragma unroll
                for (int i = 0; i < QB; ++i) {
                    const bool have = in && i < nn0;
                    p[i] = have ? (isg ? Gs : Ps)[i * k + kk] : 0.0;
                    g[i] = have && !pairs ? Gs[i * k + kk] : 0.0;
                }
#pragma unroll
                for (int i = 0; i < QB; ++i) {
                    if (i >= nn0) break;
                    if (sweep == 0) asm volatile("bar.sync %0, %1;" ::"r"(i + 1), "r"(bar_n) : "memory");
                    if (*(volatile int *)&pan_stop == i) break;
                    const double tau = pan_sc[i][0], v0 = pan_sc[i][1], alpha = pan_sc[i][2];
                    double pi = p[i], gi = g[i];
                    if (pairs) {
                        const double o = __shfl_xor_sync(0xffffffffu, pi, 1);
                        gi = isg ? pi : o;
                        pi = isg ? o : pi;
                    }
                    const double cf = tau * fma(-alpha, pi, gi);
                    const double rv = fma(-v0, cf, pi);
                    if (in && !isg) cfs[i * k + kk] = cf;
                    if (in && (isg || !pairs) && c == 0) a.R[(size_t)(j0 + i) * pitch + kk] = rv;
                    if (pairs) {
                        const double mul = isg ? rv : cf;
#pragma unroll
                        for (int ip = i + 1; ip < QB; ++ip)
                            p[ip] = fma(-(isg ? pan_rr[i][ip] : pan_pc[i][ip]), mul, p[ip]);
                    } else {
#pragma unroll
                        for (int ip = i + 1; ip < QB; ++ip) {
                            p[ip] = fma(-pan_pc[i][ip], cf, p[ip]);
                            g[ip] = fma(-pan_rr[i][ip], rv, g[ip]);
                        }
                    }
                }
            }
        }
        __syncthreads();
        const int nb = pan_stop;
        const int j1 = j0 + nb;
        // reflector entries of the panel's own rows (below the diagonal) come from the panel
        // block; the rows below it had the in-panel updates above, or get them here where they
        // were too many for that (one thread per row, in registers)
        for (int t = tid; t < nn0 * nb; t += blockDim.x) {
            const int ip = t / nb, i = t % nb;
            const int rg = j0 + ip;
            if (i < ip && rg >= r0 && rg < r1) Ys[(size_t)(rg - r0) * ld + j0 + i] = pan_pc[i][ip];
        }
        if (!pipe_rows)
            for (int r = rs + tid; r < nr; r += blockDim.x) {
                double v[QB];
#pragma unroll
                for (int i = 0; i < QB; ++i) v[i] = (i < nb) ? Ys[(size_t)r * ld + j0 + i] : 0.0;
#pragma unroll
                for (int i = 0; i < QB; ++i)
#pragma unroll
                    for (int ip = i + 1; ip < QB; ++ip)
                        if (ip < nb) v[ip] = fma(-v[i], cfs[i * k + j0 + ip], v[ip]);
#pragma unroll
                for (int i = 1; i < QB; ++i)
                    if (i < nb) Ys[(size_t)r * ld + j0 + i] = v[i];
            }
        __syncthreads();
        const int nn1 = min(QB, k - j1);
        if (j1 < k) gram_pass(j0, nb, j1, nn1, acc_buf(blk + 1), pub_buf(blk + 1));
        j0 = j1;
        nn0 = nn1;
        ++blk;
    }

    // ---------------------------------------------------------- Q = E - V W, gauge
    // V rows of this CTA in place (v_j is 0 above row j, v0 on the diagonal, 0 where
    // tau = 0); the first k rows also go to global memory for the triangular solve.
    __syncthreads();
    for (int t = tid; t < nr * k; t += blockDim.x) {
        const int rl = t / k, j = t % k, rg = r0 + rl;
        double v = 0.0;
        if (rg == j) v = v0s[j];
        else if (rg > j) v = Ys[rl * ld + j];
        if (taus[j] == 0.0) v = 0.0;
        if (FACT) {
            // 2^-exponent(v_0), v_0 being the column's largest entry: the reflector is the same, and
            // the trailing update's row grids see columns of one size
            const int e = (__double2hiint(v0s[j]) >> 20) & 0x7FF;
            v = e > 0 && e < 2046 ? v * __hiloint2double((2046 - e) << 20, 0) : v;
            a.V[(size_t)rg * pitch + j] = v;
        }
        Ys[rl * ld + j] = v;
        if (!FACT && rg < k) a.V[(size_t)rg * k + j] = v;
    }
    if (FACT && c == 0)
        for (int j = tid; j < k; j += blockDim.x) {
            a.taus[j] = taus[j];
            a.sgn[j] = alps[j] < 0.0 ? -1.0 : 1.0;
        }
    if (FACT && !a.S) return;   // a lone panel: its S and W are the whole matrix's
    if (!FACT && c == 0) {
        __syncthreads();
        for (int t = tid; t < k * k; t += blockDim.x) {
            int rr = t / k;
            if (alps[rr] < 0.0) a.R[t] = -a.R[t];
        }
    }
    __syncthreads();
    // S = V^T V (upper triangle): this CTA's rows, two chains per entry, summed over
    // the CTAs with FP64 atomics
    // (rows i and k-1-i of the triangle together have k+1 entries: no lane idles)
    for (int e = tid; e < (k + 1) / 2 * (k + 1); e += blockDim.x) {
        const int a0 = e / (k + 1), f = e % (k + 1);
        const bool first = f < k - a0;
        const int i = first ? a0 : k - 1 - a0, j = first ? a0 + f : f - 1;
        if (!first && i == a0) continue;   // the middle row of an odd k is listed once
        const int rs = max(0, j - r0);
        if (rs >= nr) continue;
        double s0 = 0.0, s1 = 0.0;
        int rl = rs;
        for (; rl + 1 < nr; rl += 2) {
            s0 = fma(Ys[rl * ld + i], Ys[rl * ld + j], s0);
            s1 = fma(Ys[(rl + 1) * ld + i], Ys[(rl + 1) * ld + j], s1);
        }
        if (rl < nr) s0 = fma(Ys[rl * ld + i], Ys[rl * ld + j], s0);
        if (det) a.spart[(size_t)c * k * k + (size_t)i * k + j] = s0 + s1;
        else atomicAdd(&a.S[(size_t)i * k + j], s0 + s1);
    }
    if (det) {
        // slots of CTAs without rows at or below column j hold no entry: zero them
        for (int e = tid; e < k * k; e += blockDim.x) {
            const int i = e / k, j = e % k;
            if (j >= i && max(0, j - r0) >= nr) a.spart[(size_t)c * k * k + e] = 0.0;
        }
        if (!grid_barrier(a.bar, a.G, ++ep, a.err, a.bar_extra, a.spin_limit)) return;
        // S = the G partials in a fixed order, each CTA a share of the entries
        const int lane = tid & 31, part = tid % DET_LANES;
        for (int wb = c * blockDim.x + tid - lane; wb < k * k * DET_LANES; wb += a.G * blockDim.x) {
            const int u = wb + lane;
            const int e = min(u / DET_LANES, k * k - 1);
            const double v = det_sum(a.spart + e, (size_t)k * k, a.G, part);
            if (part == 0 && u / DET_LANES < k * k && e % k >= e / k) a.S[e] = v;
        }
    }
    if (!grid_barrier(a.bar, a.G, ++ep, a.err, a.bar_extra, a.spin_limit)) return;
    for (int cb = c; cb < (k + QR_WC - 1) / QR_WC; cb += a.G) {   // a small grid solves several blocks
        const double *V = FACT ? nullptr : a.V;
        if (wy_packed(k)) wy_solve_cta<true>(k, cb, a.S, V, taus, a.W, Gs);
        else wy_solve_cta<false>(k, cb, a.S, V, taus, a.W, Gs);
        __syncthreads();
    }
    if (FACT) return;
    if (!grid_barrier(a.bar, a.G, ++ep, a.err, a.bar_extra, a.spin_limit)) return;
    // Q rows of this CTA: (E - V W) with column c negated where alpha_c < 0; a thread owns one
    // column and the same number of rows, known at compile time, in every pass: a predicated-off
    // FP64 instruction takes the pipe as long as one that runs
    {
        const int grp = blockDim.x / k;
        const int share = (nr + grp - 1) / grp;
        if (share <= 1) q_rows<1>(a, alps, Ys, ld, r0, nr);
        else if (share <= 2) q_rows<2>(a, alps, Ys, ld, r0, nr);
        else if (share <= 3) q_rows<3>(a, alps, Ys, ld, r0, nr);
        else if (share <= 4) q_rows<4>(a, alps, Ys, ld, r0, nr);
        else if (share <= 6) q_rows<6>(a, alps, Ys, ld, r0, nr);
        else q_rows<8>(a, alps, Ys, ld, r0, nr);
    }
}

size_t qr_smem_bytes(int rows_per, int k, bool slab)
{
    const size_t panel = 3 * (size_t)QB * k;
    const size_t solve = qr_wy_smem_bytes(k) / sizeof(double);
    return sizeof(double) * ((slab ? 0 : (size_t)rows_per * (k | 1)) + 3 * (size_t)k +
                             (panel > solve ? panel : solve));
}

// Rows per CTA and the grid.  The kernel holds one CTA per SM (512 threads at ~100
// registers), so the grid never exceeds the SM count: a floor rows_min above
// ceil(n / #SM) that would not fit shared memory gives way down to ceil(n / #SM), and
// where even that block does not fit, the row blocks go to a global slab (*slab_out).
// A slab grid leaves two SMs free: the corner spectrum of the previous step, which
// runs for milliseconds at such sizes and holds an SM, must not keep a CTA of the
// grid-synchronous factorisation waiting.  Returns 0 when the kernel's other shared
// memory does not fit either.
int qr_layout(int n, int k, int rows_min, int *G_out, int *rows_out, bool *slab_out = nullptr, bool force_slab = false)
{
    const int sms = device_sm_count();
    int base = (n + sms - 1) / sms;
    if (base < 1) base = 1;
    int rows_per = rows_min > base ? rows_min : base;
    while (rows_per > base && qr_smem_bytes(rows_per, k, false) > QR_SMEM_MAX) {
        rows_per = (rows_per * 3) / 4;
        if (rows_per < base) rows_per = base;
    }
    const bool slab = force_slab || qr_smem_bytes(rows_per, k, false) > QR_SMEM_MAX;
    if (slab && sms > 4) rows_per = (n + sms - 3) / (sms - 2);
    *G_out = (n + rows_per - 1) / rows_per;
    *rows_out = rows_per;
    if (slab_out) *slab_out = slab;
    return qr_smem_bytes(rows_per, k, slab) <= QR_SMEM_MAX;
}

}  // namespace

size_t qr_scratch_doubles(int k) { return (size_t)3 * QB * k + 8; }
size_t qr_det_gram_doubles(int k, int gmax) { return (size_t)2 * gmax * QB * k; }
size_t qr_det_s_doubles(int k, int gmax) { return (size_t)gmax * k * k; }
int qr_det_gmax(int n) { return n < QR_DET_GMAX ? n : QR_DET_GMAX; }
size_t qr_rowbuf_doubles(int k) { return (size_t)2 * QB * k; }

size_t qr_slab_doubles(int n, int k, bool force)
{
    int G, rp;
    bool slab = false;
    if (n < k || k < 1 || k > QR_MAX_COLS || !qr_layout(n, k, 1, &G, &rp, &slab, force) || !slab) return 0;
    return (size_t)G * rp * (k | 1);
}

bool qr_force_slab_from_env()
{
    const char *e = getenv("CTM_QR_SLAB");
    return e && e[0] == '1';
}

int qr_supported(int n, int k)
{
    int G, rp;
    return n >= k && k >= 1 && k <= QR_MAX_COLS && qr_layout(n, k, 1, &G, &rp);
}

size_t qr_sk_doubles(int n, int k)
{
    (void)n;
    (void)k;
    return 0;
}

size_t qr_wy_doubles(int n, int k) { return (size_t)k * k + 3 * (size_t)k * k + 2 * (size_t)k; }

// The accumulators and the barrier count before a factorisation: one launch for all three (three
// memset nodes and the gaps between them took 3 to 6 us more of a step)
__global__ void qr_zero_kernel(int nsbuf, double *sbuf, int ns, double *S, unsigned *bar)
{
    const int t0 = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    for (int t = t0; t < nsbuf; t += nt) sbuf[t] = 0.0;
    for (int t = t0; t < ns; t += nt) S[t] = 0.0;
    if (t0 < 2) bar[t0] = 0;
}

// pitch > 0: one panel of the blocked factorisation (Q unused; V, R in the wider matrices)
static cudaError_t qr_factor_launch(int n, int k, int rows_per, const double *Y, double *Q, double *R, QrScratch s,
                                    cudaStream_t st, int pitch = 0, double *taus = nullptr, double *sgn = nullptr)
{
    const int G = (n + rows_per - 1) / rows_per;
    const bool slab = pitch == 0 && (s.force_slab || qr_smem_bytes(rows_per, k, false) > QR_SMEM_MAX);
    if (slab && (!s.yslab || s.yslab_elems < (size_t)G * rows_per * (k | 1))) return cudaErrorInvalidValue;
    const size_t smem = qr_smem_bytes(rows_per, k, slab);
    if (smem > QR_SMEM_MAX) return cudaErrorInvalidValue;
    void (*kern)(QrArgs) = pitch > 0 ? qr_kernel<false, true> : slab ? qr_kernel<true> : qr_kernel<false>;
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, QR_THREADS, smem);
    if (per_sm * device_sm_count() < G) return cudaErrorCooperativeLaunchTooLarge;
    if (s.gpart && (!s.spart || G > s.gmax)) return cudaErrorInvalidValue;
    const int zb = (k * k + 1023) / 1024;
    CTM_COUNT_LAUNCH(1);
    qr_zero_kernel<<<zb < device_sm_count() ? zb : device_sm_count(), 256, 0, st>>>(3 * QB * k, s.sbuf, s.S ? k * k : 0,
                                                                                 s.S, s.bar);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    QrArgs a{n, k, G, rows_per, Y, R, Q, s.V, s.S, s.W, s.sbuf, s.rowbuf, s.bar, s.err, s.bar_extra,
             s.spin_limit > 0 ? s.spin_limit : QR_SPIN_LIMIT, s.gpart, s.spart, slab ? s.yslab : nullptr, pitch, taus,
             sgn};
    void *args[] = {&a};
    CTM_COUNT_LAUNCH(1);
    return cudaLaunchCooperativeKernel((void *)kern, dim3(G), dim3(QR_THREADS), args, smem, st);
}

#include <map>
#include <mutex>
#include <utility>
#include <vector>
static std::mutex g_qr_mu;
static std::map<std::pair<int, int>, int> g_qr_rows;   // (n, k) -> rows per CTA, for rows_min == 1

// rows per CTA: tuned once per (n, k) by timing the factorisation (eager calls only)
static int qr_pick_rows(int n, int k, const double *Y, double *Q, double *R, QrScratch s, cudaStream_t st)
{
    int G, rp0;
    bool slab = false;
    qr_layout(n, k, s.rows_min > 0 ? s.rows_min : 1, &G, &rp0, &slab, s.force_slab);
    if (s.rows_min > 1 || s.bar_extra || slab) return rp0;   // slab: one block per SM, nothing to tune
    {
        std::lock_guard<std::mutex> lk(g_qr_mu);
        auto it = g_qr_rows.find({n, k});
        if (it != g_qr_rows.end()) return it->second;
    }
    const int tkey[2] = {n, k};
    int tval = 0;
    int per_sm = 0;
    if (tune_cache_lookup("qr", tkey, 2, &tval, 1) && tval >= 1 && qr_smem_bytes(tval, k, false) <= QR_SMEM_MAX &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, qr_kernel<false>, QR_THREADS,
                                                      qr_smem_bytes(tval, k, false)) == cudaSuccess &&
        (long long)per_sm * device_sm_count() >= (n + tval - 1) / tval) {
        std::lock_guard<std::mutex> lk(g_qr_mu);
        g_qr_rows[{n, k}] = tval;
        return tval;
    }
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(st, &cs);
    if (cs != cudaStreamCaptureStatusNone) return rp0;
    int best = rp0;
    float best_ms = 1e30f;
    std::vector<std::pair<int, float>> timed;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return rp0;
    // fewer rows than rp0 puts several CTAs on an SM (the launch checks they all fit)
    for (int rp : {rp0, 8, 12, 16, 24, 32, 48, 64, 96, 128}) {
        if ((rp < rp0 && rp * 2 < rp0) || (rp != rp0 && rp < 8) || qr_smem_bytes(rp, k, false) > QR_SMEM_MAX)
            continue;
        float ms = 1e30f;
        for (int rep = 0; rep < 4; ++rep) {   // first run warms up; the fastest of three counts
            float t = 0.f;
            cudaEventRecord(e0, st);
            cudaError_t e = qr_factor_launch(n, k, rp, Y, Q, R, s, st);
            cudaEventRecord(e1, st);
            if (e != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess) {
                ms = 1e30f;
                cudaGetLastError();
                break;
            }
            cudaEventElapsedTime(&t, e0, e1);
            if (rep && t < ms) ms = t;
        }
        int herr = 0;
        cudaMemcpy(&herr, s.err, sizeof(int), cudaMemcpyDeviceToHost);
        if (herr) break;   // a bounded wait expired: keep the default, the caller will report it
        if (ms < best_ms) {
            best_ms = ms;
            best = rp;
        }
        timed.emplace_back(rp, ms);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    // Timed alone, grids of 108 and 144 CTAs tie at n = 2592, k = 72; inside the step the
    // corner spectrum's kernels run beside the QR, and the 144-CTA grid left them 8 SMs and
    // made the step 8 % slower.  So take the fewest CTAs (most rows) within 3 % of the fastest.
    for (auto &t : timed)
        if (t.second <= 1.03f * best_ms && t.first > best) best = t.first;
    {
        std::lock_guard<std::mutex> lk(g_qr_mu);
        g_qr_rows[{n, k}] = best;
    }
    tune_cache_store("qr", tkey, 2, &best, 1);
    return best;
}

// ---------------------------------------------------------------- blocked, for many columns
// At k = 480 the one-launch factorisation is bound by the FP64 pipe: 4 n k^2 multiply-adds with Q
// formed, 13 ms at n = 12000.  Here panels of QR_NB columns (or all k in one) are factored by that kernel (FACT),
// and what is a contraction runs on the tensor cores as FP64 slices (gemm_split.cu, T = 8, whose
// error is below the FP64 sums'): the trailing update A -= V (A^T V T)^T of each panel, and, once
// all reflectors are known, S = V^T V and Q = E - V W with W = U^{-1} V_top^T as above.  The
// reflectors are scaled to one size (a power of two each) because the update's grids are per row
// of V.  With several panels A = Y is copied to Q's buffer and factored there, rows above the panel becoming R's.
constexpr int QR_NB = 64;   // an engine tile's K and N (48: 12000 x 480 4.52 ms against 4.31)

struct QrBlockedWork {
    double *V, *Z, *X, *taus, *sgn;
    SplitWork sw;
    size_t bytes;
};
static QrBlockedWork qr_blocked_work(int n, int k, int width, void *base_)
{
    QrBlockedWork w{};
    char *base = (char *)base_;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *p = base ? base + off : nullptr;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    w.V = (double *)take(sizeof(double) * (size_t)n * k);
    w.Z = (double *)take(sizeof(double) * (size_t)k * width);
    w.X = (double *)take(sizeof(double) * (size_t)k * width);
    w.taus = (double *)take(sizeof(double) * k);
    w.sgn = (double *)take(sizeof(double) * k);
    // A^T V and V X^T of the first panel, V^T V, V W: the largest of each operand
    const int shapes[4][3] = {{k, width, n}, {n, k, width}, {k, k, n}, {n, k, k}};
    for (auto &m : shapes) {
        const SplitPlan p = split_plan_caps(m[0], m[1], m[2], SPLIT_F64_T);
        if (p.a_pack_bytes > w.sw.a_pack_cap) w.sw.a_pack_cap = p.a_pack_bytes;
        if (p.b_pack_bytes > w.sw.b_pack_cap) w.sw.b_pack_cap = p.b_pack_bytes;
        if (p.partial_bytes > w.sw.partial_cap) w.sw.partial_cap = p.partial_bytes;
    }
    w.sw.e_cap = n;
    w.sw.Apk = (unsigned char *)take(w.sw.a_pack_cap);
    w.sw.Bpk = (unsigned char *)take(w.sw.b_pack_cap);
    w.sw.partial = take(w.sw.partial_cap + 8);
    w.sw.eA = (int *)take(sizeof(int) * (size_t)n);
    w.sw.eB = (int *)take(sizeof(int) * (size_t)n);
    w.bytes = off;
    return w;
}

// Columns 4b .. 4b + 3 of W = -U^{-1} V_top^T diag(sgn), so that Q = E diag(sgn) + V W has the gauge
__global__ void __launch_bounds__(QR_THREADS) qr_blocked_w_kernel(int k, const double *S, const double *V,
                                                                  const double *taus, const double *sgn, double *W)
{
    extern __shared__ double sm[];
    if (wy_packed(k)) wy_solve_cta<true>(k, blockIdx.x, S, V, taus, W, sm);
    else wy_solve_cta<false>(k, blockIdx.x, S, V, taus, W, sm);
    __syncthreads();
    for (int t = threadIdx.x; t < k * QR_WC; t += blockDim.x) {
        const int j = blockIdx.x * QR_WC + t % QR_WC;
        if (j < k) W[(size_t)(t / QR_WC) * k + j] *= -sgn[j];
    }
}
// R from the panels' blocks (in R) and the updated rows above them (in A), with the gauge
__global__ void qr_blocked_r_kernel(int k, int width, const double *A, const double *sgn, double *R)
{
    const int i = blockIdx.x;
    for (int j = threadIdx.x; j < k; j += blockDim.x) {
        const size_t o = (size_t)i * k + j;
        R[o] = j < i ? 0.0 : sgn[i] * (j / width == i / width ? R[o] : A[o]);
    }
}
__global__ void qr_blocked_diag_kernel(int k, const double *sgn, double *Q)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < k) Q[(size_t)j * k + j] += sgn[j];
}

// Rows per CTA of a panel: one CTA per SM, two SMs left free as for the slab
static int qr_panel_rows(int n, int rows_min)
{
    const int sms = device_sm_count(), g = sms > 4 ? sms - 2 : sms, base = (n + g - 1) / g;
    return base > rows_min ? base : rows_min;
}

// Where each form pays, by n k^2 (us: the kernel alone : one panel : 64-column panels).  Below
// 5e7 the kernel alone: 2592 x 72 225 : 318, 2048 x 128 434 : 462, 3000 x 120 449 : 447.  Then one
// panel, for S and Q by the engine: 6144 x 96 498 : 455, 4608 x 128 600 : 549, 8192 x 128
// 845 : 643, 1728 x 192 668 : 635 : 849, 4800 x 192 1153 : 870 : 1006, 6000 x 240 1969 : 1303 : 1348.
// From 3.9e8 panels: 6400 x 256 1492 (one panel) : 1433, 5120 x 320 1933 : 1766, 8000 x 320
// 4346 (kernel) : 2019, 4608 x 512 6589 : 2895, 12000 x 480 12928 : 4289.  |Y - QR| / |Y| there is
// 2e-16 to 6e-16 and |Q^T Q - 1| 8e-15 to 3.5e-14, by the kernel alone 4e-16 to 9e-16 and
// 1.4e-14 to 5.5e-14.
constexpr int QR_ONE_PANEL_MIN = 96;
constexpr double QR_ONE_PANEL_NK2 = 5e7, QR_PANELS_NK2 = 3.9e8;
// Panel width of the blocked form (k: one panel), or 0 for the one-launch kernel
static int qr_blocked_width(int n, int k, const QrScratch &s)
{
    if (!s.blocked || s.force_slab) return 0;
    const double nk2 = (double)n * k * k;
    if (k < QR_ONE_PANEL_MIN || nk2 < QR_ONE_PANEL_NK2) return 0;
    const int width = nk2 >= QR_PANELS_NK2 ? QR_NB : k;
    const int rows = qr_panel_rows(n, s.rows_min);
    if (qr_smem_bytes(rows, width, false) > QR_SMEM_MAX) return 0;
    if (s.gpart && (n + rows - 1) / rows > s.gmax) return 0;
    return qr_blocked_work(n, k, width, nullptr).bytes <= s.blocked_bytes ? width : 0;
}

static cudaError_t qr_blocked(int n, int k, int width, const double *Y, double *Q, double *R, QrScratch s,
                              cudaStream_t st)
{
    QrBlockedWork w = qr_blocked_work(n, k, width, s.blocked);
    w.sw.err = s.err;
    const bool lone = width >= k;   // one panel, read from Y itself
    double *A = Q;
    cudaError_t e = cudaSuccess;
    if (!lone) e = cudaMemcpyAsync(A, Y, sizeof(double) * (size_t)n * k, cudaMemcpyDeviceToDevice, st);
    if (!lone && e == cudaSuccess) e = cudaMemsetAsync(w.V, 0, sizeof(double) * (size_t)n * k, st);
    for (int j0 = 0; j0 < k && e == cudaSuccess; j0 += width) {
        const int nb = k - j0 < width ? k - j0 : width, m = n - j0, j1 = j0 + nb, rem = k - j1;
        double *Vp = w.V + (size_t)j0 * k + j0;
        QrScratch sp = s;
        sp.V = Vp;
        if (lone) sp.S = nullptr;
        e = qr_factor_launch(m, nb, qr_panel_rows(m, s.rows_min), lone ? Y : A + (size_t)j0 * k + j0, nullptr,
                             R + (size_t)j0 * k + j0, sp, st, k, w.taus + j0, w.sgn + j0);
        if (e != cudaSuccess || rem == 0) continue;
        double *At = A + (size_t)j0 * k + j1;
        // Z = A^T V, X = -Z T, A += V X^T
        e = gemm_split(GemmF64{rem, nb, m, At, idx_lin(1), idx_lin(k), Vp, idx_lin(k), idx_lin(1), w.Z, idx_lin(width),
                               idx_lin(1), 1.0, 0.0},
                       SPLIT_F64_T, w.sw, st, nullptr);
        if (e == cudaSuccess)
            e = gemm_f64(GemmF64{rem, nb, nb, w.Z, idx_lin(width), idx_lin(1), s.W, idx_lin(nb), idx_lin(1), w.X,
                                 idx_lin(width), idx_lin(1), -1.0, 0.0},
                         1, nullptr, 0, st);
        if (e == cudaSuccess)
            e = gemm_split(GemmF64{m, rem, nb, Vp, idx_lin(k), idx_lin(1), w.X, idx_lin(1), idx_lin(width), At,
                                   idx_lin(k), idx_lin(1), 1.0, 1.0},
                           SPLIT_F64_T, w.sw, st, nullptr);
    }
    if (e != cudaSuccess) return e;
    CTM_COUNT_LAUNCH(3);
    qr_blocked_r_kernel<<<k, 128, 0, st>>>(k, width, A, w.sgn, R);
    // S in two parts: the engine's error is in units of the columns' largest entries, which are the
    // v_0 of order 1 in the first k rows and ~1 / sqrt(n) below (in one part: |Q^T Q - 1| 1.0e-13
    // at n = 12000, k = 480)
    const double *Vb = w.V + (size_t)k * k;
    if (n > k)
        e = gemm_split(GemmF64{k, k, n - k, Vb, idx_lin(1), idx_lin(k), Vb, idx_lin(k), idx_lin(1), s.S, idx_lin(k),
                               idx_lin(1), 1.0, 0.0},
                       SPLIT_F64_T, w.sw, st, nullptr);
    if (e == cudaSuccess)
        e = gemm_split(GemmF64{k, k, k, w.V, idx_lin(1), idx_lin(k), w.V, idx_lin(k), idx_lin(1), s.S, idx_lin(k),
                               idx_lin(1), 1.0, n > k ? 1.0 : 0.0},
                       SPLIT_F64_T, w.sw, st, nullptr);
    if (e != cudaSuccess) return e;
    qr_blocked_w_kernel<<<(k + QR_WC - 1) / QR_WC, QR_THREADS, qr_wy_smem_bytes(k), st>>>(k, s.S, w.V, w.taus, w.sgn,
                                                                                          s.W);
    e = gemm_split(GemmF64{n, k, k, w.V, idx_lin(k), idx_lin(1), s.W, idx_lin(k), idx_lin(1), Q, idx_lin(k), idx_lin(1),
                           1.0, 0.0},
                   SPLIT_F64_T, w.sw, st, nullptr);
    if (e != cudaSuccess) return e;
    qr_blocked_diag_kernel<<<(k + 127) / 128, 128, 0, st>>>(k, w.sgn, Q);
    return cudaGetLastError();
}

cudaError_t qr_householder(int n, int k, const double *Y, double *Q, double *R, QrScratch s, cudaStream_t st)
{
    int G, rp;
    if (!qr_supported(n, k) || !s.V) return cudaErrorInvalidValue;
    const int width = qr_blocked_width(n, k, s);
    if (width) return qr_blocked(n, k, width, Y, Q, R, s, st);
    if (!qr_layout(n, k, s.rows_min > 0 ? s.rows_min : 1, &G, &rp, nullptr, s.force_slab) &&
        !qr_layout(n, k, 1, &G, &rp, nullptr, s.force_slab))
        return cudaErrorInvalidValue;
    const int rows_per = qr_pick_rows(n, k, Y, Q, R, s, st);
    return qr_factor_launch(n, k, rows_per, Y, Q, R, s, st);
}

cudaError_t qr_prepare()
{
    cudaError_t e = cudaFuncSetAttribute(qr_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, QR_SMEM_MAX);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(qr_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, QR_SMEM_MAX);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(qr_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, QR_SMEM_MAX);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(qr_blocked_w_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, QR_SMEM_MAX);
    return e;
}
