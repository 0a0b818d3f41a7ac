// solve_kernels.cu -- the cycle (Sec. 4): restriction b_c = R r, interpolation
// x = P x_c, Jacobi F/C sweeps x_i <- x_i + d_i (b_i - A_i x) (Eq. (2.4)), the dense
// coarsest solve, and the FP64 outer-iteration kernels (residual, norms, block dots
// for classical Gram-Schmidt, updates).
#include "setup_kernels.cuh"

namespace lair {

// coarsest level: y = Ainv b (dense, FP64), with the input/output in T
template <class T>
__global__ void k_dense_apply(int n, const double *__restrict__ Ainv, const T *__restrict__ b, T *__restrict__ y) {
    pdl_enter();
    int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    int nw = (gridDim.x * blockDim.x) >> 5;
    for (int r = wid; r < n; r += nw) {
        double acc = 0.0;
        for (int c = lane; c < n; c += 32) acc = fma(Ainv[(size_t)r * n + c], (double)b[c], acc);
        acc = warp_sum(acc);
        if (lane == 0) y[r] = (T)acc;
    }
}

template <class T>
void dense_apply(int n, const double *Ainv, const T *b, T *y, cudaStream_t s) {
    launch_pdl(k_dense_apply<T>, grid_for((long long)n * 32, 256), 256, 0, s, n, Ainv, b, y);
    count_launch();
}
template void dense_apply<double>(int, const double *, const double *, double *, cudaStream_t);
template void dense_apply<float>(int, const double *, const float *, float *, cudaStream_t);

// ---------------------------------------------------------------------------------------
// FP64 outer iteration
// ---------------------------------------------------------------------------------------
constexpr int RED_THREADS = 256;

// ---------------------------------------------------------------------------------------
// Reductions of the outer iteration. A warp FP64 instruction occupies an SM for 19 cycles whatever its lanes hold, so
// what a reduction costs is its number of such instructions, not its bytes: five butterfly additions per value and
// warp, over many warps with one or two elements a thread, took several times the products themselves. So the kernels
// run few blocks with many elements per thread (red_blocks), and a warp reduces eight values together: each half,
// quarter and eighth of the warp goes on with its own values, nine additions for eight values instead of forty.
// Block partials go to part[k * RED_PARTS + block]; k_finish sums them in a fixed order.
// ---------------------------------------------------------------------------------------

// the warp's sums of v[0..8); value k is complete in the four lanes whose bits 4, 3 and 2 are bits 2, 1 and 0 of k
__device__ __forceinline__ double warp_sum8(const double (&v)[8]) {
    const int lane = threadIdx.x & 31;
    const bool h = lane & 16, q = lane & 8, e = lane & 4;
    double a[4], c[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = (h ? v[k + 4] : v[k]) + __shfl_xor_sync(0xffffffffu, h ? v[k] : v[k + 4], 16);
#pragma unroll
    for (int k = 0; k < 2; ++k) c[k] = (q ? a[k + 2] : a[k]) + __shfl_xor_sync(0xffffffffu, q ? a[k] : a[k + 2], 8);
    double r = (e ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, e ? c[0] : c[1], 4);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    return r + __shfl_xor_sync(0xffffffffu, r, 1);
}
__device__ __forceinline__ int warp_sum8_index() { return (threadIdx.x >> 2) & 7; }

// part[k * RED_PARTS + blockIdx.x] = the block's sum of v[k], k < m <= MM
template <int MM>
__device__ __forceinline__ void block_partials(const double (&v)[MM], int m, double *part) {
    static_assert(MM % 8 == 0, "values in groups of eight");
    __shared__ double red[RED_THREADS / 32][MM];
#pragma unroll
    for (int g = 0; g < MM; g += 8)
        if (g < m) {
            double w[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) w[k] = v[g + k];
            const double r = warp_sum8(w);
            if ((threadIdx.x & 3) == 0) red[threadIdx.x >> 5][g + warp_sum8_index()] = r;
        }
    __syncthreads();
    if ((int)threadIdx.x < m) {
        double t = 0.0;
        for (int w = 0; w < RED_THREADS / 32; ++w) t += red[w][threadIdx.x];
        part[threadIdx.x * RED_PARTS + blockIdx.x] = t;
    }
}

// blocks of a reduction over n elements: two or more elements per thread, at most two blocks per SM
static int red_blocks(int n) {
    const int want = (n + RED_THREADS * 2 - 1) / (RED_THREADS * 2), most = 2 * device_sms();
    const int g = want < most ? (want > 0 ? want : 1) : most;
    return g < RED_PARTS ? g : RED_PARTS;
}

// out[k] = sum of the nb partials of vector k (fixed order); acc (if any): acc[k] = out[k] when first, else += out[k];
// inv (if any): 1 / sqrt(out[0]), 0 for a zero vector
__global__ void __launch_bounds__(128) k_finish(int m, int nb, const double *part, double *out, double *acc, int first,
                                                double *inv) {
    pdl_enter();
    const int k = blockIdx.x;
    if (k >= m) return;
    __shared__ double red[4];
    double t = 0.0;
    for (int b = threadIdx.x; b < nb; b += 128) t += part[k * RED_PARTS + b];
    t = warp_sum(t);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        const double u = ((red[0] + red[1]) + red[2]) + red[3];
        out[k] = u;
        if (acc) acc[k] = first ? u : acc[k] + u;
        if (inv && k == 0) *inv = u > 0.0 ? 1.0 / sqrt(u) : 0.0;
    }
}

static void finish(int m, int nb, const double *part, double *out, double *acc, int first, cudaStream_t s,
                   double *inv = nullptr) {
    launch_pdl(k_finish, m, 128, 0, s, m, nb, part, out, acc, first, inv);
    count_launch();
}

void finish_residual(const double *part, double *out, double *inv, cudaStream_t s) {
    finish(1, RED_PARTS, part, out, nullptr, 1, s, inv);
}

// |v|^2 as block partials
__global__ void __launch_bounds__(RED_THREADS) k_norm2(int n, const double *v, double *part) {
    pdl_enter();
    double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {
        double x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = v[i + k * stride];
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[0] = fma(x[k], x[k], acc[0]);
    }
    for (; i < n; i += stride) acc[0] = fma(v[i], v[i], acc[0]);
    block_partials<8>(acc, 1, part);
}

void norm2(int n, const double *v, double *part, double *out, cudaStream_t s) {
    const int nb = red_blocks(n);
    launch_pdl(k_norm2, nb, RED_THREADS, 0, s, n, v, part);
    count_launch();
    finish(1, nb, part, out, nullptr, 1, s);
}

// x += sum_k y_k Z_k (y on the device)
__global__ void k_add_combo(int n, int m, const double *__restrict__ Z, long long ldz, const double *__restrict__ y,
                            double *__restrict__ x) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double v = x[i];
        for (int k = 0; k < m; ++k) v = fma(y[k], Z[k * ldz + i], v);
        x[i] = v;
    }
}

void add_combo(int n, int m, const double *Z, long long ldz, const double *y, double *x, cudaStream_t s) {
    k_add_combo<<<grid_for(n, 256, device_sms() * 8), 256, 0, s>>>(n, m, Z, ldz, y, x);
    count_launch();
}

// ---------------------------------------------------------------------------------------
// One classical Gram-Schmidt step with re-orthogonalisation (CGS2) of w against the m <= 32
// columns of X in three streaming passes over X instead of four:
//   pass 1: part_k = X_k . w
//   pass 2: w <- w - sum_k h1_k X_k, then part_k = X_k . w (the new w)
//   pass 3: w <- w - sum_k h2_k X_k, then part_0 = w . w
// Each thread loads X_k[i] once per pass and keeps it in registers for both of its uses.
// The w update accumulates fma(-h_k, X_k[i], .) in ascending k. Bound by the FP64 units (4 m n fma a step).
// ---------------------------------------------------------------------------------------
template <int MM, int PASS>
__global__ void __launch_bounds__(RED_THREADS, MM <= 16 ? 2 : 1) k_cgs_pass(int n, int m,
                                                                            const double *__restrict__ X, long long ldx,
                                                                            const double *h, double *__restrict__ w,
                                                                            double *part) {
    pdl_enter();
    double acc[PASS < 3 ? MM : 8];
    __shared__ double hs[MM];
#pragma unroll
    for (int k = 0; k < (PASS < 3 ? MM : 8); ++k) acc[k] = 0.0;
    if (PASS > 1) {
        if ((int)threadIdx.x < MM) hs[threadIdx.x] = (int)threadIdx.x < m ? h[threadIdx.x] : 0.0;
        __syncthreads();
    }
#pragma unroll(MM <= 8 ? 2 : 1)
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        double x[MM];
#pragma unroll
        for (int k = 0; k < MM; ++k) x[k] = k < m ? X[k * ldx + i] : 0.0;
        double v = w[i];
        if (PASS > 1) {
#pragma unroll
            for (int k = 0; k < MM; ++k)
                if (k < m) v = fma(-hs[k], x[k], v);
            w[i] = v;
        }
        if (PASS < 3) {
#pragma unroll
            for (int k = 0; k < MM; ++k)
                if (k < m) acc[k] = fma(x[k], v, acc[k]);
        } else {
            acc[0] = fma(v, v, acc[0]);
        }
    }
    block_partials<(PASS < 3 ? MM : 8)>(acc, PASS < 3 ? m : 1, part);
}

template <int MM>
static void cgs_passes(int n, int m, const double *X, long long ldx, double *w, double *part, double *h1, double *h2,
                       double *hsum, double *nrm, double *inv, cudaStream_t s) {
    int nb = red_blocks(n);
    if (MM > 16 && nb > device_sms()) nb = device_sms();   // one block per SM is resident
    launch_pdl(k_cgs_pass<MM, 1>, nb, RED_THREADS, 0, s, n, m, X, ldx, (const double *)nullptr, w, part);
    finish(m, nb, part, h1, hsum, 1, s);
    launch_pdl(k_cgs_pass<MM, 2>, nb, RED_THREADS, 0, s, n, m, X, ldx, (const double *)h1, w, part);
    finish(m, nb, part, h2, hsum, 0, s);
    launch_pdl(k_cgs_pass<MM, 3>, nb, RED_THREADS, 0, s, n, m, X, ldx, (const double *)h2, w, part);
    finish(1, nb, part, nrm, nullptr, 1, s, inv);
    count_launch(3);
}

// (MM: columns kept in registers; 24 beside 16 and 32: 512^2 FD, FGMRES(30) 3.49 -> 3.35 ms, 101^3 FP64 7.83 -> 7.55 ms)
void cgs2(int n, int m, const double *X, long long ldx, double *w, double *part, double *h1, double *h2, double *hsum,
          double *nrm, double *inv, cudaStream_t s) {
    if (m <= 8) cgs_passes<8>(n, m, X, ldx, w, part, h1, h2, hsum, nrm, inv, s);
    else if (m <= 16) cgs_passes<16>(n, m, X, ldx, w, part, h1, h2, hsum, nrm, inv, s);
    else if (m <= 24) cgs_passes<24>(n, m, X, ldx, w, part, h1, h2, hsum, nrm, inv, s);
    else cgs_passes<32>(n, m, X, ldx, w, part, h1, h2, hsum, nrm, inv, s);
}

// v <- v * *inv, and its copy c as the cycle's right-hand side. The inverse norm comes from the kernel that summed the
// norm: formed here by every thread, its root and division cost the FP64 units more than the whole vector costs HBM
// (101^3: 14.1 us -> 6.5).
template <class T>
__global__ void __launch_bounds__(256) k_scale(int n, double *__restrict__ v, const double *inv, T *__restrict__ c) {
    pdl_enter();
    const double f = *inv;
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {
        double x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = v[i + k * stride] * f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[i + k * stride] = x[k];
            c[i + k * stride] = (T)x[k];
        }
    }
    for (; i < n; i += stride) {
        const double x = v[i] * f;
        v[i] = x;
        c[i] = (T)x;
    }
}

template <class T>
void scale(int n, double *v, const double *inv, T *c, cudaStream_t s) {
    launch_pdl(k_scale<T>, grid_for(n, 256, device_sms() * 8), 256, 0, s, n, v, inv, c);
    count_launch();
}
template void scale<float>(int, double *, const double *, float *, cudaStream_t);
template void scale<double>(int, double *, const double *, double *, cudaStream_t);

// precision conversions and plain vector updates
__global__ void k_d2f(int n, const double *__restrict__ a, float *__restrict__ b) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}
__global__ void k_f2d(int n, const float *__restrict__ a, double *__restrict__ b) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        b[i] = (double)a[i];
}
// x += e, four elements of a thread in flight (bound by HBM; 192^3: 34.7 us with one -> 31.8)
template <class T>
__global__ void __launch_bounds__(256) k_axpy(int n, const T *__restrict__ e, double *__restrict__ x) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (; i + 3 * stride < n; i += 4 * stride) {
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = x[i + k * stride] + (double)e[i + k * stride];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[i + k * stride] = v[k];
    }
    for (; i < n; i += stride) x[i] += (double)e[i];
}

void d2f(int n, const double *a, float *b, cudaStream_t s) { k_d2f<<<grid_for(n, 256, device_sms() * 8), 256, 0, s>>>(n, a, b); count_launch(); }
void f2d(int n, const float *a, double *b, cudaStream_t s) { k_f2d<<<grid_for(n, 256, device_sms() * 8), 256, 0, s>>>(n, a, b); count_launch(); }
void axpy_f(int n, const float *e, double *x, cudaStream_t s) { k_axpy<float><<<grid_for(n, 256, device_sms() * 8), 256, 0, s>>>(n, e, x); count_launch(); }
void axpy_d(int n, const double *e, double *x, cudaStream_t s) { k_axpy<double><<<grid_for(n, 256, device_sms() * 8), 256, 0, s>>>(n, e, x); count_launch(); }

// adjoint gradient on the pattern of A: g[k] = -lambda_i x_j
__global__ void k_grad_A(int n, const int *__restrict__ rp, const int *__restrict__ col, const double *__restrict__ lam,
                         const double *__restrict__ x, double *__restrict__ g) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double li = lam[i];
        for (int k = rp[i]; k < rp[i + 1]; ++k) g[k] = -li * x[col[k]];
    }
}

void grad_A(const DCsr &A, const double *lam, const double *x, double *g, cudaStream_t s) {
    k_grad_A<<<grid_for(A.nr, 256), 256, 0, s>>>(A.nr, A.rp, A.col, lam, x, g);
    count_launch();
}

// ---------------------------------------------------------------------------------------
// batched systems: per-system residuals, norms, dots and updates over row tiles. The rows of
// every system are cut into tiles of at most SEG_TILE rows (tile t: system tile[t].x, rows
// [tile[t].y, tile[t].z)); a CTA works on one tile at a time, so a large system is spread over
// many SMs. Reductions write one partial per tile; seg_reduce then sums the partials of each
// system in tile order (one warp per system), so the result does not depend on scheduling.
// ---------------------------------------------------------------------------------------
constexpr int SEG_GRID = 152 * 8;

__device__ __forceinline__ double block_sum(double v, double *red) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    __syncthreads();
    return t;
}

__global__ void __launch_bounds__(256) k_tile_residual(SegTiles st, const int *__restrict__ rp, const int *__restrict__ col,
                                                       const double *__restrict__ val, const double *__restrict__ b,
                                                       const double *__restrict__ x, double *__restrict__ r,
                                                       float *__restrict__ r32) {
    __shared__ double red[8];
    for (int t = blockIdx.x; t < st.ntiles; t += gridDim.x) {
        const int4 tl = st.tile[t];
        if (st.active && !st.active[tl.x]) continue;
        double ss = 0.0;
        for (int i = tl.y + threadIdx.x; i < tl.z; i += blockDim.x) {
            double acc = 0.0;
            for (int k = rp[i]; k < rp[i + 1]; ++k) acc = fma(val[k], x[col[k]], acc);
            const double ri = b[i] - acc;
            r[i] = ri;
            if (r32) r32[i] = (float)ri;
            ss = fma(ri, ri, ss);
        }
        const double tsum = block_sum(ss, red);
        if (threadIdx.x == 0) st.part[t] = tsum;
    }
}

__global__ void __launch_bounds__(256) k_tile_norm2(SegTiles st, const double *__restrict__ v) {
    __shared__ double red[8];
    for (int t = blockIdx.x; t < st.ntiles; t += gridDim.x) {
        const int4 tl = st.tile[t];
        if (st.active && !st.active[tl.x]) continue;
        double ss = 0.0;
        for (int i = tl.y + threadIdx.x; i < tl.z; i += blockDim.x) ss = fma(v[i], v[i], ss);
        const double tsum = block_sum(ss, red);
        if (threadIdx.x == 0) st.part[t] = tsum;
    }
}

// One pass of the batched CGS2 step over the tiles of the running systems (m <= 31 and m <= MM <= SEG_TILE_PARTS
// columns of X, h per system at h[q * hs]), each thread loading X_k[i] once for both of its uses:
//   PASS 1: part[t][k] = X_k . w over the tile
//   PASS 2: w <- w - sum_k h_k X_k, then part[t][k] = X_k . w (the new w)
//   PASS 3: w <- w - sum_k h_k X_k, then part[t][0] = w . w
// The update accumulates fma(-h_k, X_k[i], .) in ascending k and every partial is a warp sum followed by the
// sum over the warps in order, as in k_tile_norm2.
template <int MM, int PASS>
__global__ void __launch_bounds__(256) k_tile_cgs(SegTiles st, int m, const double *__restrict__ X, long long ldx,
                                                  int hs, const double *h, double *__restrict__ w) {
    pdl_enter();
    __shared__ double red[8][MM];
    __shared__ double hsh[MM];
    for (int t = blockIdx.x; t < st.ntiles; t += gridDim.x) {
        const int4 tl = st.tile[t];
        if (st.active && !st.active[tl.x]) continue;
        if (PASS > 1 && (int)threadIdx.x < MM) hsh[threadIdx.x] = (int)threadIdx.x < m ? h[(size_t)tl.x * hs + threadIdx.x] : 0.0;
        __syncthreads();
        double acc[PASS < 3 ? MM : 8];
#pragma unroll
        for (int k = 0; k < (PASS < 3 ? MM : 8); ++k) acc[k] = 0.0;
        for (int i = tl.y + threadIdx.x; i < tl.z; i += blockDim.x) {
            double x[MM];
#pragma unroll
            for (int k = 0; k < MM; ++k) x[k] = k < m ? X[k * ldx + i] : 0.0;
            double v = w[i];
            if (PASS > 1) {
#pragma unroll
                for (int k = 0; k < MM; ++k)
                    if (k < m) v = fma(-hsh[k], x[k], v);
                w[i] = v;
            }
            if (PASS < 3) {
#pragma unroll
                for (int k = 0; k < (PASS < 3 ? MM : 8); ++k)
                    if (k < m) acc[k] = fma(x[k], v, acc[k]);
            } else {
                acc[0] = fma(v, v, acc[0]);
            }
        }
        const int nout = PASS < 3 ? m : 1;
#pragma unroll
        for (int g = 0; g < (PASS < 3 ? MM : 8); g += 8)
            if (g < nout) {
                double u[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) u[k] = acc[g + k];
                const double v = warp_sum8(u);
                if ((threadIdx.x & 3) == 0) red[threadIdx.x >> 5][g + warp_sum8_index()] = v;
            }
        __syncthreads();
        if ((int)threadIdx.x < nout) {
            double s2 = 0.0;
            for (int ww = 0; ww < (int)(blockDim.x >> 5); ++ww) s2 += red[ww][threadIdx.x];
            st.part[(size_t)t * SEG_TILE_PARTS + threadIdx.x] = s2;
        }
        __syncthreads();
    }
}

// out[q * hs + k] = sum of the system's tile partials part[t * pw + k] (k < m): lane l adds tiles l, l + 32, ... and the
// lanes' sums are added as a tree. acc_out (if any): = the same when first, else += it. One warp per system, eight
// values at a time so that their loads overlap (one after another: 1,100 cycles each).
__global__ void __launch_bounds__(256) k_seg_reduce(SegTiles st, int pw, int m, int hs, double *out, double *acc_out,
                                                    int first) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    for (int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < st.nseg; q += (gridDim.x * blockDim.x) >> 5) {
        if (st.active && !st.active[q]) continue;
        const int t0 = st.first[q], t1 = st.first[q + 1];
        for (int g = 0; g < m; g += 8) {
            double v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = 0.0;
            for (int t = t0 + lane; t < t1; t += 32)
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (g + k < m) v[k] += st.part[(size_t)t * pw + g + k];
            const double r = warp_sum8(v);
            const int k = g + warp_sum8_index();
            if ((lane & 3) == 0 && k < m) {
                out[(size_t)q * hs + k] = r;
                if (acc_out) acc_out[(size_t)q * hs + k] = first ? r : acc_out[(size_t)q * hs + k] + r;
            }
        }
    }
}

// x_i += sum_{k < cnt[q]} y[q * hs + k] Z_k[i] for the rows of system q
__global__ void __launch_bounds__(256) k_tile_add_combo(SegTiles st, const int *__restrict__ cnt, const double *__restrict__ Z,
                                                        long long ldz, int hs, const double *__restrict__ y,
                                                        double *__restrict__ x) {
    for (int t = blockIdx.x; t < st.ntiles; t += gridDim.x) {
        const int4 tl = st.tile[t];
        if (st.active && !st.active[tl.x]) continue;
        const int m = cnt[tl.x];
        if (m == 0) continue;
        const double *yq = y + (size_t)tl.x * hs;
        for (int i = tl.y + threadIdx.x; i < tl.z; i += blockDim.x) {
            double v = x[i];
            for (int k = 0; k < m; ++k) v = fma(yq[k], Z[k * ldz + i], v);
            x[i] = v;
        }
    }
}

// v <- v / |v| per running system, and c = the same in T (the cycle's right-hand side)
template <class T>
__global__ void __launch_bounds__(256) k_tile_scale(SegTiles st, double *v, const double *nrm2, T *c) {
    pdl_enter();
    __shared__ double inv_s;   // one thread's root and division for the tile: they are what the FP64 units cost
    for (int t = blockIdx.x; t < st.ntiles; t += gridDim.x) {
        const int4 tl = st.tile[t];
        if (st.active && !st.active[tl.x]) continue;
        __syncthreads();
        if (threadIdx.x == 0) inv_s = nrm2[tl.x] > 0.0 ? 1.0 / sqrt(nrm2[tl.x]) : 0.0;
        __syncthreads();
        const double inv = inv_s;
        for (int i = tl.y + threadIdx.x; i < tl.z; i += blockDim.x) {
            const double x = v[i] * inv;
            v[i] = x;
            c[i] = (T)x;
        }
    }
}

template <class T>
__global__ void __launch_bounds__(256) k_tile_axpy(SegTiles st, const uint8_t *__restrict__ active, const T *__restrict__ e,
                                                   double *__restrict__ x) {
    for (int t = blockIdx.x; t < st.ntiles; t += gridDim.x) {
        const int4 tl = st.tile[t];
        if (st.active && !st.active[tl.x]) continue;
        if (!active[tl.x]) continue;
        for (int i = tl.y + threadIdx.x; i < tl.z; i += blockDim.x) x[i] += (double)e[i];
    }
}

// ---------------------------------------------------------------------------------------
// device-side control of the batched outer loops: one thread per system decides, from the
// per-system norms the tile kernels reduced, whether the system goes on, and keeps its Krylov
// state; the flags feed the tile kernels (SegTiles.active) of the next step directly, so the
// host never has to read a norm to continue. count (zero on entry) receives the number of
// systems still running. The arithmetic of the stopping tests and Givens rotations is the
// oracle's (separate roundings, no fused operations).
// ---------------------------------------------------------------------------------------
__global__ void k_bat_bnorm(int nseg, const double *__restrict__ nrm2, double *__restrict__ bn) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q < nseg) bn[q] = nrm2[q] > 0.0 ? sqrt(nrm2[q]) : 1.0;
}

// stationary refinement, iteration it: from ||r_q||^2, deactivate converged systems; count the running ones
// (each running system then receives one more cycle)
__global__ void k_bat_stat_check(BatchCtl c, const double *__restrict__ nrm2, int it, int *count) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= c.nseg || !c.run[q]) return;
    const double r = __ddiv_rn(sqrt(nrm2[q]), c.bn[q]);
    c.rl[q] = r;
    if (!isfinite(r)) {
        *c.nan = 1;
        c.run[q] = 0;
        return;
    }
    if (r <= c.tol || it >= c.max_iter) {
        c.run[q] = 0;
        return;
    }
    c.its[q] += 1;
    atomicAdd(count, 1);
}

// FGMRES restart: beta = ||r_q||, the stopping test on it, g = beta e_1 for the systems that go on
__global__ void k_bat_fg_restart(BatchCtl c, const double *__restrict__ nrm2, int *count) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= c.nseg) return;
    c.jd[q] = 0;
    const double beta = sqrt(nrm2[q]);
    const double r = __ddiv_rn(beta, c.bn[q]);
    c.rl[q] = r;
    if (!isfinite(r)) {
        *c.nan = 1;
        c.done[q] = 1;
    }
    if (r <= c.tol || c.its[q] >= c.max_iter) c.done[q] = 1;
    c.run[q] = c.done[q] ? 0 : 1;
    if (!c.run[q]) return;
    double *g = c.g + (size_t)q * (c.m + 1);
    for (int k = 0; k <= c.m; ++k) g[k] = 0.0;
    g[0] = beta;
    atomicAdd(count, 1);
}

// FGMRES step j of every running system: the new Hessenberg column (the Gram-Schmidt sums h[q * hs + k],
// k <= j, and ||w||), the earlier rotations applied to it, a new rotation, the residual estimate and the
// stopping test; a system that stops keeps its step count in jd
__global__ void k_bat_fg_givens(BatchCtl c, int j, const double *hsum, const double *nrm2w,
                                int *count) {
    pdl_enter();
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= c.nseg || !c.run[q]) return;
    const int m = c.m;
    double hc[BATCH_HS + 1];
    for (int k = 0; k <= j; ++k) hc[k] = hsum[(size_t)q * c.hs + k];
    const double hn = sqrt(nrm2w[q]);
    hc[j + 1] = hn;
    double *cs = c.cs + (size_t)q * m, *sn = c.sn + (size_t)q * m, *g = c.g + (size_t)q * (m + 1);
    double *Hq = c.Hm + (size_t)q * (m + 1) * m;
    for (int k = 0; k < j; ++k) {
        const double t = __dadd_rn(__dmul_rn(cs[k], hc[k]), __dmul_rn(sn[k], hc[k + 1]));
        hc[k + 1] = __dadd_rn(__dmul_rn(-sn[k], hc[k]), __dmul_rn(cs[k], hc[k + 1]));
        hc[k] = t;
    }
    const double den = sqrt(__dadd_rn(__dmul_rn(hc[j], hc[j]), __dmul_rn(hc[j + 1], hc[j + 1])));
    cs[j] = den > 0.0 ? __ddiv_rn(hc[j], den) : 1.0;
    sn[j] = den > 0.0 ? __ddiv_rn(hc[j + 1], den) : 0.0;
    hc[j] = den;
    g[j + 1] = __dmul_rn(-sn[j], g[j]);
    g[j] = __dmul_rn(cs[j], g[j]);
    for (int k = 0; k <= j; ++k) Hq[(size_t)k * m + j] = hc[k];
    c.its[q] += 1;
    const double est = __ddiv_rn(fabs(g[j + 1]), c.bn[q]);
    if (est <= c.tol || hn == 0.0 || !isfinite(est) || c.its[q] >= c.max_iter || j == m - 1) {
        c.run[q] = 0;
        c.jd[q] = j + 1;
    } else {
        atomicAdd(count, 1);
    }
}

// y_q = H_q^{-1} g_q (upper triangular, jd_q x jd_q) for the update x += Z y
__global__ void k_bat_fg_solve_y(BatchCtl c, double *__restrict__ y) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= c.nseg) return;
    const int jd = c.jd[q], m = c.m;
    const double *Hq = c.Hm + (size_t)q * (m + 1) * m, *g = c.g + (size_t)q * (m + 1);
    double *yq = y + (size_t)q * c.hs;
    for (int k = jd - 1; k >= 0; --k) {
        double acc = g[k];
        for (int cc = k + 1; cc < jd; ++cc) acc = __dsub_rn(acc, __dmul_rn(Hq[(size_t)k * m + cc], yq[cc]));
        yq[k] = __ddiv_rn(acc, Hq[(size_t)k * m + k]);
    }
}

void bat_bnorm(int nseg, const double *nrm2, double *bn, cudaStream_t s) {
    k_bat_bnorm<<<(nseg + 127) / 128, 128, 0, s>>>(nseg, nrm2, bn);
    count_launch();
}
void bat_stat_check(const BatchCtl &c, const double *nrm2, int it, int *count, cudaStream_t s) {
    k_bat_stat_check<<<(c.nseg + 127) / 128, 128, 0, s>>>(c, nrm2, it, count);
    count_launch();
}
void bat_fg_restart(const BatchCtl &c, const double *nrm2, int *count, cudaStream_t s) {
    k_bat_fg_restart<<<(c.nseg + 127) / 128, 128, 0, s>>>(c, nrm2, count);
    count_launch();
}
void bat_fg_givens(const BatchCtl &c, int j, const double *hsum, const double *nrm2w, int *count, cudaStream_t s) {
    launch_pdl(k_bat_fg_givens, (c.nseg + 127) / 128, 128, 0, s, c, j, hsum, nrm2w, count);
    count_launch();
}
void bat_fg_solve_y(const BatchCtl &c, double *y, cudaStream_t s) {
    k_bat_fg_solve_y<<<(c.nseg + 127) / 128, 128, 0, s>>>(c, y);
    count_launch();
}

static int seg_grid(const SegTiles &st) { return st.ntiles < SEG_GRID ? (st.ntiles > 0 ? st.ntiles : 1) : SEG_GRID; }

static void seg_reduce(const SegTiles &st, int pw, int m, int hs, double *out, double *acc, int first, cudaStream_t s) {
    launch_pdl(k_seg_reduce, (st.nseg + 7) / 8, 256, 0, s, st, pw, m, hs, out, acc, first);
    count_launch();
}

template <int MM>
static void seg_cgs_mm(const SegTiles &st, int pass, int m, const double *X, long long ldx, int hs, const double *h,
                       double *w, cudaStream_t s) {
    if (pass == 1) launch_pdl(k_tile_cgs<MM, 1>, seg_grid(st), 256, 0, s, st, m, X, ldx, hs, h, w);
    else if (pass == 2) launch_pdl(k_tile_cgs<MM, 2>, seg_grid(st), 256, 0, s, st, m, X, ldx, hs, h, w);
    else launch_pdl(k_tile_cgs<MM, 3>, seg_grid(st), 256, 0, s, st, m, X, ldx, hs, h, w);
    count_launch();
}

void seg_cgs_pass(const SegTiles &st, int pass, int m, const double *X, long long ldx, int hs, const double *h, double *w,
                  double *out, double *acc, cudaStream_t s) {
    if (m <= 8) seg_cgs_mm<8>(st, pass, m, X, ldx, hs, h, w, s);
    else if (m <= 16) seg_cgs_mm<16>(st, pass, m, X, ldx, hs, h, w, s);
    else if (m <= 24) seg_cgs_mm<24>(st, pass, m, X, ldx, hs, h, w, s);
    else seg_cgs_mm<32>(st, pass, m, X, ldx, hs, h, w, s);
    if (pass < 3) seg_reduce(st, SEG_TILE_PARTS, m, hs, out, acc, pass == 1, s);
    else seg_reduce(st, SEG_TILE_PARTS, 1, 1, out, nullptr, 1, s);
}

void seg_add_combo(const SegTiles &st, const int *cnt, const double *Z, long long ldz, int hs, const double *y, double *x,
                   cudaStream_t s) {
    k_tile_add_combo<<<seg_grid(st), 256, 0, s>>>(st, cnt, Z, ldz, hs, y, x);
    count_launch();
}
template <class T>
void seg_scale(const SegTiles &st, double *v, const double *nrm2, T *c, cudaStream_t s) {
    launch_pdl(k_tile_scale<T>, seg_grid(st), 256, 0, s, st, v, nrm2, c);
    count_launch();
}
template void seg_scale<float>(const SegTiles &, double *, const double *, float *, cudaStream_t);
template void seg_scale<double>(const SegTiles &, double *, const double *, double *, cudaStream_t);
void seg_residual(const DCsr &A, const SegTiles &st, const double *b, const double *x, double *r, float *r32,
                  double *norm2, cudaStream_t s) {
    k_tile_residual<<<seg_grid(st), 256, 0, s>>>(st, A.rp, A.col, A.val, b, x, r, r32);
    count_launch();
    seg_reduce(st, 1, 1, 1, norm2, nullptr, 1, s);
}
void seg_norm2(const SegTiles &st, const double *v, double *norm2, cudaStream_t s) {
    k_tile_norm2<<<seg_grid(st), 256, 0, s>>>(st, v);
    count_launch();
    seg_reduce(st, 1, 1, 1, norm2, nullptr, 1, s);
}
template <class T>
void seg_axpy(const SegTiles &st, const uint8_t *active, const T *e, double *x, cudaStream_t s) {
    k_tile_axpy<T><<<seg_grid(st), 256, 0, s>>>(st, active, e, x);
    count_launch();
}
template void seg_axpy<float>(const SegTiles &, const uint8_t *, const float *, double *, cudaStream_t);
template void seg_axpy<double>(const SegTiles &, const uint8_t *, const double *, double *, cudaStream_t);

__global__ void k_gather_int(int m, const int *__restrict__ idx, const int *__restrict__ src, int *__restrict__ out) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m; t += gridDim.x * blockDim.x) out[t] = src[idx[t]];
}

void gather_int(int m, const int *idx, const int *src, int *out, cudaStream_t s) {
    k_gather_int<<<grid_for(m, 256), 256, 0, s>>>(m, idx, src, out);
    count_launch();
}

// rows and entries of F and C rows: out = {n_F, nnz_F, n_C, nnz_C}
__global__ void k_cf_stats(int n, const int *__restrict__ rp, const int8_t *__restrict__ cf,
                           unsigned long long *__restrict__ out) {
    unsigned long long a = 0, b = 0, c = 0, d = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        unsigned long long len = (unsigned long long)(rp[i + 1] - rp[i]);
        if (cf[i] == CF_F) { a += 1; b += len; } else { c += 1; d += len; }
    }
    a = warp_sum(a); b = warp_sum(b); c = warp_sum(c); d = warp_sum(d);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(out + 0, a); atomicAdd(out + 1, b); atomicAdd(out + 2, c); atomicAdd(out + 3, d);
    }
}

void cf_stats(const DCsr &A, const int8_t *cf, unsigned long long *out4, cudaStream_t s) {
    k_cf_stats<<<grid_for(A.nr, 256), 256, 0, s>>>(A.nr, A.rp, cf, out4);
    count_launch();
}

}  // namespace lair
