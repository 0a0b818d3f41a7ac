// sell.cu -- sliced-ELL copies of the cycle's matrices and the kernels that stream them.
//
// A view holds a subset of a matrix's rows (all rows, or only the F rows or only the C rows of
// a level) in slices of 32 rows. Inside a slice, entry j of the slice's r-th row sits at
// slice_ptr[s] + 32 j + r, so one thread owns one row and the 32 threads of a warp read 32
// consecutive values and column indices per step: every load is coalesced and a thread keeps
// several independent loads in flight. Rows are ordered by decreasing length inside windows of
// 256 rows to keep the padding of a slice small; row[] maps a view row back to its matrix row.
// The sweeps of a level then read only the rows they update (F rows, or C rows).
#include "setup_kernels.cuh"

#include <climits>

namespace lair {

constexpr int SELL_WINDOW = 256;

// F rows in ascending order from the exclusive scan of the C flags: F point i has F index i - scan[i]
__global__ void k_frows(int n, const int8_t *__restrict__ cf, const int *__restrict__ cscan, int *__restrict__ frows) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        if (cf[i] != CF_C) frows[i - cscan[i]] = i;
}

// ---------------------------------------------------------------------------------------
// Building many views at once. Views are described by SellDesc entries; view p owns windows
// [win0, win0 + its windows), linear slices [lin0, lin0 + its slices) and, in the slice-length
// array cnt, positions [sl0, sl0 + its slices). Every kernel finds the view of its window or
// slice by binary search over the descriptors.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ int find_desc(const SellDesc *__restrict__ d, int nd, int key, int which) {
    int lo = 0, hi = nd - 1;     // last descriptor whose start <= key
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const int st = which == 0 ? d[mid].win0 : d[mid].lin0;
        if (st <= key) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Ascending bitonic sort of 32 R distinct keys held by a warp, element e = 32 r + lane in key[r]: exchanges at
// distance < 32 through shuffles, the others inside a lane's registers (compile-time indices only).
template <int R>
__device__ __forceinline__ void warp_sort_keys(unsigned (&key)[R], int lane) {
#pragma unroll
    for (int k = 2; k <= 32 * R; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int r2 = r ^ (j >> 5);
                    if (r2 > r) {
                        const bool up = ((32 * r + lane) & k) == 0;
                        if (up ? key[r] > key[r2] : key[r] < key[r2]) {
                            const unsigned t = key[r];
                            key[r] = key[r2];
                            key[r2] = t;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const unsigned pk = __shfl_xor_sync(0xffffffffu, key[r], j);
                    const bool up = ((32 * r + lane) & k) == 0, lower = (lane & j) == 0;
                    if (lower == up ? pk < key[r] : pk > key[r]) key[r] = pk;
                }
            }
        }
    }
}

constexpr int SORT_WARPS = 8;                 // windows in flight per CTA (one per warp)
constexpr int SELL_RPL = SELL_WINDOW / 32;    // rows of a window per lane
constexpr int SELL_COUNT_SORT = 16;           // windows with fewer distinct lengths than this: counting sort

// Order the rows of every window by decreasing length (ties: window position), one warp per window: row t of
// the window is lane t % 32's entry t / 32, so the loads of a window are coalesced and every lane has eight
// independent row lengths in flight. A window already in non-increasing order (the interior of a stencil)
// is written as it is, one with a narrow range of lengths goes through a counting sort by length, the others
// through a register bitonic sort of (length, position) keys.
__global__ void __launch_bounds__(32 * SORT_WARPS) k_sell_sort_multi(const SellDesc *__restrict__ d, int nd,
                                                                     int nwin) {
    __shared__ int stage[SORT_WARPS][SELL_WINDOW];
    const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
    for (int w = blockIdx.x * SORT_WARPS + wq; w < nwin; w += gridDim.x * SORT_WARPS) {
        const int p = find_desc(d, nd, w, 0);
        const int *rows_in = d[p].rows_in, *rp = d[p].rp;
        int *row_out = d[p].row_out;
        const int w0 = (w - d[p].win0) * SELL_WINDOW;
        const int cnt = min(SELL_WINDOW, d[p].nrows - w0);
        int rid[SELL_RPL], len[SELL_RPL];
#pragma unroll
        for (int k = 0; k < SELL_RPL; ++k) {
            const int t = 32 * k + lane;
            rid[k] = t < cnt ? (rows_in ? rows_in[w0 + t] : w0 + t) : -1;
        }
#pragma unroll
        for (int k = 0; k < SELL_RPL; ++k) len[k] = rid[k] >= 0 ? rp[rid[k] + 1] - rp[rid[k]] : -1;
        bool ok = true;
#pragma unroll
        for (int k = 0; k < SELL_RPL; ++k) {
            const int down = __shfl_down_sync(0xffffffffu, len[k], 1);
            const int wrap = __shfl_sync(0xffffffffu, k + 1 < SELL_RPL ? len[k + 1 < SELL_RPL ? k + 1 : k] : 0, 0);
            const int next = lane < 31 ? down : (k + 1 < SELL_RPL ? wrap : -1);
            if (32 * k + lane + 1 < cnt && len[k] < next) ok = false;
        }
        if (__all_sync(0xffffffffu, ok)) {
#pragma unroll
            for (int k = 0; k < SELL_RPL; ++k)
                if (32 * k + lane < cnt) row_out[w0 + 32 * k + lane] = rid[k];
            continue;
        }
        // few distinct lengths (a stencil's boundary rows): a counting sort, longest first, window order inside
        // a length -- the same order as the stable sort, at one ballot per length and row register
        int lo = INT_MAX, hi = -1;
#pragma unroll
        for (int k = 0; k < SELL_RPL; ++k)
            if (len[k] >= 0) {
                lo = min(lo, len[k]);
                hi = max(hi, len[k]);
            }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (hi - lo < SELL_COUNT_SORT) {
            const unsigned below = (1u << lane) - 1u;
            int pos[SELL_RPL];
            int base = 0;
            for (int v = hi; v >= lo; --v) {
#pragma unroll
                for (int k = 0; k < SELL_RPL; ++k) {
                    const unsigned m = __ballot_sync(0xffffffffu, len[k] == v);
                    if (len[k] == v) pos[k] = base + __popc(m & below);
                    base += __popc(m);
                }
            }
#pragma unroll
            for (int k = 0; k < SELL_RPL; ++k)
                if (len[k] >= 0) row_out[w0 + pos[k]] = rid[k];
            continue;
        }
        // keys: (2^23 - 1 - length) in the high bits, the window position in the low 8; padding last
        unsigned key[SELL_RPL];
#pragma unroll
        for (int k = 0; k < SELL_RPL; ++k) {
            const int t = 32 * k + lane;
            stage[wq][t] = rid[k];
            key[k] = t < cnt ? ((unsigned)(0x7fffff - min(len[k], 0x7fffff)) << 8) | (unsigned)t : 0xffffffffu;
        }
        __syncwarp();
        warp_sort_keys<SELL_RPL>(key, lane);
#pragma unroll
        for (int k = 0; k < SELL_RPL; ++k)
            if (32 * k + lane < cnt) row_out[w0 + 32 * k + lane] = stage[wq][key[k] & 0xffu];
        __syncwarp();
    }
}

// batched systems: the system of row i (the last q with seg[q] <= i)
__device__ __forceinline__ int system_of(const int *__restrict__ seg, int nseg, int i) {
    int lo = 0, hi = nseg - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (seg[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// slice lengths in entries (32 x longest row of the slice), one warp per slice; also their
// 64-bit sum per group (two groups: FP32 and FP64 views), so that an int overflow of the offsets is caught on
// the host. Each warp adds its own sums once at the end.
__global__ void k_sell_len_multi(const SellDesc *__restrict__ d, int nd, int nlin, int *__restrict__ cnt,
                                 unsigned long long *__restrict__ gsum) {
    const int lane = threadIdx.x & 31;
    unsigned long long s0 = 0, s1 = 0;
    for (int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < nlin; q += (gridDim.x * blockDim.x) >> 5) {
        const int p = find_desc(d, nd, q, 1);
        const SellDesc &v = d[p];
        const int sl = q - v.lin0;
        const int r = sl * 32 + lane;
        int l = 0, sy = -2;
        if (r < v.nrows) {
            const int i = v.row_out[r];
            l = v.rp[i + 1] - v.rp[i];
            if (v.nseg > 0) sy = system_of(v.seg, v.nseg, i);
        }
        l = __reduce_max_sync(0xffffffffu, l);
        if (v.nseg > 0) {
            // the slice's system when all its rows share one (lane 0 always holds a row)
            const int sy0 = __shfl_sync(0xffffffffu, sy, 0);
            const bool one = __all_sync(0xffffffffu, sy == -2 || sy == sy0);
            if (lane == 0) v.slice_sys[sl] = one ? sy0 : -1;
        }
        if (lane == 0) {
            cnt[v.sl0 + sl] = 32 * l;
            if (v.group == 0) s0 += 32ull * (unsigned long long)l;
            else s1 += 32ull * (unsigned long long)l;
        }
    }
    if (lane == 0) {
        if (s0) atomicAdd(&gsum[0], s0);
        if (s1) atomicAdd(&gsum[1], s1);
    }
}

// entries of the views [p0, p1) (one element type), one thread per row slot of a slice
template <class T>
__global__ void k_sell_fill_multi(const SellDesc *__restrict__ d, int p0, int p1, int lin_end) {
    const int lin_beg = d[p0].lin0;
    const long long nslot = 32ll * (lin_end - lin_beg);
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nslot; e += (long long)gridDim.x * blockDim.x) {
        const int q = lin_beg + (int)(e >> 5), lane = (int)(e & 31);
        const int p = p0 + find_desc(d + p0, p1 - p0, q, 1);
        const SellDesc &v = d[p];
        const int sl = q - v.lin0;
        const int *sptr = v.slice_ptr;
        const int base = sptr[sl] + lane, len = (sptr[sl + 1] - sptr[sl]) >> 5;
        const int r = sl * 32 + lane;
        // padding entries carry value 0 and a column that is valid for x: the row's last column
        // (a row index is not one when the matrix is rectangular, as P and R are)
        int b = 0, en = 0, pad = 0;
        if (r < v.nrows) {
            const int i = v.row_out[r];
            b = v.rp[i];
            en = v.rp[i + 1];
            pad = en > b ? v.col[en - 1] : 0;
            if (v.sdinv) static_cast<T *>(v.sdinv)[r] = (T)v.dinv[i];
        }
        int *scol = v.scol;
        T *sval = static_cast<T *>(v.sval);
        for (int j = 0; j < len; ++j) {
            const bool in = b + j < en;
            scol[base + 32 * j] = in ? v.col[b + j] : pad;
            sval[base + 32 * j] = in ? (T)v.val[b + j] : T(0);
        }
    }
}

// The matrix entries, the Jacobi diagonal and b are read once per launch: they are loaded with the
// streaming (evict-first) policy, so that they pass through L2 without pushing out x, which every row
// gathers from and which stays in L2 from one kernel of the cycle to the next.
//
// y[row[r]] = (view row r) . x. RPT rows per thread: the thread of lane l in group g takes row l of each of
// the slices g RPT, ..., g RPT + RPT - 1, so every load of a warp stays coalesced and a thread keeps RPT
// independent sums in flight; each row is still summed alone in column order.
template <class T, int RPT>
__global__ void __launch_bounds__(256) k_sell_spmv(SellView v, const T *__restrict__ x, T *__restrict__ y) {
    pdl_enter();
    const int *__restrict__ sptr = v.slice_ptr;
    const int *__restrict__ scol = v.col;
    const T *__restrict__ sval = static_cast<const T *>(v.val);
    const int nsl = (v.nrows + 31) >> 5;
    const long long nthr = (long long)((nsl + RPT - 1) / RPT) * 32;
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < nthr; u += (long long)gridDim.x * blockDim.x) {
        const int lane = (int)(u & 31), s0 = (int)(u >> 5) * RPT;
        int base[RPT], len[RPT], r[RPT];
        int lmax = 0;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            bool on = s0 + k < nsl;
            if (on && v.run) {
                const int q = v.slice_sys[s0 + k];
                on = q < 0 || v.run[q];
            }
            r[k] = on ? (s0 + k) * 32 + lane : v.nrows;
            base[k] = 0;
            len[k] = 0;
            if (on) {
                const int a = __ldg(sptr + s0 + k);
                base[k] = a + lane;
                len[k] = (__ldg(sptr + s0 + k + 1) - a) >> 5;
            }
            lmax = max(lmax, len[k]);
        }
        T acc[RPT];
#pragma unroll
        for (int k = 0; k < RPT; ++k) acc[k] = T(0);
#pragma unroll 4
        for (int j = 0; j < lmax; ++j)
#pragma unroll
            for (int k = 0; k < RPT; ++k)
                if (j < len[k])
                    acc[k] = fma(__ldcs(sval + base[k] + 32 * j), __ldg(x + __ldcs(scol + base[k] + 32 * j)), acc[k]);
#pragma unroll
        for (int k = 0; k < RPT; ++k)
            if (r[k] < v.nrows) y[v.row[r[k]]] = acc[k];
    }
}

// one Jacobi sweep over the view's rows (x_i + d_i (b_i - A_i x)), RPT rows per thread as above; then the
// entries of the other rows (copy[], ncopy of them) are copied from x to xo, one per thread
template <class T, int RPT>
__global__ void __launch_bounds__(256) k_sell_sweep(SellView v, const int *__restrict__ copy, int ncopy,
                                                    const T *__restrict__ b, const T *__restrict__ x, T *__restrict__ xo) {
    pdl_enter();
    const int *__restrict__ sptr = v.slice_ptr;
    const int *__restrict__ scol = v.col;
    const T *__restrict__ sval = static_cast<const T *>(v.val);
    const T *__restrict__ sd = static_cast<const T *>(v.dinv);
    const int nsl = (v.nrows + 31) >> 5;
    const long long nthr = (long long)((nsl + RPT - 1) / RPT) * 32;
    const long long total = nthr + ncopy;
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < total; u += (long long)gridDim.x * blockDim.x) {
        if (u < nthr) {
            const int lane = (int)(u & 31), s0 = (int)(u >> 5) * RPT;
            int base[RPT], len[RPT], r[RPT];
            int lmax = 0;
#pragma unroll
            for (int k = 0; k < RPT; ++k) {
                bool on = s0 + k < nsl;
                if (on && v.run) {
                    const int q = v.slice_sys[s0 + k];
                    on = q < 0 || v.run[q];
                }
                r[k] = on ? (s0 + k) * 32 + lane : v.nrows;
                base[k] = 0;
                len[k] = 0;
                if (on) {
                    const int a = __ldg(sptr + s0 + k);
                    base[k] = a + lane;
                    len[k] = (__ldg(sptr + s0 + k + 1) - a) >> 5;
                }
                lmax = max(lmax, len[k]);
            }
            T acc[RPT];
#pragma unroll
            for (int k = 0; k < RPT; ++k) acc[k] = T(0);
#pragma unroll 4
            for (int j = 0; j < lmax; ++j)
#pragma unroll
                for (int k = 0; k < RPT; ++k)
                    if (j < len[k])
                        acc[k] = fma(__ldcs(sval + base[k] + 32 * j), __ldg(x + __ldcs(scol + base[k] + 32 * j)), acc[k]);
#pragma unroll
            for (int k = 0; k < RPT; ++k)
                if (r[k] < v.nrows) {
                    const int i = v.row[r[k]];
                    xo[i] = fma(__ldcs(sd + r[k]), __ldcs(b + i) - acc[k], x[i]);
                }
        } else {
            const int j = copy[u - nthr];
            xo[j] = x[j];
        }
    }
}

// The same product and sweep for launches of about one wave (one_wave). Those are bound by their chain of
// dependent loads -- slice offset, columns, gathered x, then row and b -- and by the launch itself, not by bandwidth.
// So a thread has one row and brings everything that does not depend on the previous kernel of the cycle (offsets,
// the first NB values and columns, the Jacobi diagonal, the row's index) into registers before it waits for that
// kernel; then come NB gathers at once and the sum, in column order as above. x, b and xo are plain pointers: their
// loads must stay behind the wait. More registers and fewer resident warps than the kernels above, which is why
// larger views do not take it.
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// An entry stays in registers from here on: left alone, the compiler may move its loads past the wait into the branch
// that uses them (FP64 sweeps with 32 instead of 88 registers; 301^2 FD, solve 3.14 -> 3.20 ms).
__device__ __forceinline__ void hold(int &c, float &w) { asm volatile("" : "+r"(c), "+f"(w)); }
__device__ __forceinline__ void hold(int &c, double &w) { asm volatile("" : "+r"(c), "+d"(w)); }

template <class T, int NB>
struct RowHead {
    int base = 0, len = 0, i = -1;
    int c[NB];
    T w[NB];
    // row slot u of the view (u < 32 * slices); a slice of a stopped system has no row
    __device__ __forceinline__ void load(const SellView &v, int u, int nrows) {
        const int sl = u >> 5, lane = u & 31;
        bool on = true;
        if (v.run) {
            const int q = v.slice_sys[sl];
            on = q < 0 || v.run[q];
        }
        if (on) {
            const int a = __ldg(v.slice_ptr + sl);
            base = a + lane;
            len = (__ldg(v.slice_ptr + sl + 1) - a) >> 5;
        }
        if (on && u < nrows) i = __ldg(v.row + u);
        const T *val = static_cast<const T *>(v.val);
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            c[k] = k < len ? __ldg(v.col + base + 32 * k) : 0;
            w[k] = k < len ? __ldg(val + base + 32 * k) : T(0);
        }
#pragma unroll
        for (int k = 0; k < NB; ++k) hold(c[k], w[k]);
    }
    __device__ __forceinline__ T sum(const SellView &v, const T *x) const {
        T acc = T(0);
        {
            T xv[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) xv[k] = k < len ? x[c[k]] : T(0);
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (k < len) acc = fma(w[k], xv[k], acc);
        }
        const T *val = static_cast<const T *>(v.val);
        for (int j = NB; j < len; j += NB) {
            int cc[NB];
            T ww[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                cc[k] = j + k < len ? __ldg(v.col + base + 32 * (j + k)) : 0;
                ww[k] = j + k < len ? __ldg(val + base + 32 * (j + k)) : T(0);
            }
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (j + k < len) acc = fma(ww[k], x[cc[k]], acc);
        }
        return acc;
    }
};

constexpr int WAVE_THREADS = 128;

template <class T, int NB>
__global__ void __launch_bounds__(WAVE_THREADS) k_sell_spmv_wave(SellView v, const T *x, T *y) {
    pdl_launch_next();
    const int u = blockIdx.x * WAVE_THREADS + threadIdx.x;
    RowHead<T, NB> h;
    if (u < ((v.nrows + 31) & ~31)) h.load(v, u, v.nrows);
    pdl_wait_previous();
    const T acc = h.sum(v, x);
    if (h.i >= 0) y[h.i] = acc;
}

template <class T, int NB>
__global__ void __launch_bounds__(WAVE_THREADS) k_sell_sweep_wave(SellView v, const int *copy, int ncopy, const T *b,
                                                                  const T *x, T *xo) {
    pdl_launch_next();
    const int u = blockIdx.x * WAVE_THREADS + threadIdx.x, nthr = (v.nrows + 31) & ~31;
    if (u >= nthr) {   // a warp has rows or copies, never both
        const int j = u - nthr < ncopy ? __ldg(copy + (u - nthr)) : -1;
        pdl_wait_previous();
        if (j >= 0) xo[j] = x[j];
        return;
    }
    RowHead<T, NB> h;
    h.load(v, u, v.nrows);
    const T d = h.i >= 0 ? __ldg(static_cast<const T *>(v.dinv) + u) : T(0);
    pdl_wait_previous();
    T bi = T(0), xi = T(0);
    if (h.i >= 0) {
        bi = b[h.i];
        xi = x[h.i];
    }
    const T acc = h.sum(v, x);
    if (h.i >= 0) xo[h.i] = fma(d, bi - acc, xi);
}

// One-point interpolation (one-point P, or the identity blocks of the nodal hierarchy: at most one entry per
// row, every entry 1): x_i = x_c[col_i] + 0, or 0 for a row without an entry -- the bits of fma(1, x_c[col_i], 0)
// that the sliced-ELL product gives (a -0 becomes +0). One column per row from the dense column array, one
// gather, one write: coalesced everywhere but the gather.
//
// Two flags above the column (P1_MASK) spare the sweeps their copies of the rows they do not touch (split_levels):
// P1_SECOND: the coarse point is a C point of a level whose result lies in two vectors, F points in the first and C
// points in the second; P1_BOTH: the row is a C point, written to x and x2, so that the F sweeps can go from one to the
// other without carrying the C points along.
template <class T>
__device__ __forceinline__ void p1_row(int c, int mask, const T *xc, const T *xc2, T *x, T *x2, int i) {
    const T v = c >= 0 ? ((c & ~mask & P1_SECOND) ? xc2 : xc)[c & mask] + T(0) : T(0);
    x[i] = v;
    if (c >= 0 && (c & ~mask & P1_BOTH)) x2[i] = v;
}

template <class T>
__global__ void __launch_bounds__(256) k_p1_interp(int n, const int *__restrict__ p1col, int mask,
                                                   const int *__restrict__ blk_sys, const uint8_t *run,
                                                   const T *__restrict__ xc, const T *__restrict__ xc2,
                                                   T *__restrict__ x, T *__restrict__ x2) {
    pdl_enter();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (run) {
            const int q = blk_sys[i >> 5];
            if (q >= 0 && !run[q]) continue;
        }
        p1_row<T>(__ldcs(p1col + i), mask, xc, xc2, x, x2, i);
    }
}

// the same for about one wave, a row per thread: the column is read before the previous kernel has finished
template <class T>
__global__ void __launch_bounds__(256) k_p1_interp_wave(int n, const int *p1col, int mask, const int *blk_sys,
                                                        const uint8_t *run, const T *xc, const T *xc2, T *x, T *x2) {
    pdl_launch_next();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    bool on = i < n;
    if (on && run) {
        const int q = blk_sys[i >> 5];
        on = q < 0 || run[q];
    }
    const int c = on ? __ldg(p1col + i) : -1;
    pdl_wait_previous();
    if (on) p1_row<T>(c, mask, xc, xc2, x, x2, i);
}

template <class T>
void p1_interp(int n, const int *p1col, bool flags, const int *blk_sys, const uint8_t *run, const T *xc, const T *xc2,
               T *x, T *x2, cudaStream_t s) {
    if (n <= 0) return;
    const int mask = flags ? P1_MASK : 0x7fffffff;
    if (one_wave<T>(n))
        launch_pdl(k_p1_interp_wave<T>, (n + 255) / 256, 256, 0, s, n, p1col, mask, blk_sys, run, xc, xc2, x, x2);
    else
        launch_pdl(k_p1_interp<T>, grid_for(n, 256, device_sms() * 16), 256, 0, s, n, p1col, mask, blk_sys, run, xc, xc2, x,
                   x2);
    count_launch();
}
template void p1_interp<float>(int, const int *, bool, const int *, const uint8_t *, const float *, const float *, float *,
                               float *, cudaStream_t);
template void p1_interp<double>(int, const int *, bool, const int *, const uint8_t *, const double *, const double *,
                                double *, double *, cudaStream_t);

// adds the flags to a level's columns: cf_c, the coarse level's splitting (NULL: its result is in one vector); cf, the
// level's own (NULL: its sweeps carry all rows along)
__global__ void k_p1_flags(int n, int *__restrict__ p1col, const int8_t *__restrict__ cf, const int8_t *__restrict__ cf_c) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int c = p1col[i];
        if (c < 0) continue;
        if (cf_c && cf_c[c] == CF_C) c |= P1_SECOND;
        if (cf && cf[i] == CF_C) c |= P1_BOTH;
        p1col[i] = c;
    }
}

void launch_p1_flags(int n, int *p1col, const int8_t *cf, const int8_t *cf_c, cudaStream_t s) {
    if (n <= 0) return;
    k_p1_flags<<<grid_for(n, 256), 256, 0, s>>>(n, p1col, cf, cf_c);
    count_launch();
}

// ---------------------------------------------------------------------------------------
// The bottom of the V-cycle in one launch: the restrictions of the smallest levels, the coarsest solve, and on the way
// up their interpolations and F/C sweeps, in one CTA with a block barrier between phases instead of a kernel boundary.
// Every row is computed by one thread with the arithmetic of k_sell_spmv, k_sell_sweep, k_p1_interp and k_dense_apply
// (same entries, same order), so the cycle's result is the same bits either way. Stopped batched systems are not
// skipped here.
//
// What bounds it is latency: read from L2, the chain slice offset -> column -> gathered x -> fma costs over a
// microsecond a phase however few rows there are. So everything the phases read lies in shared memory: level
// descriptors, row lists, diagonals and as many of the views' entries as fit (with 16-bit columns) lie ready in one
// contiguous image, packed when the hierarchy is built (k_bottom_pack), which the kernel copies with 16-byte cp.async
// before it waits for its predecessor (the image does not depend on it). The vectors live in shared memory too. A phase
// then takes 500 to 900 cycles in FP32. Views that do not fit are read from global memory eight entries at a time.
//
// The coarsest product is n^2 FP64 operations on an SM with two FP64 lanes (10 us for n = 128): the CTA is the first of
// a cluster of BOTTOM_CTAS, whose others wait at the cluster barrier, take their share of the rows of that product and
// write them back through distributed shared memory. Spreading the other phases over the cluster as well was slower:
// a cluster barrier after rows were written to eight copies of x takes 1,300 to 2,800 cycles, a block barrier 80.
// 512^2 FD one-point FP32: V-cycle 107 us with a kernel per phase down to the coarsest level, 98 us with this.
// ---------------------------------------------------------------------------------------
namespace {

template <class T>
__device__ __forceinline__ const T *bottom_at(const unsigned char *sm, int off) {
    return reinterpret_cast<const T *>(sm + off);
}

__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();   // .aligned: the warp arrives as one
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the value at shared-memory address a of the cluster, and a store to one
__device__ __forceinline__ void far_load(unsigned a, float &v) {
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void far_load(unsigned a, double &v) {
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void far_store(unsigned a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void far_store(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// the sum of this thread's row of the view against x (shared), entries in ascending order as everywhere
template <class T>
__device__ __forceinline__ T bottom_row(const unsigned char *sm, const BottomView<T> &v, const T *x) {
    const int lane = threadIdx.x & 31;
    const int2 sl = bottom_at<int2>(sm, v.o_ptr)[threadIdx.x >> 5];   // first entry, longest row
    T acc = T(0);
    if (v.o_val >= 0) {
        const uint16_t *col = bottom_at<uint16_t>(sm, v.o_col) + sl.x + lane;
        const T *val = bottom_at<T>(sm, v.o_val) + sl.x + lane;
#pragma unroll 4
        for (int j = 0; j < sl.y; ++j) acc = fma(val[32 * j], x[col[32 * j]], acc);
    } else {
        const int *col = v.col + sl.x + lane;
        const T *val = v.val + sl.x + lane;
        for (int j = 0; j < sl.y; j += 8) {
            int c[8];
            T w[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const bool in = j + k < sl.y;
                c[k] = in ? __ldg(col + 32 * (j + k)) : 0;
                w[k] = in ? __ldg(val + 32 * (j + k)) : T(0);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (j + k < sl.y) acc = fma(w[k], x[c[k]], acc);
        }
    }
    return acc;
}

// y = (view) x
template <class T>
__device__ __forceinline__ void bottom_spmv(const unsigned char *sm, const BottomView<T> &v, const T *x, T *y) {
    if ((int)threadIdx.x >= v.nrows) return;
    const T acc = bottom_row<T>(sm, v, x);
    y[bottom_at<uint16_t>(sm, v.o_row)[threadIdx.x]] = acc;
}

// one Jacobi sweep in place: the new values are written once all rows have read the old ones
template <class T>
__device__ __forceinline__ void bottom_sweep(const unsigned char *sm, const BottomView<T> &v, const T *b, T *x) {
    const bool in = (int)threadIdx.x < v.nrows;
    int i = 0;
    T xn = T(0);
    if (in) {
        i = bottom_at<uint16_t>(sm, v.o_row)[threadIdx.x];
        const T acc = bottom_row<T>(sm, v, x);
        xn = fma(bottom_at<T>(sm, v.o_dinv)[threadIdx.x], b[i] - acc, x[i]);
    }
    __syncthreads();
    if (in) x[i] = xn;
    __syncthreads();
}

}  // namespace

// Lays the image out and fills it, one CTA per view (four per level: R, P, AF, AC). The entries of a view go into the
// image as long as they fit in cap bytes, deepest level first and the F rows (swept twice) before the others; every CTA
// works the layout out for itself from the views' lengths. lv: the levels with the offsets of lists and vectors already
// set (host). The image starts with its own size, then the descriptors; entries take the bytes from o_entries on.
template <class T>
__global__ void __launch_bounds__(256) k_bottom_pack(const BottomLevel<T> *__restrict__ lv, int nl, int o_desc,
                                                     int o_entries, int cap, unsigned char *__restrict__ img) {
    __shared__ int ofs[4 * BOTTOM_LEVELS], beg[4 * BOTTOM_LEVELS], num[4 * BOTTOM_LEVELS], total;
    const int t = threadIdx.x, nv = 4 * nl;
    for (int q = t; q < nv; q += blockDim.x) {
        const BottomView<T> &v = lv[q >> 2].v[q & 3];
        beg[q] = v.nrows > 0 ? v.ptr[0] : 0;
        num[q] = v.nrows > 0 ? v.ptr[(v.nrows + 31) >> 5] - beg[q] : 0;
    }
    __syncthreads();
    if (t == 0) {
        const int order[4] = {BOTTOM_AF, BOTTOM_AC, BOTTOM_R, BOTTOM_P};
        int at = o_entries;
        for (int l = nl - 1; l >= 0; --l)
            for (int k = 0; k < 4; ++k) {
                const int q = 4 * l + order[k];
                const long long bytes = (long long)num[q] * (int)(sizeof(T) + sizeof(uint16_t));   // a multiple of 64
                ofs[q] = -1;
                if (num[q] > 0 && at + bytes <= cap) {
                    ofs[q] = at;
                    at += (int)bytes;
                }
            }
        total = at;
    }
    __syncthreads();
    const int q = blockIdx.x;
    if (q == 0) {
        if (t < 4) reinterpret_cast<int *>(img)[t] = t == 0 ? total : 0;
        const int words = nl * (int)(sizeof(BottomLevel<T>) / sizeof(int));
        for (int k = t; k < words; k += blockDim.x)
            reinterpret_cast<int *>(img + o_desc)[k] = reinterpret_cast<const int *>(lv)[k];
        __syncthreads();
        for (int p = t; p < nv; p += blockDim.x) {
            BottomView<T> &v = reinterpret_cast<BottomLevel<T> *>(img + o_desc)[p >> 2].v[p & 3];
            v.o_val = ofs[p];
            v.o_col = ofs[p] >= 0 ? ofs[p] + num[p] * (int)sizeof(T) : -1;
        }
    }
    const BottomLevel<T> &L = lv[q >> 2];
    const BottomView<T> &v = L.v[q & 3];
    if ((q & 3) == BOTTOM_P && L.p1col)
        for (int k = t; k < L.n; k += blockDim.x) reinterpret_cast<int16_t *>(img + L.o_p1)[k] = (int16_t)L.p1col[k];
    for (int k = t; k < v.nrows; k += blockDim.x) {
        reinterpret_cast<uint16_t *>(img + v.o_row)[k] = (uint16_t)v.row[k];
        if (v.dinv) reinterpret_cast<T *>(img + v.o_dinv)[k] = v.dinv[k];
    }
    for (int k = t; k < (v.nrows + 31) >> 5; k += blockDim.x) {
        const int a = v.ptr[k];
        reinterpret_cast<int2 *>(img + v.o_ptr)[k] = make_int2(ofs[q] >= 0 ? a - beg[q] : a, (v.ptr[k + 1] - a) >> 5);
    }
    if (ofs[q] < 0) return;
    T *val = reinterpret_cast<T *>(img + ofs[q]);
    uint16_t *col = reinterpret_cast<uint16_t *>(img + ofs[q] + num[q] * (int)sizeof(T));
#pragma unroll 4
    for (int k = t; k < num[q]; k += blockDim.x) {
        val[k] = v.val[beg[q] + k];
        col[k] = (uint16_t)v.col[beg[q] + k];
    }
}

template <class T>
__global__ void __cluster_dims__(BOTTOM_CTAS, 1, 1) __launch_bounds__(BOTTOM_THREADS) k_cycle_bottom(BottomArgs<T> a) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, rank = blockIdx.x, n = a.nc, nl = a.nl;
    const int mine = n > rank ? (n - rank + BOTTOM_CTAS - 1) / BOTTOM_CTAS : 0;   // rows rank, rank + 8, ... of Ainv
    pdl_launch_next();
    const unsigned own = (unsigned)__cvta_generic_to_shared(sm);
    unsigned first;   // the first CTA's shared memory
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(first) : "r"(own));
    if (rank == 0) {
        const int total = __ldg(reinterpret_cast<const int *>(a.img));
        for (int k = 16 * t; k < total; k += 16 * BOTTOM_THREADS)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(own + k), "l"(a.img + k) : "memory");
    }
    if (a.o_ainv >= 0)
        for (int k = t; k < mine * n; k += BOTTOM_THREADS)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(own + a.o_ainv + 8 * k),
                         "l"(a.Ainv + (size_t)(rank + k / n * BOTTOM_CTAS) * n + k % n)
                         : "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
    const BottomLevel<T> *lv = bottom_at<BottomLevel<T>>(sm, a.o_desc);   // rank 0 only
    T *cb = reinterpret_cast<T *>(sm + a.o_cb);
    if (rank == 0) {
        pdl_wait_previous();
        if (t < a.n0) reinterpret_cast<T *>(sm + a.o_b0)[t] = a.b[t];
        __syncthreads();
        for (int l = 0; l < nl; ++l) {
            bottom_spmv<T>(sm, lv[l].v[BOTTOM_R], bottom_at<T>(sm, lv[l].o_b),
                           l + 1 < nl ? reinterpret_cast<T *>(sm + lv[l + 1].o_b) : cb);
            __syncthreads();
        }
    }
    cluster_barrier();   // the coarsest right-hand side is complete in the first CTA
    if (rank > 0) {
        if (t < n) {
            T v;
            far_load(first + a.o_cb + t * (int)sizeof(T), v);
            cb[t] = v;
        }
        __syncthreads();
    }
    // x = Ainv b, row rank + 8 k in this CTA, four rows per warp. A lane sums its columns in ascending order and the
    // lanes' sums are added in k_dense_apply's butterfly order (16, 8, 4, 2, 1), but four rows share the first two
    // steps: each half, then each quarter of the warp goes on with its own rows (a warp FP64 instruction takes 19
    // cycles of the SM whatever its lanes hold).
    for (int r0 = 4 * w; r0 < mine; r0 += 4 * (BOTTOM_THREADS / 32)) {
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        if (a.o_ainv >= 0) {
            const double *A = bottom_at<double>(sm, a.o_ainv) + r0 * n;
#pragma unroll 2
            for (int c = lane; c < n; c += 32) {
                const double xc = (double)cb[c];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (r0 + k < mine) acc[k] = fma(A[k * n + c], xc, acc[k]);
            }
        } else {
            const double *A = a.Ainv + (size_t)(rank + r0 * BOTTOM_CTAS) * n;
#pragma unroll 4
            for (int c = lane; c < n; c += 32) {
                const double xc = (double)cb[c];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (r0 + k < mine) acc[k] = fma(__ldg(A + (size_t)k * BOTTOM_CTAS * n + c), xc, acc[k]);
            }
        }
        const bool h16 = lane & 16, h8 = lane & 8;
        const double s0 = __shfl_xor_sync(0xffffffffu, h16 ? acc[0] : acc[2], 16);
        const double s1 = __shfl_xor_sync(0xffffffffu, h16 ? acc[1] : acc[3], 16);
        const double p0 = (h16 ? acc[2] : acc[0]) + s0, p1 = (h16 ? acc[3] : acc[1]) + s1;
        double v = (h8 ? p1 : p0) + __shfl_xor_sync(0xffffffffu, h8 ? p0 : p1, 8);
        for (int o = 4; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        const int k = (h16 ? 2 : 0) + (h8 ? 1 : 0);
        if ((lane & 7) == 0 && r0 + k < mine)
            far_store(first + a.o_cx + (rank + (r0 + k) * BOTTOM_CTAS) * (int)sizeof(T), (T)v);
    }
    cluster_barrier();   // the coarsest solution is complete in the first CTA
    if (rank > 0) return;
    const int sq[3] = {a.seq.x, a.seq.y, a.seq.z};
    for (int l = nl - 1; l >= 0; --l) {
        const BottomLevel<T> &L = lv[l];
        const T *xc = bottom_at<T>(sm, l + 1 < nl ? lv[l + 1].o_x : a.o_cx);
        T *x = reinterpret_cast<T *>(sm + L.o_x);
        if (L.p1col) {
            if (t < L.n) {
                const int c = bottom_at<int16_t>(sm, L.o_p1)[t];
                x[t] = c >= 0 ? xc[c] + T(0) : T(0);
            }
        } else {
            bottom_spmv<T>(sm, L.v[BOTTOM_P], xc, x);
        }
        __syncthreads();
        for (int k = 0; k < 3 && sq[k] >= 0; ++k)
            bottom_sweep<T>(sm, L.v[sq[k] == CF_F ? BOTTOM_AF : BOTTOM_AC], bottom_at<T>(sm, L.o_b), x);
    }
    if (t < a.n0) a.x[t] = bottom_at<T>(sm, a.o_x0)[t];
}

template <class T>
void bottom_pack(const BottomLevel<T> *lv, int nl, int o_desc, int o_entries, int cap, unsigned char *img,
                 cudaStream_t s) {
    k_bottom_pack<T><<<4 * nl, 256, 0, s>>>(lv, nl, o_desc, o_entries, cap, img);
    count_launch();
}
template void bottom_pack<float>(const BottomLevel<float> *, int, int, int, int, unsigned char *, cudaStream_t);
template void bottom_pack<double>(const BottomLevel<double> *, int, int, int, int, unsigned char *, cudaStream_t);

// whether the device can hold the bottom kernel's cluster
template <class T>
bool bottom_fits() {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(BOTTOM_CTAS);
    cfg.blockDim = dim3(BOTTOM_THREADS);
    cfg.dynamicSmemBytes = BOTTOM_SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = BOTTOM_CTAS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    const bool ok = cudaFuncSetAttribute(k_cycle_bottom<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, BOTTOM_SMEM) ==
                        cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&n, k_cycle_bottom<T>, &cfg) == cudaSuccess && n > 0;
    if (!ok) cudaGetLastError();
    return ok;
}
template bool bottom_fits<float>();
template bool bottom_fits<double>();

template <class T>
void cycle_bottom(const BottomArgs<T> &a, cudaStream_t s) {
    launch_pdl(k_cycle_bottom<T>, BOTTOM_CTAS, BOTTOM_THREADS, BOTTOM_SMEM, s, a);
    count_launch();
}
template void cycle_bottom<float>(const BottomArgs<float> &, cudaStream_t);
template void cycle_bottom<double>(const BottomArgs<double> &, cudaStream_t);

// the system of every 32-row block: that of its first row when its last row has the same one, else -1
__global__ void k_blk_sys(int n, const int *__restrict__ seg, int nseg, int *__restrict__ blk_sys) {
    const int nb = (n + 31) >> 5;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) {
        const int q0 = system_of(seg, nseg, 32 * b), q1 = system_of(seg, nseg, min(32 * b + 31, n - 1));
        blk_sys[b] = q0 == q1 ? q0 : -1;
    }
}

void launch_blk_sys(int n, const int *seg, int nseg, int *blk_sys, cudaStream_t s) {
    if (n <= 0) return;
    k_blk_sys<<<grid_for((n + 31) / 32, 256), 256, 0, s>>>(n, seg, nseg, blk_sys);
    count_launch();
}

// the dense column array of a P with at most one entry per row
__global__ void k_p1_cols(int n, const int *__restrict__ rp, const int *__restrict__ col, int *__restrict__ p1col) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        p1col[i] = rp[i + 1] > rp[i] ? col[rp[i]] : -1;
}

void launch_p1_cols(int n, const int *rp, const int *col, int *p1col, cudaStream_t s) {
    if (n <= 0) return;
    k_p1_cols<<<grid_for(n, 256), 256, 0, s>>>(n, rp, col, p1col);
    count_launch();
}

// The outer iteration's product y = A z with z = the cycle's result x (FP32, widened exactly, or FP64), which is also
// written out: in one kernel, whose gathers read half the bytes in mixed precision, or as a conversion and
// k_sell_spmv<double>, whose arithmetic the kernel has.
template <class T>
__global__ void __launch_bounds__(256) k_sell_spmv_keep(SellView v, const T *x, double *z, double *y) {
    pdl_enter();
    const int *__restrict__ sptr = v.slice_ptr;
    const int *__restrict__ scol = v.col;
    const double *__restrict__ sval = static_cast<const double *>(v.val);
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < v.nrows; q += gridDim.x * blockDim.x) {
        const int sl = q >> 5;
        bool on = true;
        if (v.run) {
            const int sy = v.slice_sys[sl];
            on = sy < 0 || v.run[sy];
        }
        const int a = __ldg(sptr + sl), base = a + (q & 31);
        const int len = on ? (__ldg(sptr + sl + 1) - a) >> 5 : 0;   // a stopped system: y = 0, which nothing reads
        const int i = __ldg(v.row + q);
        double acc = 0.0;
#pragma unroll 4
        for (int j = 0; j < len; ++j) acc = fma(__ldcs(sval + base + 32 * j), (double)x[__ldcs(scol + base + 32 * j)], acc);
        y[i] = acc;
        z[i] = (double)x[i];
    }
}

// Both ways give the same bits. Which one: the fused kernel converts x once per entry, on FP64 units that take as long
// for a conversion as for an fma, the pair once per row; the pair costs a launch and reads x again. In mixed precision
// they cross at about KEEP_ENTRIES_PER_SM entries (us, fused / pair): 300^2 8.0 / 10.6, 512^2 11.9 / 12.5, 700^2 17.2 /
// 17.2, 900^2 23.7 / 22.3; 42^3 8.6 / 10.8, 53^3 11.1 / 12.3, 64^3 13.8 / 13.2, 101^3 36 / 30, 150^3 107 / 74; DG-P2 64^2
// 9.6 / 11.7, 90^2 11.6 / 12.7, 110^2 13.7 / 13.4, 150^2 17.9 / 16.0, 256^2 40 / 31. Batches keep the fused kernel, which
// does not work on systems that have stopped (512 systems, mean of all iterations: 123.5 / 125.3). A form with one row
// per thread and the matrix read ahead, as in the cycle, was slower: 53^3 16.8, FP64 11.9 against 9.4.
constexpr int KEEP_ENTRIES_PER_SM = 10240;

template <class T>
void sell_spmv_keep(const SellView &v, long long nnz, const T *x, double *z, double *y, cudaStream_t s) {
    if (v.nrows <= 0) return;
    const int grid = grid_for(v.nrows, 256, device_sms() * 16);
    if constexpr (sizeof(T) == 4) {
        if (!v.run && nnz > (long long)KEEP_ENTRIES_PER_SM * device_sms()) {
            f2d(v.nrows, x, z, s);
            launch_pdl(k_sell_spmv<double, 1>, grid, 256, 0, s, v, (const double *)z, y);
            count_launch();
            return;
        }
    }
    launch_pdl(k_sell_spmv_keep<T>, grid, 256, 0, s, v, x, z, y);
    count_launch();
}
template void sell_spmv_keep<float>(const SellView &, long long, const float *, double *, double *, cudaStream_t);
template void sell_spmv_keep<double>(const SellView &, long long, const double *, double *, double *, cudaStream_t);

// r = b - A x over all rows of an FP64 view of A (r and its FP32 copy each optional), and the block partial
// of |r|^2 in part[blockIdx.x] (gridDim.x = RED_PARTS blocks, summed by finish_residual)
constexpr int RES_THREADS = 512;

__global__ void __launch_bounds__(RES_THREADS) k_sell_residual(SellView v, const double *__restrict__ b,
                                                               const double *__restrict__ x, double *__restrict__ r,
                                                               float *__restrict__ r32, double *__restrict__ part) {
    __shared__ double red[RES_THREADS / 32];
    const int *__restrict__ sptr = v.slice_ptr;
    const int *__restrict__ scol = v.col;
    const double *__restrict__ sval = static_cast<const double *>(v.val);
    double ss = 0.0;
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < v.nrows; q += gridDim.x * blockDim.x) {
        const int sl = q >> 5;
        const int base = __ldg(sptr + sl) + (q & 31);
        const int len = (__ldg(sptr + sl + 1) - __ldg(sptr + sl)) >> 5;
        double acc = 0.0;
#pragma unroll 4
        for (int j = 0; j < len; ++j) acc = fma(__ldcs(sval + base + 32 * j), __ldg(x + __ldcs(scol + base + 32 * j)), acc);
        const int i = v.row[q];
        const double ri = b[i] - acc;
        if (r) r[i] = ri;
        if (r32) r32[i] = (float)ri;
        ss = fma(ri, ri, ss);
    }
    for (int o = 16; o >= 1; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < RES_THREADS / 32; ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

void sell_residual(const SellView &v, const double *b, const double *x, double *r, float *r32, double *part,
                   cudaStream_t s) {
    k_sell_residual<<<RED_PARTS, RES_THREADS, 0, s>>>(v, b, x, r, r32, part);
    count_launch();
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
void launch_frows(int n, const int8_t *cf, const int *cscan, int *frows, cudaStream_t s) {
    k_frows<<<grid_for(n, 256), 256, 0, s>>>(n, cf, cscan, frows);
    count_launch();
}

void launch_sell_prepare_multi(const SellDesc *d, int nd, int nwin, int nlin, int *cnt, unsigned long long *gsum,
                               cudaStream_t s) {
    if (nwin <= 0) return;
    k_sell_sort_multi<<<grid_for((long long)nwin, SORT_WARPS, device_sms() * 16), 32 * SORT_WARPS, 0, s>>>(d, nd, nwin);
    k_sell_len_multi<<<grid_for((long long)nlin * 32, 256), 256, 0, s>>>(d, nd, nlin, cnt, gsum);
    count_launch(2);
}

void launch_sell_fill_multi(const SellDesc *d, int p0, int p1, int lin_beg, int lin_end, bool fp32, cudaStream_t s) {
    if (p1 <= p0 || lin_end <= lin_beg) return;
    const int grid = grid_for(32ll * (lin_end - lin_beg), 256);
    if (fp32) k_sell_fill_multi<float><<<grid, 256, 0, s>>>(d, p0, p1, lin_end);
    else k_sell_fill_multi<double><<<grid, 256, 0, s>>>(d, p0, p1, lin_end);
    count_launch();
}

template <class T>
void sell_spmv(const SellView &v, const T *x, T *y, cudaStream_t s) {
    if (v.nrows <= 0) return;
    if (v.tb == 0 && one_wave<T>(v.nrows)) {
        const int grid = (v.nrows + WAVE_THREADS - 1) / WAVE_THREADS;
        if (v.long_rows) launch_pdl(k_sell_spmv_wave<T, 16>, grid, WAVE_THREADS, 0, s, v, x, y);
        else launch_pdl(k_sell_spmv_wave<T, 8>, grid, WAVE_THREADS, 0, s, v, x, y);
        count_launch();
        return;
    }
    // every row is summed alone by one thread, so the schedule (block size, grid cap, rows per thread) never
    // changes the result
    const int tb = v.tb > 0 ? v.tb : 256;
    const int cap = v.grid > 0 ? v.grid : device_sms() * 16;
    const long long nsl = (v.nrows + 31) / 32;
    if (v.rpt == 2) launch_pdl(k_sell_spmv<T, 2>, grid_for((nsl + 1) / 2 * 32, tb, cap), tb, 0, s, v, x, y);
    else launch_pdl(k_sell_spmv<T, 1>, grid_for(nsl * 32, tb, cap), tb, 0, s, v, x, y);
    count_launch();
}

template <class T>
void sell_sweep(const SellView &v, const int *copy, int ncopy, const T *b, const T *x, T *xo, cudaStream_t s) {
    if (v.nrows + ncopy <= 0) return;
    if (v.tb == 0 && one_wave<T>((long long)v.nrows + ncopy)) {
        const int grid = (((v.nrows + 31) & ~31) + ncopy + WAVE_THREADS - 1) / WAVE_THREADS;
        if (v.long_rows) launch_pdl(k_sell_sweep_wave<T, 16>, grid, WAVE_THREADS, 0, s, v, copy, ncopy, b, x, xo);
        else launch_pdl(k_sell_sweep_wave<T, 8>, grid, WAVE_THREADS, 0, s, v, copy, ncopy, b, x, xo);
        count_launch();
        return;
    }
    const int tb = v.tb > 0 ? v.tb : 256;
    const int cap = v.grid > 0 ? v.grid : device_sms() * 16;
    const long long nsl = (v.nrows + 31) / 32;
    if (v.rpt == 2)
        launch_pdl(k_sell_sweep<T, 2>, grid_for((nsl + 1) / 2 * 32 + ncopy, tb, cap), tb, 0, s, v, copy, ncopy, b, x, xo);
    else
        launch_pdl(k_sell_sweep<T, 1>, grid_for(nsl * 32 + ncopy, tb, cap), tb, 0, s, v, copy, ncopy, b, x, xo);
    count_launch();
}

template void sell_spmv<float>(const SellView &, const float *, float *, cudaStream_t);
template void sell_spmv<double>(const SellView &, const double *, double *, cudaStream_t);
template void sell_sweep<float>(const SellView &, const int *, int, const float *, const float *, float *, cudaStream_t);
template void sell_sweep<double>(const SellView &, const int *, int, const double *, const double *, double *,
                                 cudaStream_t);

}  // namespace lair
