// The coarsest level's solve (included by solver.cu inside its anonymous
// namespace): x = A^{-1} b with the explicit inverse of the operator of at most
// kMaxCoarse cells, formed once per coefficient set.
//
// The inverse comes from a banded L D L^T (A is a symmetric M-matrix: no
// pivoting) with the cells numbered so that the longest side is slowest -- half
// bandwidth w = the product of the two shorter sides, at most 56 -- and one pair
// of triangular solves per unit vector, a warp each.  Every CTA factors the
// whole band in its own shared memory (the factor is a chain of n steps, each
// w^2 / 2 multiply-adds and one barrier: nothing to gain from sharing it) and
// then solves the columns of its own warps, so one launch does both.  Bound by
// that chain's latency.  A dense LU in global memory by one CTA took 54 ms at
// 14x5x7 cells and 3.2 ms at 20x9 per coefficient set, and its triangular solves
// 1.2 ms and 0.18 ms per V-cycle, n dependent warp reductions each.

// A sub-grid of nx (fastest) x nm x ns cells; a 2D level has nm = 1 and its rows
// on the slow axis, so its beta_v is bz here.
template <typename T>
struct CoarseOp {
    int nx, nm, ns, n, w, sx, sm, ss;  // sx, sm, ss: strides of the banded numbering
    const T *bx, *by, *bz;
};

template <typename T>
CoarseOp<T> coarse_op(const Level<T> &C)
{
    const bool d3 = C.bw != nullptr;
    CoarseOp<T> o;
    o.nx = C.nx;
    o.nm = d3 ? C.ny : 1;
    o.ns = d3 ? C.nz : C.ny;
    o.n = o.nx * o.nm * o.ns;
    o.bx = C.bu;
    o.by = d3 ? C.bv : nullptr;
    o.bz = d3 ? C.bw : C.bv;
    if (o.nx >= o.nm && o.nx >= o.ns) {
        o.sm = 1, o.ss = o.nm, o.sx = o.w = o.nm * o.ns;
    } else if (o.ns >= o.nm) {
        o.sx = 1, o.sm = o.nx, o.ss = o.w = o.nx * o.nm;
    } else {
        o.sx = 1, o.ss = o.nx, o.sm = o.w = o.nx * o.ns;
    }
    return o;
}

// Band storage in elements: rows of w + 1 (diagonal, then the w entries below it).
template <typename T>
size_t coarse_band_elems(const CoarseOp<T> &o)
{
    return (size_t)o.n * (o.w + 1);
}

// gband: where the band lives if it does not fit in shared memory (one CTA then).
template <typename T>
__global__ void __launch_bounds__(1024) k_coarse_inverse(CoarseOp<T> o, int ncw, T *gband, T *inv)
{
    pdl_entry();
    extern __shared__ __align__(16) unsigned char coarse_smem[];
    T *const dinv = reinterpret_cast<T *>(coarse_smem);
    T *const ys = dinv + o.n;
    T *const band = gband ? gband : ys + (size_t)ncw * o.n;
    const int n = o.n, w = o.w, w1 = w + 1, tid = threadIdx.x, nt = blockDim.x;
    for (int q = tid; q < n * w1; q += nt) band[q] = T(0);
    __syncthreads();
    for (int c = tid; c < n; c += nt) {
        const int r = c / o.nx, i = c - r * o.nx, k = r / o.nm, j = r - k * o.nm;
        const int fx = r * (o.nx + 1) + i, fy = (r + k) * o.nx + i, p = i * o.sx + j * o.sm + k * o.ss;
        const int pl = o.nx * o.nm;
        T *row = band + (size_t)p * w1;
        T d = T(0);
        if (i > 0) d += o.bx[fx];
        if (i < o.nx - 1) {
            d += o.bx[fx + 1];
            row[o.sx] = -o.bx[fx + 1];
        }
        if (j > 0) d += o.by[fy];
        if (j < o.nm - 1) {
            d += o.by[fy + o.nx];
            row[o.sm] = -o.by[fy + o.nx];
        }
        if (k > 0) d += o.bz[c];
        d += (k < o.ns - 1 ? T(1) : T(2)) * o.bz[c + pl];
        if (k < o.ns - 1) row[o.ss] = -o.bz[c + pl];
        row[0] = d;
        if (p == 0) dinv[0] = T(1) / d;
    }
    __syncthreads();
    // A = L D L^T; the band keeps D L^T's rows (unscaled), dinv the 1 / D.  A
    // thread's entries (r, s), 1 <= s <= r <= w, of the step's update are the same
    // in every step: at most two (w <= 56, or the block covers them).
    constexpr int kPairs = 2;
    int pr[kPairs], ps[kPairs], pd[kPairs];  // r; s; offset of row k + s, entry r - s, from row k
#pragma unroll
    for (int u = 0; u < kPairs; ++u) {
        const int e = tid + u * nt;
        int r = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
        while ((r + 1) * (r + 2) / 2 <= e) ++r;
        while (r * (r + 1) / 2 > e) --r;
        const int sq = e - r * (r + 1) / 2;
        pr[u] = ++r;
        ps[u] = sq + 1;
        pd[u] = (sq + 1) * w1 + (r - sq - 1);
    }
    for (int k = 0; k + 1 < n; ++k) {
        const T di = dinv[k];
        const int m = min(w, n - 1 - k);
        T *row = band + (size_t)k * w1;
#pragma unroll
        for (int u = 0; u < kPairs; ++u) {
            const int r = pr[u];
            if (r > m) continue;
            T *a = row + pd[u];
            const T v = *a - row[r] * di * row[ps[u]];
            *a = v;
            if (r == 1) dinv[k + 1] = T(1) / v;
        }
        __syncthreads();
    }
    // column t of A^{-1}: L y = e_t, z = D^{-1} y, L^T x = z
    const int lane = tid & 31, wp = tid >> 5;
    if (wp >= ncw) return;
    T *const y = ys + (size_t)wp * n;
    for (int t = blockIdx.x * ncw + wp; t < n; t += gridDim.x * ncw) {
        const int tr = t / o.nx, tk = tr / o.nm;
        const int pt = (t - tr * o.nx) * o.sx + (tr - tk * o.nm) * o.sm + tk * o.ss;
        for (int k = lane; k < n; k += 32) y[k] = k == pt ? T(1) : T(0);
        __syncwarp();
        // (w <= 56: at most two entries of a row per lane, the next row's loaded ahead)
        auto ld = [&](int k, int r) { return k < n && r <= min(w, n - 1 - k) ? band[(size_t)k * w1 + r] : T(0); };
        T a0 = ld(pt, lane + 1), a1 = ld(pt, lane + 33);
        for (int k = pt; k < n; ++k) {
            const T g = y[k] * dinv[k];
            const int m = min(w, n - 1 - k);
            const T c0 = a0, c1 = a1;
            a0 = ld(k + 1, lane + 1);
            a1 = ld(k + 1, lane + 33);
            if (lane + 1 <= m) y[k + lane + 1] -= c0 * g;
            if (lane + 33 <= m) y[k + lane + 33] -= c1 * g;
            __syncwarp();
        }
        for (int k = lane; k < n; k += 32) y[k] *= dinv[k];
        __syncwarp();
        auto lt = [&](int k, int r) { return r <= min(w, k) ? band[(size_t)(k - r) * w1 + r] * dinv[k - r] : T(0); };
        a0 = lt(n - 1, lane + 1);
        a1 = lt(n - 1, lane + 33);
        for (int k = n - 1; k > 0; --k) {
            const T xk = y[k];
            const int m = min(w, k);
            const T c0 = a0, c1 = a1;
            a0 = lt(k - 1, lane + 1);
            a1 = lt(k - 1, lane + 33);
            if (lane + 1 <= m) y[k - lane - 1] -= c0 * xk;
            if (lane + 33 <= m) y[k - lane - 33] -= c1 * xk;
            __syncwarp();
        }
        for (int c = lane; c < n; c += 32) {
            const int r = c / o.nx, k = r / o.nm;
            inv[(size_t)t * n + c] = y[(c - r * o.nx) * o.sx + (r - k * o.nm) * o.sm + k * o.ss];
        }
        __syncwarp();
    }
}

// One row of the inverse times b, by a warp: lanes over the columns, a fixed
// shuffle tree (every lane gets the value).  Both coarsest-level solves -- the
// kernel below and the cluster kernel -- go through it, so they give the same bits.
template <typename T>
__device__ __forceinline__ T inv_row(const T *__restrict__ row, const T *b, int n, int lane)
{
    T s = T(0);
    for (int c = lane; c < n; c += 32) s = fma3(row[c], b[c], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// x = A^{-1} b, a warp per row (8 rows per CTA).
template <typename T>
__global__ void __launch_bounds__(256) k_coarse_solve(int n, const T *__restrict__ inv, const T *__restrict__ b,
                                                      T *__restrict__ x, const int *bsel, const int *xsel)
{
    pdl_entry();
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= n) return;
    b = at_sel(b, bsel, n);
    x = at_sel(x, xsel, n);
    const T s = inv_row(inv + (size_t)r * n, b, n, lane);
    if (lane == 0) x[r] = s;
}

template <typename T>
T *coarse_inv(const wec_poisson *P)
{
    if constexpr (sizeof(T) == 8) return P->inv64; else return P->inv32;
}

// the matrix of the dense level (P->dense, mg_cluster.cuh): its own where that level is not the coarsest
template <typename T>
T *dense_mat(const wec_poisson *P)
{
    if constexpr (sizeof(T) == 8) return P->dense64; else return P->dense32;
}

constexpr int kCoarseSmem = 227 * 1024;

// inv <- the inverse of level C's operator (n x n); band: n x (w + 1) scratch for
// a band that exceeds shared memory (FP64 with n w above ~28,000).
template <typename T>
void launch_coarse_inverse(const Level<T> &C, T *inv, T *band, cudaStream_t st)
{
    const CoarseOp<T> o = coarse_op(C);
    const size_t be = coarse_band_elems(o);
    const int threads = std::min(1024, std::max(128, (o.w * (o.w + 1) / 2 + 31) / 32 * 32));
    // columns per CTA: a warp each, enough CTAs that one round covers them where they fit
    int ncw = std::min(threads / 32, std::max(2, (o.n + 147) / 148));
    auto bytes = [&](int c) { return (be + (size_t)(c + 1) * o.n) * sizeof(T); };
    while (ncw > 1 && bytes(ncw) > kCoarseSmem) --ncw;
    const bool fits = bytes(ncw) <= kCoarseSmem;
    if (!fits) ncw = threads / 32;
    const size_t smem = fits ? bytes(ncw) : (size_t)(ncw + 1) * o.n * sizeof(T);
    launch_k(k_coarse_inverse<T>, fits ? (o.n + ncw - 1) / ncw : 1, threads, smem, st, o, ncw, fits ? (T *)nullptr : band,
             inv);
}
