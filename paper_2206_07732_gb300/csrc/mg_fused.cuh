// Fused multigrid V-cycle kernels (included by solver.cu).
//
// The V-cycle of solver.cu -- red-black Gauss-Seidel, residual restriction by
// the sum of four children, piecewise-constant prolongation -- launched as:
//   k_mg_pre    per fine level: nu1 smoothing sweeps from x = 0, the residual and
//               its restriction, in one kernel.  Each CTA owns a TX x TY tile and
//               loads it with a halo of H = 2 max(nu1, nu2) cells into shared
//               memory; a colour pass leaves exact values one cell further in
//               than the previous one (the first red pass from x = 0 reads no
//               neighbour), so after 2 nu1 passes the tile and one ring around
//               it are exact, which is what the residual needs.  Halo cells are
//               recomputed redundantly.
//   k_mg_cluster (mg_cluster.cuh) the coarse levels, down to the coarsest level's
//               solve and back up.
//   k_mg_post   per fine level: prolongation + correction and nu2 sweeps, same
//               tiling.
// A cell update is x = (b + sum_f beta_f x_nb) * (1 / d) with the reciprocal of
// the diagonal formed once per coefficient set (poisson_build) and staged with
// the tile (the one-pass kernels of solver.cu divide by d instead: the two
// V-cycles agree to rounding).  Face
// coefficients are zero on the Neumann walls and x is zero outside the domain,
// so a tile update needs no boundary branches (the staging zeroes the wall
// faces); 1/d is zero outside the domain, which keeps those cells at zero.
#pragma once

namespace wec {
namespace {

// Tile shapes (interior cells) of the fused level kernels; the autotuner picks
// one per level and precision.
constexpr int kNumTiles = 4;
constexpr int kTileX[kNumTiles] = {64, 32, 32, 16};
constexpr int kTileY[kNumTiles] = {16, 16, 8, 8};

// q = k / d for 0 <= k < 2^16, 2 <= d < 2^16 by one multiply-high with m = magic_u16(d):
// with m = floor(2^32 / d) + 1 the error term k (m - 2^32 / d) / 2^32 < 2^-16 < 1 / d.
__host__ __device__ inline unsigned magic_u16(unsigned d) { return 0xffffffffu / d + 1u; }
__device__ __forceinline__ int div_u16(int k, unsigned m) { return (int)__umulhi((unsigned)k, m); }

// One element global -> shared without a register round trip (cp.async); with
// in == false the element is zero-filled and nothing is read (src must still be
// a valid address).  Completed by cp_async_wait_all() + __syncthreads().
template <typename T>
__device__ __forceinline__ void cp_async_el(T *dst, const T *src, bool in = true)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = in ? (int)sizeof(T) : 0;
    if constexpr (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

template <typename T>
struct TileView {
    int ex, ey, gx0, gy0, nx, ny;
    T *x, *b, *id, *bu, *bv;  // shared: x, b, 1/d [ey][ex]; bu[ey][ex+1]; bv[ey+1][ex]

    // d of cell (li, lj), as diag_at: the top row's Dirichlet face counts twice
    __device__ __forceinline__ T diag(int li, int lj) const
    {
        const T f = gy0 + lj == ny - 1 ? T(2) : T(1);
        return ((bu[lj * (ex + 1) + li] + bu[lj * (ex + 1) + li + 1]) + bv[lj * ex + li]) + f * bv[(lj + 1) * ex + li];
    }

    // sum_f beta_f x_nb, as offsum_at (walls have beta = 0, outside x = 0)
    __device__ __forceinline__ T offsum(int li, int lj) const
    {
        const int c = lj * ex + li;
        return ((bu[lj * (ex + 1) + li] * x[c - 1] + bu[lj * (ex + 1) + li + 1] * x[c + 1]) + bv[lj * ex + li] * x[c - ex]) +
               bv[(lj + 1) * ex + li] * x[c + ex];
    }
};

// Stage b, 1/d, x (xg + prolonged xc when xg is given, else 0), bu, bv of the
// tile (zero outside the domain; bu, bv also zero on the Neumann walls).
template <typename T>
__device__ void tile_load(TileView<T> &t, const T *__restrict__ bu, const T *__restrict__ bv,
                          const T *__restrict__ b, const T *__restrict__ idg, const T *xg, const T *__restrict__ xc)
{
    const int nx = t.nx, ny = t.ny, ex = t.ex, ey = t.ey;
    const unsigned mex = magic_u16(ex), mex1 = magic_u16(ex + 1);
    for (int k = threadIdx.x; k < ex * ey; k += blockDim.x) {
        const int lj = div_u16(k, mex), li = k - lj * ex, gi = t.gx0 + li, gj = t.gy0 + lj;
        const bool in = gi >= 0 && gi < nx && gj >= 0 && gj < ny;
        cp_async_el(t.b + k, in ? b + gj * nx + gi : b, in);
        cp_async_el(t.id + k, in ? idg + gj * nx + gi : idg, in);
    }
    for (int k = threadIdx.x; k < (ex + 1) * ey; k += blockDim.x) {
        const int lj = div_u16(k, mex1), li = k - lj * (ex + 1), gi = t.gx0 + li, gj = t.gy0 + lj;
        const bool in = gi > 0 && gi < nx && gj >= 0 && gj < ny;  // Neumann wall faces count as zero
        cp_async_el(t.bu + k, in ? bu + gj * (nx + 1) + gi : bu, in);
    }
    for (int k = threadIdx.x; k < ex * (ey + 1); k += blockDim.x) {
        const int lj = div_u16(k, mex), li = k - lj * ex, gi = t.gx0 + li, gj = t.gy0 + lj;
        const bool in = gi >= 0 && gi < nx && gj > 0 && gj <= ny;  // bottom wall zero, top (Dirichlet) kept
        cp_async_el(t.bv + k, in ? bv + gj * nx + gi : bv, in);
    }
#pragma unroll 4
    for (int k = threadIdx.x; k < ex * ey; k += blockDim.x) {
        const int lj = div_u16(k, mex), li = k - lj * ex, gi = t.gx0 + li, gj = t.gy0 + lj;
        T xv = T(0);
        if (xg && gi >= 0 && gi < nx && gj >= 0 && gj < ny)
            xv = xg[gj * nx + gi] + xc[(gj >> 1) * (nx >> 1) + (gi >> 1)];
        t.x[k] = xv;
    }
    cp_async_wait_all();
    __syncthreads();
}

// One colour pass over the tile's cells at least m from its edge: the ones a later
// pass, the residual or the result still needs -- each pass before the last needs
// one ring more than the one after it (passing over the whole tile every time spent
// 1.3 times the updates in FP64, where the pipe bounds them).  first: from x = 0,
// b / d.  Threads walk the cells of the colour.
template <typename T>
__device__ void tile_pass(TileView<T> &t, int color, bool first, int m, unsigned mwh)
{
    const int ex = t.ex, ey = t.ey, wh = ex >> 1;
    const int par = (color - t.gx0 - t.gy0) & 1;  // column parity of the colour in row 0
    for (int k = threadIdx.x + m * wh; k < wh * (ey - m); k += blockDim.x) {
        const int lj = div_u16(k, mwh), q = k - lj * wh;
        const int li = 2 * q + ((par - lj) & 1);
        const int c = lj * ex + li;
        if (first) {
            t.x[c] = t.b[c] * t.id[c];
        } else if (li >= m && li < ex - m) {
            t.x[c] = (t.b[c] + t.offsum(li, lj)) * t.id[c];
        }
    }
    __syncthreads();
}

template <typename T>
__device__ __forceinline__ void tile_setup(TileView<T> &t, unsigned char *smem_raw, int nx, int ny, int kTX, int kTY,
                                           int H)
{
    t.nx = nx;
    t.ny = ny;
    t.ex = kTX + 2 * H;
    t.ey = kTY + 2 * H;
    t.gx0 = blockIdx.x * kTX - H;
    t.gy0 = blockIdx.y * kTY - H;
    T *p = reinterpret_cast<T *>(smem_raw);
    t.x = p;
    t.b = t.x + t.ex * t.ey;
    t.id = t.b + t.ex * t.ey;
    t.bu = t.id + t.ex * t.ey;
    t.bv = t.bu + (t.ex + 1) * t.ey;
}

// nu1 sweeps from zero, then the smoothed iterate (tile interior) into xp and
// the restricted residual into bc.
template <typename T, int kTX, int kTY>
__global__ void __launch_bounds__(256) k_mg_pre(int nx, int ny, const T *__restrict__ bu, const T *__restrict__ bv,
                                                const T *__restrict__ b, const T *__restrict__ idg,
                                                T *__restrict__ xp, T *__restrict__ bc, int nu1, int H,
                                                const int *bsel)
{
    pdl_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const long long n = (long long)nx * ny;
    b = at_sel(b, bsel, n);
    TileView<T> t;
    tile_setup(t, smem_raw, nx, ny, kTX, kTY, H);
    const unsigned mwh = magic_u16(t.ex >> 1);
    tile_load(t, bu, bv, b, idg, (const T *)nullptr, (const T *)nullptr);
    // pass p of 2 nu1 leaves what the residual on the tile needs: a ring around it
    // and one ring per pass to come
    const int m0 = H - 2 * nu1;
    for (int q = 0; q < nu1; ++q) {
        tile_pass(t, 0, q == 0, m0 + 2 * q, mwh);
        tile_pass(t, 1, false, m0 + 2 * q + 1, mwh);
    }
    const int ncx = nx >> 1, ncy = ny >> 1;
    for (int k = threadIdx.x; k < (kTX / 2) * (kTY / 2); k += blockDim.x) {
        int I = k % (kTX / 2), J = k / (kTX / 2);
        int gI = blockIdx.x * (kTX / 2) + I, gJ = blockIdx.y * (kTY / 2) + J;
        if (gI >= ncx || gJ >= ncy) continue;
        T r[4];
        int qq = 0;
        for (int dj = 0; dj < 2; ++dj)
            for (int di = 0; di < 2; ++di) {
                int li = H + 2 * I + di, lj = H + 2 * J + dj, c = lj * t.ex + li;
                T ax = t.diag(li, lj) * t.x[c] - t.offsum(li, lj);
                r[qq++] = t.b[c] - ax;
            }
        bc[gJ * ncx + gI] = ((r[0] + r[1]) + r[2]) + r[3];
    }
    for (int k = threadIdx.x; k < kTX * kTY; k += blockDim.x) {
        int li = H + k % kTX, lj = H + k / kTX, gi = t.gx0 + li, gj = t.gy0 + lj;
        if (gi < nx && gj < ny) xp[gj * nx + gi] = t.x[lj * t.ex + li];
    }
}

// x = xp + P x_c, then nu2 sweeps; writes the tile interior of x (in TO: the
// level-0 result of an FP32 V-cycle is stored widened to FP64).  Reads xp and
// writes x (different arrays): tiles read their halos while others write.
template <typename T, int kTX, int kTY, typename TO>
__global__ void __launch_bounds__(256) k_mg_post(int nx, int ny, const T *__restrict__ bu, const T *__restrict__ bv,
                                                 const T *__restrict__ b, const T *__restrict__ idg,
                                                 const T *__restrict__ xp, TO *x, const T *__restrict__ xc,
                                                 int nu2, int H, const int *bsel, const int *xsel)
{
    pdl_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const long long n = (long long)nx * ny;
    b = at_sel(b, bsel, n);
    x = at_sel(x, xsel, n);
    TileView<T> t;
    tile_setup(t, smem_raw, nx, ny, kTX, kTY, H);
    const unsigned mwh = magic_u16(t.ex >> 1);
    tile_load(t, bu, bv, b, idg, xp, xc);
    const int m0 = H - 2 * nu2 + 1;
    for (int q = 0; q < nu2; ++q) {
        tile_pass(t, 0, false, m0 + 2 * q, mwh);
        tile_pass(t, 1, false, m0 + 2 * q + 1, mwh);
    }
    for (int k = threadIdx.x; k < kTX * kTY; k += blockDim.x) {
        int li = H + k % kTX, lj = H + k / kTX, gi = t.gx0 + li, gj = t.gy0 + lj;
        if (gi < nx && gj < ny) x[gj * nx + gi] = TO(t.x[lj * t.ex + li]);
    }
}

template <typename T>
size_t tile_smem(int H, int kTX, int kTY)
{
    const size_t ex = kTX + 2 * H, ey = kTY + 2 * H;
    return sizeof(T) * (3 * ex * ey + (ex + 1) * ey + ex * (ey + 1));
}

}  // namespace
}  // namespace wec
