// The coarse part of a V-cycle in one launch: one thread-block cluster holds
// every level from lb down to the dense level in its shared memory (included by
// solver.cu inside its anonymous namespace; 2D and 3D, FP64 and FP32).
//
// Below some 10^5 cells a level's kernels cost their launch and latency (6 to
// 12 us each) whatever the size.  Here a level is cut into slabs along its slow
// axis (z in 3D, y in 2D), one CTA each, with one halo layer on either side; a
// colour pass updates the CTA's own cells and stores those of its first and last
// layer into the neighbour's halo through distributed shared memory, and waits
// for theirs -- which orders a CTA with its neighbours alone, so the kernel ends in a
// cluster barrier (cl_arrive).  Slabs have an even number of layers, so the children
// of a coarse cell lie in one CTA, which restricts them into the b of the CTA
// that owns the coarse layer; the prolongation reads the coarse iterate from its
// owner.  FP32 levels of at most kClSingle cells run in CTA 0 alone, with block
// barriers; FP64 ones are spread as far as they go (the FP64 pipe does two
// operations per clock and SM).  Bound by the barriers (about 0.5 us each over
// a cluster), shared-memory latency and, since every phase is short, by the
// instructions it takes to start one.
//
// A thread keeps the coefficients, b and 1/d of its own cells -- the two cells
// 2 ih, 2 ih + 1 of a row, one of each colour -- in registers through a level's
// sweeps, so a pass is six (2D: four) loads of neighbours, the multiply-adds, one
// store and a barrier.  The iterate is colour-packed in shared memory (all cells
// of colour 0, then those of colour 1, i / 2 fastest).  Wall faces count as zero
// and layers outside the domain hold x = 0: every cell update is the same terms,
// and a term with a zero factor leaves the sum as it is.  In 3D the terms and
// their order are those of the per-level kernels: the same bits.
constexpr int kClLevels = 14;
constexpr int kClThreads = 512;
constexpr int kClSingle = 2048;  // FP32 cells
constexpr int kClSmem = 225 * 1024;  // dynamic; the plan's copy takes up to 1.4 KB more
template <typename T>
constexpr int cl_pairs = sizeof(T) == 4 ? 4 : 2;  // cell pairs per thread, at most

template <typename T>
struct ClLevel {
    int nx, nm, ns;       // sizes: x, middle (2D: 1), slow axis
    int t, nct;           // layers per CTA, CTAs with layers
    unsigned mh, mm, mcm; // magic_u16 of nx / 2 (also the coarse nx), nm, nm / 2
    int ox, ob, oid, obx, oby, obz;  // shared-memory offsets in elements
    int pk;               // 1/d colour-packed in global memory
    const T *bx, *by, *bz, *id;
};

template <typename T>
struct ClPlan {
    int L, nu1, nu2, C, n;      // levels (the last one dense), sweeps, CTAs of the cluster, cells of the dense level
    int ors, oxl, obl, oinv;    // residuals; dense level's x and b (natural order), this CTA's rows (-1: in global)
    int bpk, opk;               // b read / x written colour-packed in global memory
    int n0;                     // cells of the first level
    int unit;                   // cluster t: b = the unit vector of cell t, x to column t of out (row-major)
    const T *inv;
    ClLevel<T> v[kClLevels];
};

// count elements global -> shared by threads t0, t0 + dt, ...: 16 bytes at a time
// where both sides are aligned
template <typename T>
__device__ __forceinline__ void cl_copy(T *dst, const T *src, int count, int t0, int dt)
{
    constexpr int V = 16 / sizeof(T);
    int done = 0;
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if ((((unsigned)(size_t)src | d) & 15) == 0) {
        const int nv = count / V;
        for (int k = t0; k < nv; k += dt)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16 * k), "l"(src + (long long)k * V)
                         : "memory");
        done = nv * V;
    }
    for (int k = done + t0; k < count; k += dt) cp_async_el(dst + k, src + k);
}

// a thread's cell pair of a level: coefficients, b and 1/d of the cell of each colour
template <typename T, int D>
struct ClPair {
    T f[2][2 * D], b[2], id[2];
    int x;     // shared-memory index of the colour-0 cell's x
    int fl;    // parity of the colour-0 cell's i | lowest layer << 1 | highest << 2 | domain top << 3; -1: no cells
    int c;     // natural index in the CTA's slab of the pair's first cell
};

// Remote halo stores: asynchronous, counted in bytes by the receiving CTA's
// mbarrier, so a pass waits for its two neighbours' layers alone; a cluster
// barrier per pass (whose release fence also waits for every other store) took
// 1.1 thousand cycles where this takes some 0.7.
__device__ __forceinline__ unsigned cl_addr(const void *p, int rank)
{
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
template <typename T>
__device__ __forceinline__ void cl_store_async(unsigned dst, T v, unsigned mbar)
{
    if constexpr (sizeof(T) == 4)
        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst),
                     "r"(__float_as_uint(v)), "r"(mbar)
                     : "memory");
    else
        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst),
                     "l"(__double_as_longlong(v)), "r"(mbar)
                     : "memory");
}
__device__ __forceinline__ void cl_expect(unsigned long long *b, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(b)),
                 "r"(bytes)
                 : "memory");
}
// The two halves of a cluster barrier, for the end of the kernel: a CTA's shared memory
// has to stay until every CTA has made its last access to it.  The halo exchange does
// not order that: it reaches one CTA further per pass, 2 nu2 - 1 in all on the first
// level, where the owner of a coarse layer can be half the cluster away (a slab has two
// layers at least, so a level of two per CTA lies above one on half the CTAs).
// Arriving before the last pass and waiting behind it hides the barrier.
__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cl_depart() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// waits for the phase of the given parity, at most about 0.1 s; false if that runs out
__device__ __forceinline__ bool cl_wait(unsigned long long *b, unsigned parity)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(b);
    for (int it = 0; it < (1 << 22); ++it) {
        unsigned ok;
        asm volatile(
            "{ .reg .pred p; mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// K: cell pairs per thread of the largest slab, at most.  The levels on the way
// down, the dense level and the levels on the way up are one loop, so the code of
// a level is fetched once; the plan is copied to shared memory first (as kernel
// parameters each level's first use was a chain of constant-cache misses).
template <typename T, int D, int K, typename OT>
__global__ void __launch_bounds__(kClThreads, 1)
    k_mg_cluster(const __grid_constant__ ClPlan<T> MP, const T *__restrict__ bg, const int *bsel, OT *out,
                 const int *osel)
{
    extern __shared__ __align__(16) unsigned char cl_smem[];
    __shared__ ClPlan<T> M;
    __shared__ __align__(8) unsigned long long hbar[2];  // halo layers from the CTA below, above
    __shared__ int bad;                                  // a wait ran out: the result is NaN
    const int tid = threadIdx.x, nt = blockDim.x;
    {
        const int words = (int)((offsetof(ClPlan<T>, v) + (size_t)(MP.L - 1) * sizeof(ClLevel<T>)) / 4);
        for (int w = tid; w < words; w += nt)
            reinterpret_cast<unsigned *>(&M)[w] = reinterpret_cast<const unsigned *>(&MP)[w];
    }
    if (tid == 0) {
        for (int s = 0; s < 2; ++s)
            asm volatile("mbarrier.init.shared.b64 [%0], 1;" ::"r"((unsigned)__cvta_generic_to_shared(hbar + s)) : "memory");
        bad = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    pdl_entry();
    __syncthreads();
    T *const sm = reinterpret_cast<T *>(cl_smem);
    cg::cluster_group cl = cg::this_cluster();
    const int C = M.C, rank = C > 1 ? (int)cl.block_rank() : 0, last = M.L - 1, nu1 = M.nu1, nu2 = M.nu2;
    auto remote = [&](T *p, int r) { return C > 1 ? cl.map_shared_rank(p, r) : p; };
    auto layers = [&](const ClLevel<T> &v) { return max(0, min(v.t, v.ns - rank * v.t)); };
    auto bar = [&](bool wide) {
        if (wide) cl.sync(); else __syncthreads();
    };
    const int rows = (M.n + C - 1) / C;  // rows of the dense level per CTA
    // A pass's halo layers are expected (armed) before this CTA's stores of that
    // pass, so a neighbour cannot be a pass further when they are: it needs those.
    auto arm = [&](const ClLevel<T> &v) {
        const unsigned bytes = (unsigned)sizeof(T) * ((v.nx * v.nm) >> 1);
        const int k0 = rank * v.t;
        if (tid != 0 || v.nct == 1 || k0 >= v.ns || bad) return;  // (no second arrival in an incomplete phase)
        if (rank > 0) cl_expect(hbar, bytes);
        if (k0 + v.t < v.ns) cl_expect(hbar + 1, bytes);
    };
    unsigned par0 = 0, par1 = 0;  // (warp 0)

    // ---- stage: b and the coefficients of the first level by all threads, array
    // by array; the other levels a warp per array, and this CTA's rows of the
    // dense level's matrix, in flight while the first level is smoothed
    auto packed = [&](int o, const T *src, const ClLevel<T> &v, int tl, int pk, int t0, int dt) {
        const int pl = (v.nx * v.nm) >> 1, k0 = rank * v.t;
        if (!pk) {
            cl_copy(sm + o, src + (size_t)k0 * 2 * pl, tl * 2 * pl, t0, dt);
        } else {
            cl_copy(sm + o, src + (size_t)k0 * pl, tl * pl, t0, dt);
            cl_copy(sm + o + v.t * pl, src + (size_t)(v.ns + k0) * pl, tl * pl, t0, dt);
        }
    };
    auto stage = [&](const ClLevel<T> &v, int a, int t0, int dt) {
        const int tl = layers(v), lay = v.nx * v.nm, k0 = rank * v.t;
        if (tl == 0) return;
        if (a == 2) {
            packed(v.oid, v.id, v, tl, v.pk, t0, dt);
        } else {
            // (a: 0 beta_x, 1 beta_z, 3 beta_y)
            const T *src = a == 0 ? v.bx : a == 1 ? v.bz : v.by;
            const int per = a == 0 ? v.nm * (v.nx + 1) : a == 1 ? lay : (v.nm + 1) * v.nx;
            cl_copy(sm + (a == 0 ? v.obx : a == 1 ? v.obz : v.oby), src + (size_t)k0 * per, (tl + (a == 1 ? 1 : 0)) * per,
                    t0, dt);
        }
    };
    constexpr int NA = D == 3 ? 4 : 3;
    if (last > 0) {
        const ClLevel<T> &v = M.v[0];
        for (int a = 0; a < NA; ++a) stage(v, a, tid, nt);
        if (!M.unit && layers(v) > 0)
            packed(v.ob, at_sel(bg, bsel, (long long)v.nx * v.nm * v.ns), v, layers(v), M.bpk, tid, nt);
    } else {  // (every CTA its own copy)
        cl_copy(sm + M.obl, at_sel(bg, bsel, M.n), M.n, tid, nt);
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    for (int w = tid >> 5; w < (last - 1) * NA; w += nt >> 5) stage(M.v[1 + w / NA], w % NA, tid & 31, 32);
    if (M.oinv >= 0 && rank * rows < M.n)
        cl_copy(sm + M.oinv, M.inv + (size_t)rank * rows * M.n, min(rows, M.n - rank * rows) * M.n, tid, nt);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    // the halo layers of every level: zero
    for (int q = 0; q < last; ++q) {
        const ClLevel<T> &v = M.v[q];
        const int pl = (v.nx * v.nm) >> 1, tl = layers(v);
        for (int e = tid; e < pl; e += nt) {
            T *x = sm + v.ox + e;
            x[0] = x[(tl + 1) * pl] = x[(v.t + 2) * pl] = x[(v.t + tl + 3) * pl] = T(0);
        }
        if (M.unit && q == 0)
            for (int e = tid; e < 2 * pl * v.ns; e += nt) sm[v.ob + e] = e == (int)blockIdx.x ? T(1) : T(0);
    }
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    if (last > 0) arm(M.v[0]);
    bar(C > 1);

    ClPair<T, D> m[K];
    OT *const o = at_sel(out, osel, (long long)M.n0);
    for (int ph = 0; ph <= 2 * last; ++ph) {
        if (ph == 1 || last == 0) {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
            __syncthreads();
        }
        if (ph == last) {  // ---- the dense level: its matrix times b, the rows over the cluster's CTAs
            const int n = M.n, lane = tid & 31, r0 = rank * rows, r1 = min(n, r0 + rows);
            if (C > 1 && last > 0 && M.v[last - 1].nct == 1) cl.sync();  // (b from a level CTA 0 ran alone)
            const T *const inv = M.oinv >= 0 ? sm + M.oinv : M.inv + (size_t)r0 * n;
            for (int r = r0 + (tid >> 5); r < r1; r += nt >> 5) {
                const T s = inv_row(inv + (r - r0) * n, sm + M.obl, n, lane);
                if (lane < C) *remote(sm + M.oxl + r, lane) = s;  // x to every CTA
            }
            bar(C > 1);
            continue;
        }
        const bool down = ph < last;
        const int q = down ? ph : 2 * last - ph;
        const ClLevel<T> &v = M.v[q], &w = M.v[q + 1];
        // (the owners' coarse iterates; a dense one is everywhere)
        if (!down && v.nct > 1 && q + 1 < last) cl.sync();
        if (v.nct == 1 && rank > 0) continue;
        const int nx = v.nx, nm = v.nm, ns = v.ns, vt = v.t, half = nx >> 1, pl = nm * half, lay = 2 * pl;
        const int tl = layers(v), nh = tl * pl, k0 = rank * vt, cm = D == 3 ? nm >> 1 : 1, blk = (vt + 2) * pl, ox = v.ox;
        const bool wide = v.nct > 1;
        // the coarse iterate above cell (2 ih or 2 ih + 1, j, kk)
        const bool cdense = q + 1 == last;
        const int wt = cdense ? 0 : w.t, wn = cdense ? 1 : w.nct, wo = cdense ? M.oxl : w.ox;
        auto coarse = [&](int ih, int j, int kk) -> const T * {
            const int Kc = (k0 + kk) >> 1, J = j >> 1;
            if (cdense) return sm + wo + (Kc * cm + J) * half + ih;
            const int owner = wn > 1 ? Kc / wt : 0, kw = Kc - owner * wt;
            return remote(sm + wo + ((((ih + J + kw) & 1) * (wt + 2) + kw + 1) * cm + J) * (half >> 1) + (ih >> 1), owner);
        };
        if (!down && wide && nu2 > 0 && tl > 0) {
            // the correction of the halo layers' black cells (all a red pass reads)
            for (int e = tid; e < 2 * pl; e += nt) {
                const bool lo = e < pl;
                const int h = lo ? e : e - pl, kk = lo ? -1 : tl;
                if (lo ? k0 == 0 : k0 + tl >= ns) continue;
                const int j = div_u16(h, v.mh), ih = h - j * half;
                sm[ox + blk + (kk + 1) * pl + h] += *coarse(ih, j, kk);
            }
        }
        // ---- this thread's pairs: coefficients and b into registers
#pragma unroll
        for (int u = 0; u < K; ++u) {
            const int e = tid + u * nt;
            m[u].fl = -1;
            if (e >= nh) break;
            const int r = div_u16(e, v.mh), ih = e - r * half, kk = D == 3 ? div_u16(r, v.mm) : r;
            const int j = D == 3 ? r - kk * nm : 0, c = 2 * e, p = (j + kk) & 1;
            m[u].x = ox + pl + e;
            if (!down) {
                // += the coarse correction: the black cell (the red pass that follows
                // reads nothing else), or both where no sweep follows
                const T cc = *coarse(ih, j, kk);
                sm[m[u].x + blk] += cc;
                if (nu2 == 0) sm[m[u].x] += cc;
            }
            const T *fx = sm + v.obx + c + r, *fz = sm + v.obz + c, *fy = sm + v.oby + c + kk * nx;
            const T x0 = ih > 0 ? fx[0] : T(0), x1 = fx[1], x2 = ih < half - 1 ? fx[2] : T(0);
            const bool bp = q > 0 || M.bpk;
#pragma unroll
            for (int col = 0; col < 2; ++col) {
                const int od = p ^ col;  // the colour's cell: i = 2 ih + od
                T *f = m[u].f[col];
                f[0] = od ? x1 : x0;
                f[1] = od ? x2 : x1;
                if (D == 3) {
                    f[2] = j > 0 ? fy[od] : T(0);
                    f[3] = j < nm - 1 ? fy[nx + od] : T(0);
                }
                f[2 * D - 2] = k0 + kk > 0 ? fz[od] : T(0);
                f[2 * D - 1] = fz[lay + od];
                m[u].id[col] = sm[v.oid + (v.pk ? col * vt * pl + e : c + od)];
                m[u].b[col] = sm[v.ob + (bp ? col * vt * pl + e : c + od)];
            }
            m[u].fl = p | (wide && kk == 0 && k0 > 0 ? 2 : 0) | (wide && kk == tl - 1 && k0 + tl < ns ? 4 : 0) |
                      (k0 + kk == ns - 1 ? 8 : 0);
            m[u].c = c;
        }
        if (!down) {
            if (nu2 > 0) arm(v);
            bar(nu2 == 0 && wide);
        }
        // sum_f beta_f x_nb of a pair's cell of colour col
        auto offsum = [&](const ClPair<T, D> &a, int col) {
            const T *x = sm + a.x + (col ? 0 : blk);
            const int odd = (a.fl ^ col) & 1;
            const T *f = a.f[col];
            T s = T(0);
            s = fma3(f[0], x[odd - 1], s);
            s = fma3(f[1], x[odd], s);
            if (D == 3) {
                s = fma3(f[2], x[-half], s);
                s = fma3(f[3], x[half], s);
            }
            s = fma3(f[2 * D - 2], x[-pl], s);
            return fma3(f[2 * D - 1], x[pl], s);
        };
        // ---- the sweeps; a pass ends with the arrival of the neighbours' layers and
        // a barrier (the last one of all is only read by its own thread)
        const int nu = down ? nu1 : nu2;
        const bool lo = wide && tl > 0 && k0 > 0, hi = wide && tl > 0 && k0 + tl < ns;
        for (int s = 0; s < nu; ++s) {
#pragma unroll
            for (int col = 0; col < 2; ++col) {
                const bool fin = !down && q == 0 && s == nu - 1 && col == 1;
                if (fin && C > 1) cl_arrive();  // (no access to another CTA follows)
#pragma unroll
                for (int u = 0; u < K; ++u) {
                    if (m[u].fl < 0) break;
                    T a = T(0);  // (the first red pass: from x = 0)
                    if (col || s || !down) a = offsum(m[u], col);
                    const T val = (m[u].b[col] + a) * m[u].id[col];
                    T *const x = sm + m[u].x + col * blk;
                    *x = val;
                    // the neighbours' halo: their layer t + 1 / 0
                    if (!fin) {
                        if (m[u].fl & 2) cl_store_async(cl_addr(x + vt * pl, rank - 1), val, cl_addr(hbar + 1, rank - 1));
                        if (m[u].fl & 4) cl_store_async(cl_addr(x - vt * pl, rank + 1), val, cl_addr(hbar, rank + 1));
                    }
                }
                if (fin) continue;
                if (wide && tid < 32) {
                    bool ok = true;
                    if (lo && !bad) ok = cl_wait(hbar, par0);
                    if (hi && !bad && ok) ok = cl_wait(hbar + 1, par1);
                    if (!ok) bad = 1;
                    par0 ^= lo ? 1u : 0u;
                    par1 ^= hi ? 1u : 0u;
                    // the next pass of this level, if it exchanges layers
                    const bool more = col == 0 || s + 1 < nu, nfin = !down && q == 0 && s == nu - 1;
                    if (more && !nfin) arm(v);
                }
                __syncthreads();
            }
        }
        if (down) {
            // the residuals of this CTA's cells, then the sums over the children into
            // the coarse b at its owner (a dense one: at every CTA)
#pragma unroll
            for (int u = 0; u < K; ++u) {
                if (m[u].fl < 0) break;
#pragma unroll
                for (int col = 0; col < 2; ++col) {
                    T d = T(0);
#pragma unroll
                    for (int a = 0; a + 1 < 2 * D; ++a) d += m[u].f[col][a];
                    d += (m[u].fl & 8 ? T(2) : T(1)) * m[u].f[col][2 * D - 1];
                    const T ax = fma3(d, sm[m[u].x + col * blk], -offsum(m[u], col));
                    sm[M.ors + m[u].c + ((m[u].fl ^ col) & 1)] = m[u].b[col] - ax;
                }
            }
            __syncthreads();
            const int nc = (tl >> 1) * cm * half, K0 = k0 >> 1;
            for (int e = tid; e < nc; e += nt) {
                const int R = div_u16(e, v.mh), I = e - R * half, kc = D == 3 ? div_u16(R, v.mcm) : R, J = R - kc * cm;
                const T *rs = sm + M.ors + (2 * kc * nm + 2 * (D == 3 ? J : 0)) * nx + 2 * I;
                T s = T(0);
#pragma unroll
                for (int dk = 0; dk < 2; ++dk)
#pragma unroll
                    for (int dj = 0; dj < (D == 3 ? 2 : 1); ++dj) {
                        s += rs[(dk * nm + dj) * nx];
                        s += rs[(dk * nm + dj) * nx + 1];
                    }
                const int Kc = K0 + kc;  // the coarse layer
                if (cdense) {
                    for (int r = 0; r < C; ++r) *remote(sm + M.obl + (Kc * cm + J) * half + I, r) = s;
                } else {
                    const int owner = wn > 1 ? Kc / wt : 0, kw = Kc - owner * wt;
                    *remote(sm + w.ob + ((((I + J + kw) & 1) * wt + kw) * cm + J) * (half >> 1) + (I >> 1), owner) = s;
                }
            }
            if (!cdense) arm(w);
            bar(wide);
        } else if (q == 0) {
            // ---- x of the first level: a thread's own pairs
#pragma unroll
            for (int u = 0; u < K; ++u) {
                if (m[u].fl < 0) break;
                const int e = m[u].c >> 1;
#pragma unroll
                for (int col = 0; col < 2; ++col) {
                    const OT val = bad ? OT(NAN) : widen_out<OT>(sm[m[u].x + col * blk]);
                    const int c = m[u].c + ((m[u].fl ^ col) & 1);
                    if (M.opk)
                        o[(size_t)(col * ns + k0) * pl + e] = val;
                    else if (M.unit)
                        o[(size_t)c * M.n0 + blockIdx.x] = val;
                    else
                        o[(size_t)k0 * lay + c] = val;
                }
            }
        }
    }
    if (last == 0 && rank == 0)
        for (int c = tid; c < M.n; c += nt) o[c] = widen_out<OT>(sm[M.oxl + c]);
    if (C > 1) {
        const bool last_pass = last > 0 && nu2 > 0 && (M.v[0].nct > 1 || rank == 0);
        if (!last_pass) cl_arrive();
        cl_depart();
        // after an expired wait: the layers still on their way to this CTA (every
        // CTA has sent its last one; the others have waited for theirs)
        if (bad)
            for (int it = 0; it < 100; ++it) __nanosleep(1000);
    }
}

int g_cluster_max = 8;  // CTAs per cluster this GPU takes (16 where the occupancy query allows it)

// The plan of levels lb..end (end dense) over C CTAs: offsets and sizes; its shared memory in bytes.
template <typename T>
size_t cluster_plan(const wec_poisson *P, const Level<T> *L, int lb, int end, int C, ClPlan<T> &M)
{
    const bool d3 = P->nz > 1;
    M = ClPlan<T>();
    M.L = end - lb + 1;
    M.nu1 = P->nu1;
    M.nu2 = P->nu2;
    M.C = C;
    M.n = L[end].nx * L[end].ny * L[end].nz;
    M.n0 = L[lb].nx * L[lb].ny * L[lb].nz;
    M.inv = end == P->nlev - 1 ? coarse_inv<T>(P) : dense_mat<T>(P);
    size_t o = 0, rs = 0;
    auto take = [&o](size_t n) {
        const size_t r = o;
        o += (n + 3) & ~size_t(3);
        return (int)r;
    };
    for (int q = 0; q + 1 < M.L; ++q) {
        const Level<T> &A = L[lb + q];
        ClLevel<T> &v = M.v[q];
        v.nx = A.nx;
        v.nm = d3 ? A.ny : 1;
        v.ns = d3 ? A.nz : A.ny;
        const size_t lay = (size_t)v.nx * v.nm, cells = lay * v.ns;
        if (C == 1 || (sizeof(T) == 4 && cells <= kClSingle)) {
            v.t = v.ns;
        } else {
            v.t = (v.ns + C - 1) / C;
            v.t += v.t & 1;
        }
        v.nct = (v.ns + v.t - 1) / v.t;
        // (2D tile kernels beat more than two pairs per thread)
        if (v.t * lay > 2ull * kClThreads * std::min(cl_pairs<T>, d3 ? 4 : 2)) return kClSmem + 1;
        v.mh = magic_u16(v.nx >> 1);
        v.mm = magic_u16(std::max(2, v.nm));
        v.mcm = magic_u16(std::max(2, v.nm >> 1));
        v.bx = A.bu;
        v.by = d3 ? A.bv : nullptr;
        v.bz = d3 ? A.bw : A.bv;
        v.id = A.id;
        v.pk = d3 && sizeof(T) == 4 && lb + q < P->dense ? 1 : 0;
        v.ox = take((v.t + 2) * lay);
        v.ob = take(v.t * lay);
        rs = std::max(rs, v.t * lay);
        v.oid = take(v.t * lay);
        v.obx = take((size_t)v.t * v.nm * (v.nx + 1));
        v.oby = d3 ? take((size_t)v.t * (v.nm + 1) * v.nx) : 0;
        v.obz = take((v.t + 1) * lay);
    }
    M.ors = take(rs);
    M.oxl = take(M.n);
    M.obl = take(M.n);
    M.oinv = -1;
    const size_t rows = (size_t)(M.n + C - 1) / C * M.n;
    if ((o + rows) * sizeof(T) <= (size_t)kClSmem) M.oinv = take(rows);
    return o * sizeof(T);
}

// First level of the cluster kernel (the finest that fits; shift: that many
// levels further down), and the plan.  CTAs: enough for a pair of cells per
// thread (FP64: for a quarter of that) and for 64 rows of the dense level each,
// or as many as there are.
template <typename T>
int cluster_first(const wec_poisson *P, const Level<T> *L, int shift, ClPlan<T> &M, size_t &smem)
{
    auto plan = [&](int lb) {
        const long long cells = (long long)L[lb].nx * L[lb].ny * L[lb].nz;
        const long long nd = (long long)L[P->dense].nx * L[P->dense].ny * L[P->dense].nz;
        int C = 1;
        while (C < g_cluster_max && (cells > (sizeof(T) == 4 ? 2ll : 1ll) * kClThreads / (sizeof(T) == 4 ? 1 : 2) * C ||
                                     nd > 64 * C))
            C *= 2;
        do smem = cluster_plan(P, L, lb, P->dense, C, M); while (smem > kClSmem && (C *= 2) <= g_cluster_max);
        return smem <= kClSmem;
    };
    int lb = 0;
    while (lb < P->dense && (P->dense - lb >= kClLevels || !plan(lb))) ++lb;
    lb = std::min(lb + shift, P->dense);
    plan(lb);  // (the dense level alone always fits)
    return lb;
}

// algorithmic bytes: b and x of level lb, every level's coefficients, the dense level's matrix
template <typename T>
double cluster_bytes(const wec_poisson *P, const Level<T> *L, int lb)
{
    const Level<T> &A = L[P->dense];
    const double n = (double)A.nx * A.ny * A.nz;
    double e = n * n + 2.0 * L[lb].nx * L[lb].ny * L[lb].nz;
    for (int l = lb; l < P->dense; ++l) e += (P->nz > 1 ? 4.0 : 3.0) * L[l].nx * L[l].ny * L[l].nz;
    return e * sizeof(T);
}

template <typename T, int D, typename OT>
void launch_cluster(const ClPlan<T> &M, size_t smem, int nclusters, const T *b, const int *bsel, OT *out, const int *osel,
                    cudaStream_t st)
{
    int pairs = M.C > 1 ? kClThreads : 64;  // (the dense level's rows want warps)
    for (int q = 0; q + 1 < M.L; ++q) pairs = std::max(pairs, M.v[q].nx * M.v[q].nm * M.v[q].t / 2);
    prof::count_launch();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(M.C * nclusters);
    cfg.blockDim = dim3(std::min(kClThreads, (pairs + 31) / 32 * 32));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = M.C;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    auto kern = pairs <= kClThreads     ? k_mg_cluster<T, D, 1, OT>
                : pairs <= 2 * kClThreads ? k_mg_cluster<T, D, 2, OT>
                                          : k_mg_cluster<T, D, cl_pairs<T>, OT>;
    cudaLaunchKernelEx(&cfg, kern, M, b, bsel, out, osel);
}

// The dense level's matrix: the V-cycle of the levels from P->dense down, one
// unit vector per CTA.  That part of a V-cycle is a fixed linear map per
// coefficient set, and its levels of at most kDense cells cost some 4 us each in
// barriers and phase starts however few their cells are: applied as a matrix
// they cost one pass over 512 x 512 values.
template <typename T, int D>
void launch_dense(const wec_poisson *P, const Level<T> *L, cudaStream_t st)
{
    if (P->dense == P->nlev - 1) return;  // (the coarsest level: its inverse)
    ClPlan<T> M;
    const size_t smem = cluster_plan(P, L, P->dense, P->nlev - 1, 1, M);
    M.unit = 1;
    const Level<T> &A = L[P->dense];
    launch_cluster<T, D, T>(M, smem, A.nx * A.ny * A.nz, nullptr, nullptr, dense_mat<T>(P), nullptr, st);
}

template <typename T, int D, int K, typename OT>
int cluster_attrs_k(int *cmax)
{
    auto kern = k_mg_cluster<T, D, K, OT>;
    WEC_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kClSmem));
    WEC_CK(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(16);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = kClSmem;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int c = 0;
    if (cudaOccupancyMaxActiveClusters(&c, (void *)kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        c = 0;
    }
    if (c < 1) *cmax = 8;
    return WEC_OK;
}

template <typename T, int D, typename OT>
int cluster_attrs_one(int *cmax)
{
    if (int e = cluster_attrs_k<T, D, 1, OT>(cmax)) return e;
    if (int e = cluster_attrs_k<T, D, 2, OT>(cmax)) return e;
    return cluster_attrs_k<T, D, cl_pairs<T>, OT>(cmax);
}

int set_cluster_attrs()
{
    int c = 16;
    int e = cluster_attrs_one<double, 2, double>(&c);
    if (!e) e = cluster_attrs_one<float, 2, float>(&c);
    if (!e) e = cluster_attrs_one<float, 2, double>(&c);
    if (!e) e = cluster_attrs_one<double, 3, double>(&c);
    if (!e) e = cluster_attrs_one<float, 3, float>(&c);
    if (!e) e = cluster_attrs_one<float, 3, double>(&c);
    g_cluster_max = c;
    return e;
}
