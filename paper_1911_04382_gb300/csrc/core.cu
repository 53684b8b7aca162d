// core.cu -- the inner CG of a sparsifier with few added edges on its core.
//
// S is the tree and k added edges.  Everything but the ends of the added
// edges, the vertices between units (units.cuh) and the branching vertices
// between them can be eliminated from S exactly, unit by unit; what remains
// is the core: a tree of about n / 10 vertices and the k added edges.  CG on
// S preconditioned by the tree T is invariant under that elimination: with
// F the unit lower triangular factor, F^T S F = diag(T11, S') and F^T T F =
// diag(T11, T'), and the residual in the eliminated part stays a multiple of
// the right-hand side there (b1), so that part of every vector is one number
// per column:
//
//   r1 = c b1,  z1 = c T11^{-1} b1,  p1 = g T11^{-1} b1,  q1 = g b1,
//   b1' T11^{-1} b1 = e1,  |r|^2 = |r' + c d|^2 + c^2 |b1|^2
//
// (d: the core's original less its eliminated right-hand side).  The same
// iterates, step lengths and stop test as the CG over all n vertices, in
// vectors of a tenth of the length: one pass eliminates, the iterations run
// on the core, one pass substitutes back.  One power step with 30
// iterations of 16 FP32 columns on the 100^3 grid with 16,400 added edges:
// 15.2 ms over all vertices, 2.6 ms here (FP64: 29.5 and 4.3 ms); a
// 300,007-vertex power-law graph, 24 FP32 columns: 26.5 and 4.1 ms.  The
// core's vectors stay in L2; what is left is the grid barriers of about eight
// phases an iteration.
#include "cg.cuh"

namespace grass {

// ---------------------------------------------------------------- structure

namespace {

__global__ void k_co_flag(int64_t m, const uint8_t *in_s, const uint8_t *in_tree, int64_t *flag) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < m) flag[e] = in_s[e] && !in_tree[e];
}

// ends of the added edges as positions, marked as vertices that must survive
__global__ void k_co_extra(int64_t m, const uint8_t *in_s, const uint8_t *in_tree, const int64_t *at,
                           const int32_t *eu, const int32_t *ev, const double *ew,
                           const int32_t *pos, int32_t *xu, int32_t *xv, double *xw, uint8_t *pin) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m || !in_s[e] || in_tree[e]) return;
    const int64_t k = at[e];
    xu[k] = pos[eu[e]];
    xv[k] = pos[ev[e]];
    xw[k] = ew[e];
    pin[xu[k]] = 1;
    pin[xv[k]] = 1;
}

__global__ void k_co_vert(int64_t n, int B, const int4 *meta, const int32_t *lidx,
                          const int32_t *ord, const int32_t *core, int32_t *vert) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    if ((int)(q % B) >= meta[q / B].x) vert[core[lidx[q]]] = ord[q];
}

// core edge e: e < n1 the tree edge of core vertex e (none for the root),
// else an added edge
__device__ inline bool co_edge(int64_t e, int64_t n1, const int32_t *parent, const int32_t *xu,
                               const int32_t *xv, const int32_t *core, int32_t *a, int32_t *b) {
    if (e < n1) {
        *a = (int32_t)e;
        *b = parent[e];
        return *b >= 0;
    }
    *a = core[xu[e - n1]];
    *b = core[xv[e - n1]];
    return true;
}

__global__ void k_co_count(int64_t ne, int64_t n1, const int32_t *parent, const int32_t *xu,
                           const int32_t *xv, const int32_t *core, unsigned long long *deg) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int32_t a, b;
    if (e >= ne || !co_edge(e, n1, parent, xu, xv, core, &a, &b)) return;
    atomicAdd(deg + a, 1ull);
    atomicAdd(deg + b, 1ull);
}

__global__ void k_co_ptr(int64_t n1, const int64_t *off, int32_t *ptr, int32_t *cur) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i > n1) return;
    ptr[i] = (int32_t)off[i];
    if (i < n1) cur[i] = (int32_t)off[i];
}

__global__ void k_co_fill(int64_t ne, int64_t n1, const int32_t *parent, const int32_t *xu,
                          const int32_t *xv, const int32_t *core, int32_t *cur, int32_t *raw,
                          int32_t *row) {
    int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int32_t a, b;
    if (e >= ne || !co_edge(e, n1, parent, xu, xv, core, &a, &b)) return;
    int32_t j = atomicAdd(cur + a, 1);
    raw[j] = (int32_t)e;
    row[j] = a;
    j = atomicAdd(cur + b, 1);
    raw[j] = (int32_t)e;
    row[j] = b;
}

// every row in edge order; columns and weights
__global__ void k_co_sort(int64_t nnz, int64_t n1, const int32_t *parent, const double *w,
                          const int32_t *xu, const int32_t *xv, const double *xw,
                          const int32_t *core, const int32_t *ptr, const int32_t *raw,
                          const int32_t *row, int32_t *col, double *w64, float *w32) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nnz) return;
    const int32_t e = raw[k], r = row[k];
    int rank = 0;
    for (int32_t j = ptr[r]; j < ptr[r + 1]; ++j) rank += raw[j] < e;
    int32_t a, b;
    co_edge(e, n1, parent, xu, xv, core, &a, &b);
    const int32_t q = ptr[r] + rank;
    const double x = e < n1 ? w[e] : xw[e - n1];
    col[q] = r == a ? b : a;
    w64[q] = x;
    w32[q] = (float)x;
}

}  // namespace

// Rule: at least 2,048 vertices and 16 of them per added edge.  The core has
// about two branching vertices per end of an added edge at most, so it is
// then below n / 4 and its build (about 1 ms at a million vertices, every
// change of S) is a fraction of one solve.
// And the iterations a caller allows on S have to pay the build, which its
// first solve waits for: 160 of them in FP32 and 64 in FP64, or fewer where a
// block is large (their number times the block's bytes 256 MB, in FP64 128 MB).
// Measured, us: an iteration over all vertices / on the core, the build with
// n / 17 added edges, the iterations that pay it (with n / 200 added edges):
//   90,000 vertices  2 FP32 columns (0.7 MB)  49 / 45   565  147 (40)
//                   16 FP32 (5.8 MB)          76 / 65   590   55 (25)
//                    2 FP64 (1.4 MB)          65 / 55   586   59 (23)
//                   16 FP64 (11.5 MB)        122 / 66   556   11 (7)
//   250,000         16 FP32 (16 MB)          111 / 73   598   17 (11)
//                    4 FP64 (8 MB)           102 / 65   636   18 (11)
//   1M               2 FP32 (8 MB)           104 / 56   962   21 (13)
//                   16 FP32 (64 MB)          337 / 101  960    4 (3)
//                    2 FP64 (16 MB)          198 / 77   966    9 (6)
//                   16 FP64 (128 MB)         955 / 223  974    2 (1)
// The rule looks at the call alone: a sparsifier solved again and again by the
// same short call gets the same form, and the same bits, every time.
static bool core_wanted(const grass_sparsifier_s *S, int r, grass_prec prec, int64_t its) {
    const grass_tree_s *T = S->tree;
    const int64_t n = T->g.n, added = S->n_edges - (n - 1);
    const bool f64 = prec == GRASS_FP64;
    return T->units.built && n >= 2048 && added > 0 && 16 * added <= n &&
           (its >= (f64 ? 64 : 160) ||
            (double)its * (double)n * r * (f64 ? 8.0 : 4.0) >= (f64 ? 128e6 : 256e6));
}

// False: S keeps the CG over all vertices.
static bool core_form(grass_ctx_t ctx, grass_sparsifier_t S, CoreForm &C) {
    grass_tree_t T = S->tree;
    const GraphData &g = T->g;
    const int64_t n = g.n, m = g.m, k = S->n_edges - (n - 1);
    Arena &tmp = ctx->core_tmp;
    tmp.reset();
    tmp.chunk_min = (size_t)n * 36 + ((size_t)1 << 20);
    auto *flag = ctx->scr<int64_t>(SCR_TMP0, m + 1);
    auto *at = ctx->scr<int64_t>(SCR_TMP1, m + 1);
    auto *xu = tmp.get<int32_t>(k), *xv = tmp.get<int32_t>(k);
    auto *xw = tmp.get<double>(k);
    auto *pin = tmp.get<uint8_t>(n);
    auto *parent = tmp.get<int32_t>(n), *core = tmp.get<int32_t>(n);
    memset_d(ctx, pin, 0, n);
    launch(ctx, k_co_flag, cdiv(m, kBlock), kBlock, 0, m, (const uint8_t *)S->in_s.p,
           (const uint8_t *)T->in_tree.p, flag);
    scan_i64(ctx, flag, at, m, nullptr);
    launch(ctx, k_co_extra, cdiv(m, kBlock), kBlock, 0, m, (const uint8_t *)S->in_s.p,
           (const uint8_t *)T->in_tree.p, (const int64_t *)at, (const int32_t *)g.eu.p,
           (const int32_t *)g.ev.p, (const double *)g.ew64.p, (const int32_t *)T->units.pos, xu, xv,
           xw, pin);
    copy_d(ctx, parent, T->units.parent, n * sizeof(int32_t));
    C.low.arena.chunk_min = (size_t)n * 32 + ((size_t)1 << 20);
    int32_t *scnt = nullptr;
    int64_t n1 = 0;
    if (!unit_levels(ctx, n, parent, T->units.vid, pin, tmp, C.low, core, &scnt, &n1) ||
        4 * n1 > n || n1 < 2)
        return false;
    C.n = n1;
    C.nnz = 2 * (n1 - 1 + k);
    C.arena.chunk_min = (size_t)n1 * 56 + (size_t)k * 32 + ((size_t)1 << 19);
    UnitLevel &L = C.low.lv[0];
    L.sptr = C.arena.get<int32_t>(n1 + 1);
    unit_group(ctx, C.low, L, n1, nullptr, scnt, tmp, L.sptr);
    C.vert = C.arena.get<int32_t>(n1);
    launch(ctx, k_co_vert, cdiv(n, kBlock), kBlock, 0, n, L.B, (const int4 *)L.meta,
           (const int32_t *)L.lidx, (const int32_t *)L.ord, (const int32_t *)core, C.vert);
    C.tree.w0 = C.arena.get<double>(n1);
    C.low.w0 = T->units.w0;
    unit_factor(ctx, C.low, nullptr, C.low_f, C.tree.w0);
    // the core's adjacency
    const int64_t ne = n1 + k;
    auto *deg = tmp.get<unsigned long long>(n1 + 1);
    auto *off = tmp.get<int64_t>(n1 + 1);
    auto *cur = tmp.get<int32_t>(n1);
    auto *raw = tmp.get<int32_t>(C.nnz), *row = tmp.get<int32_t>(C.nnz);
    C.ptr = C.arena.get<int32_t>(n1 + 1);
    C.col = C.arena.get<int32_t>(C.nnz);
    C.w64 = C.arena.get<double>(C.nnz);
    C.w32 = C.arena.get<float>(C.nnz);
    memset_d(ctx, deg, 0, (n1 + 1) * sizeof(unsigned long long));
    launch(ctx, k_co_count, cdiv(ne, kBlock), kBlock, 0, ne, n1, (const int32_t *)parent,
           (const int32_t *)xu, (const int32_t *)xv, (const int32_t *)core, deg);
    scan_i64(ctx, (const int64_t *)deg, off, n1, nullptr);
    launch(ctx, k_co_ptr, cdiv(n1 + 1, kBlock), kBlock, 0, n1, (const int64_t *)off, C.ptr, cur);
    launch(ctx, k_co_fill, cdiv(ne, kBlock), kBlock, 0, ne, n1, (const int32_t *)parent,
           (const int32_t *)xu, (const int32_t *)xv, (const int32_t *)core, cur, raw, row);
    launch(ctx, k_co_sort, cdiv(C.nnz, kBlock), kBlock, 0, C.nnz, n1, (const int32_t *)parent,
           (const double *)C.tree.w0, (const int32_t *)xu, (const int32_t *)xv, (const double *)xw,
           (const int32_t *)core, (const int32_t *)C.ptr, (const int32_t *)raw, (const int32_t *)row,
           C.col, C.w64, C.w32);
    // the core's own tree, in the same order of its vertices (a preorder)
    C.tree.arena.chunk_min = (size_t)n1 * 64 + ((size_t)1 << 19);
    auto *core2 = tmp.get<int32_t>(n1);
    int32_t *scnt2 = nullptr;
    int64_t n2 = 0;
    if (!unit_levels(ctx, n1, parent, nullptr, nullptr, tmp, C.tree, core2, &scnt2, &n2))
        return false;
    unit_factor(ctx, C.tree, nullptr, C.tree_f);
    return true;
}

// S->core, once per change of S.  It is in place only when it is complete; a
// tree that is not suited, or no room for the form, leaves an empty one (the
// CG over all vertices needs none of its arrays), any other error none.
static bool core_build(grass_ctx_t ctx, grass_sparsifier_t S) {
    if (S->core) return S->core->usable;
    auto C = std::make_unique<CoreForm>();
    try {
        C->usable = core_form(ctx, S, *C);
    } catch (const Error &e) {
        ctx->core_tmp = Arena();
        if (e.st != GRASS_ERR_OOM) throw;
    }
    if (!C->usable) C = std::make_unique<CoreForm>();
    trim(ctx->core_tmp);
    S->core = std::move(C);
    return S->core->usable;
}


// ---------------------------------------------------------------- solve

template <typename T>
struct CoreKArgs {
    UnitArgs<T> low;      // level 0 alone; epos / edst by core index
    const T *Y;           // [vertices x R] right-hand side
    T *X;                 // [vertices x R] solution
    T *F;                 // [n x R] eliminated right-hand sides in unit order
    T *dv;                // [core x R]
    const int32_t *sptr;  // [core + 1] export rows of a core index
    const int32_t *vert;  // [core] vertex ids
    unsigned long long *maxbits;
};

// Forward elimination of the units: F, the exports, and this block's column
// sums of y^2 / d and of the original values squared over the eliminated
// vertices into my0, my1.
template <typename T, int R>
__device__ __forceinline__ void core_forward(const CoreKArgs<T> &k, T *ys, double *my0, double *my1) {
    constexpr int CG = UnitCols<T, R>::CG, NG = UnitCols<T, R>::NG;
    constexpr int V = UnitVec<T, CG>::V, LP = UnitVec<T, CG>::LP;
    __shared__ uint16_t s_roff_all[4][kUnitRounds + 2];
    __shared__ double s_red[32][32];
    const UnitArgs<T> &a = k.low;
    const UnitLevelArgs<T> &L = a.lv[0];
    const int G = (int)gridDim.x, me = (int)blockIdx.x;
    const bool al = ((uintptr_t)k.Y & 15) == 0 && (R * sizeof(T)) % 16 == 0;
    UnitGroup g;
    int groups = a.groups;
    while ((int)blockDim.x % (32 * groups)) groups >>= 1;
    g.nt = (int)blockDim.x / groups;
    const int gi = (int)threadIdx.x / g.nt;
    g.tid = (int)threadIdx.x - gi * g.nt;
    g.id = 1 + gi;
    const int GG = G * groups, mg = me + gi * G;
    uint16_t *s_roff = s_roff_all[gi];
    char *gsm = reinterpret_cast<char *>(ys) + (size_t)gi * a.gbytes;
    Acc<T> e1[NG][V], s1[NG][V];
    const int span = L.nu >= GG ? NG : 1, parts = NG / span;
    for (int t = mg; t < L.nu * parts; t += GG) {
        const int u = t / parts, cg0 = (t % parts) * span;
        const int4 m = L.meta[u];
        const int64_t base = (int64_t)u * L.B;
        const int size = (int)min((int64_t)L.B, L.n - base);
        const int32_t *ord = L.ord + base;
        const UnitSmem<T> s(gsm, m.y, m.x);
        unit_lists(g, L, u, m, s, s_roff);
        for (int q = 0; q < span; ++q) {
            const int c0 = (cg0 + q) * CG;
            unit_rows<T, R, CG>(g, s, ord, 0, size, k.Y + c0, al);
            cp_async_commit();
            cp_async_wait<0>();
            for (int it = g.tid; it < (m.y - size) * CG; it += g.nt) s.y[size * CG + it] = (T)0;
            g.sync();
            // a thread's pieces all hold the same V columns (the group has
            // whole warps and LP divides 32)
            for (int it = g.tid; it < m.x * LP; it += g.nt) {
                T v[V];
                uld<T, V>(s.y + it * V, true, v);
#pragma unroll
                for (int w = 0; w < NG; ++w)
                    if (w == cg0 + q) {
#pragma unroll
                        for (int x = 0; x < V; ++x) s1[w][x].add_prod(v[x], v[x]);
                    }
            }
            g.sync();
            unit_forward<T, CG>(g, s, m, s_roff);
            for (int it = g.tid; it < m.x * LP; it += g.nt) {
                const int p = it / LP, c = (it % LP) * V;
                const T d = L.coef[base + p].x;
                T v[V];
                uld<T, V>(s.y + it * V, true, v);
                ust<T, V>(k.F + (base + p) * R + c0 + c, true, v);
#pragma unroll
                for (int w = 0; w < NG; ++w)
                    if (w == cg0 + q) {
#pragma unroll
                        for (int x = 0; x < V; ++x) e1[w][x].add_prod(v[x], d * v[x]);
                    }
            }
            for (int it = g.tid; it < (m.y - m.x) * LP; it += g.nt) {
                const int j = it / LP, c = (it % LP) * V;
                T v[V];
                uld<T, V>(s.y + (m.x + j) * CG + c, true, v);
                ust<T, V>(L.exp + (int64_t)L.edst[m.w + j] * R + c0 + c, true, v);
            }
            g.sync();
        }
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NG; ++w) {
        block_cols<CG, LP, T>(e1[w], 0, s_red, my0 + w * CG);
        block_cols<CG, LP, T>(s1[w], 0, s_red, my1 + w * CG);
    }
}

// Back substitution: x = xi y / d + ... with the core's solution Xc.
template <typename T, int R>
__device__ __forceinline__ void core_backward(const CoreKArgs<T> &k, T *ys, const T *Xc,
                                              const double *xi, double &mx) {
    constexpr int CG = UnitCols<T, R>::CG, NG = UnitCols<T, R>::NG;
    constexpr int V = UnitVec<T, CG>::V, LP = UnitVec<T, CG>::LP;
    __shared__ uint16_t s_roff_all[4][kUnitRounds + 2];
    const UnitArgs<T> &a = k.low;
    const UnitLevelArgs<T> &L = a.lv[0];
    const int G = (int)gridDim.x, me = (int)blockIdx.x;
    const bool al = ((uintptr_t)k.X & 15) == 0 && (R * sizeof(T)) % 16 == 0;
    UnitGroup g;
    int groups = a.groups;
    while ((int)blockDim.x % (32 * groups)) groups >>= 1;
    g.nt = (int)blockDim.x / groups;
    const int gi = (int)threadIdx.x / g.nt;
    g.tid = (int)threadIdx.x - gi * g.nt;
    g.id = 1 + gi;
    const int GG = G * groups, mg = me + gi * G;
    uint16_t *s_roff = s_roff_all[gi];
    char *gsm = reinterpret_cast<char *>(ys) + (size_t)gi * a.gbytes;
    T tm = (T)0;
    const int span = L.nu >= GG ? NG : 1, parts = NG / span;
    __syncthreads();
    for (int t = mg; t < L.nu * parts; t += GG) {
        const int u = t / parts, cg0 = (t % parts) * span;
        const int4 m = L.meta[u];
        const int rounds = m.z & 0xffff;
        const int64_t base = (int64_t)u * L.B;
        const int size = (int)min((int64_t)L.B, L.n - base);
        const UnitSmem<T> s(gsm, m.y, m.x);
        const uint16_t *ro = L.roff + (int64_t)u * (kUnitRounds + 2);
        for (int q = g.tid; q <= rounds; q += g.nt) s_roff[q] = ro[q];
        unit_coef(g, L, u, m, s);
        for (int q = 0; q < span; ++q) {
            const int c0 = (cg0 + q) * CG;
            T sc[V];
#pragma unroll
            for (int x = 0; x < V; ++x) sc[x] = (T)xi[c0 + (g.tid % LP) * V + x];
            for (int it = g.tid; it < m.x * LP; it += g.nt) {
                T v[V];
                uld<T, V>(k.F + (base + it / LP) * R + c0 + (it % LP) * V, true, v);
#pragma unroll
                for (int x = 0; x < V; ++x) v[x] *= sc[x];
                ust<T, V>(s.y + it * V, true, v);
            }
            for (int it = g.tid; it < (m.y - m.x) * LP; it += g.nt) {
                const int j = it / LP, c = (it % LP) * V;
                T v[V];
                uld<T, V>(Xc + (int64_t)L.epos[m.w + j] * R + c0 + c, true, v);
                ust<T, V>(s.y + (m.x + j) * CG + c, true, v);
            }
            cp_async_commit();
            cp_async_wait<0>();
            g.sync();
            unit_backward<T, CG>(g, s, s_roff, rounds);
            unit_store<T, R, CG>(g, s, L.ord + base, 0, size, k.X + c0, al);
            for (int it = g.tid; it < size * CG; it += g.nt) tm = fmax(tm, fabs(s.y[it]));
            g.sync();
        }
    }
    mx = fmax(mx, (double)tm);
}

template <typename T, int R>
__global__ void __launch_bounds__(cg_max_threads<R, false>(), 1)
    k_core_cg(CGArgs<T> g, TreeKArgs<T> tk, CoreKArgs<T> k) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *ys = reinterpret_cast<T *>(smem_raw);
    __shared__ CoreScalars cs;
    unsigned int epoch = 0;
    double mx = 0.0;
    double *part0 = g.part, *part1 = g.part + (int64_t)gridDim.x * 32;
    core_forward<T, R>(k, ys, part0 + (int64_t)blockIdx.x * 32, part1 + (int64_t)blockIdx.x * 32);
    if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return;
    grid_cols2<R>(part0, cs.e1, part1, cs.s1);
    // the core's right-hand side: X = 0, R = Z = the exports' sums
    {
        constexpr int V = UnitVec<T, R>::V, LP = R / V;
        const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        const bool al = ((uintptr_t)k.Y & 15) == 0;
        for (int64_t it = gt; it < g.n * LP; it += (int64_t)gridDim.x * blockDim.x) {
            const int64_t i = it / LP;
            const int c = (int)(it % LP) * V;
            const int b = k.sptr[i], e = k.sptr[i + 1];
            T acc[V], y[V], zero[V];
#pragma unroll
            for (int x = 0; x < V; ++x) acc[x] = zero[x] = (T)0;
            uld<T, V>(k.Y + (int64_t)k.vert[i] * R + c, al, y);
#pragma unroll 4
            for (int j = b; j < e; ++j) {
                T v[V];
                uld<T, V>(k.low.lv[0].exp + (int64_t)j * R + c, true, v);
#pragma unroll
                for (int x = 0; x < V; ++x) acc[x] += v[x];
            }
#pragma unroll
            for (int x = 0; x < V; ++x) y[x] -= acc[x];
            ust<T, V>(g.X + i * R + c, true, zero);
            ust<T, V>(g.Rv + i * R + c, true, acc);
            ust<T, V>(g.Z + i * R + c, true, acc);
            ust<T, V>(k.dv + i * R + c, true, y);
        }
    }
    if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return;
    if (!cg_dev<T, R, false, true, true>(g, tk, epoch, ys, true, &cs, k.dv)) return;
    if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return;
    core_backward<T, R>(k, ys, g.X, cs.x, mx);
    if (k.maxbits) block_atomic_max(k.maxbits, mx);
}

struct CoreCall {
    grass_ctx_t ctx;
    grass_sparsifier_t S;
    grass_prec prec;
    const void *Y;
    void *X;
    double tol;
    int maxit;
    unsigned long long *maxbits;
};

template <typename T, int R>
static void core_T(const CoreCall &c) {
    grass_ctx_t ctx = c.ctx;
    CoreForm &C = *c.S->core;
    const int64_t n = c.S->tree->g.n, total = C.n * R;
    size_t smem = 0, smem_low = 0;
    TreeKArgs<T> tk;
    std::memset((void *)&tk, 0, sizeof(tk));
    tk.bar = ctx->gbar.p;
    tk.budget = ctx->wait_budget;
    tk.err = ctx->flags.p + 3;
    tk.u = unit_args<T, R>(C.tree, C.tree_f, &smem);
    CoreKArgs<T> k;
    std::memset((void *)&k, 0, sizeof(k));
    k.low = unit_args<T, R>(C.low, C.low_f, &smem_low);
    smem = std::max(smem, smem_low);
    k.low.lv[0].exp = ctx->scr<T>(SCR_CORE_E, (size_t)C.low.lv[0].nexp * R);
    k.Y = (const T *)c.Y;
    k.X = (T *)c.X;
    k.F = ctx->scr<T>(SCR_CG_XP, (size_t)n * R);
    k.dv = ctx->scr<T>(SCR_CORE_D, total);
    k.sptr = C.low.lv[0].sptr;
    k.vert = C.vert;
    k.maxbits = c.maxbits;
    CGArgs<T> a;
    std::memset((void *)&a, 0, sizeof(a));
    a.n = C.n;
    a.sptr = C.ptr;
    a.scol = C.col;
    if constexpr (sizeof(T) == 8) a.sw = C.w64;
    else a.sw = C.w32;
    a.X = ctx->scr<T>(SCR_CG_X, total);
    a.Rv = ctx->scr<T>(SCR_CG_R, total);
    a.Z = ctx->scr<T>(SCR_CG_Z, total);
    a.P = ctx->scr<T>(SCR_CG_P, total);
    a.Q = ctx->scr<T>(SCR_CG_Q, total);
    a.tol = c.tol;
    a.maxit = c.maxit;
    a.part = ctx->partials.p;
    a.iter_acc = ctx->scal.p + DS_RED + DS_ITER;
    const auto kern = k_core_cg<T, R>;
    const int threads = bounded_threads(ctx->tree_threads, cg_max_threads<R, false>());
    const int grid = coop_grid(ctx, kern, threads, smem, n * Lay<R>::TPR);
    if ((size_t)grid * 32 * 2 > ctx->partials.n) fail(GRASS_ERR_CUDA, "partials buffer too small");
    GCK(cudaMemsetAsync(tk.bar, 0, sizeof(unsigned int), ctx->stream));
    // bytes: both passes over all vertices (Y, F written and read, X, the
    // units' lists and coefficients), then the core's iterations as in
    // krylov.cu
    const double s = (double)sizeof(T), nrs = (double)total * s;
    const bool timing = ctx->tfam == GRASS_KF_CG;
    const size_t snap = ctx->iter_launches.size();
    if (timing) {
        ctx->t_snap(a.iter_acc, snap, 0);
        const double per = 2.0 * nrs + C.n * (10.0 + 4.0 * s) + 4.0 * (C.n + 1) +
                           C.nnz * (4.0 + s) + 2.0 * nrs + 13.0 * nrs;
        ctx->iter_launches.push_back({4.0 * n * R * s + n * (10.0 + 6.0 * s), per, snap});
    }
    bool timed = ctx->t_begin(GRASS_KF_CG, 0.0);
    void *args[] = {&a, &tk, &k};
    GCK(cudaLaunchCooperativeKernel((const void *)kern, dim3(grid), dim3(threads), args, smem,
                                    ctx->stream));
    ctx->launches++;
    ctx->t_end(timed);
    if (timing) ctx->t_snap(a.iter_acc, snap, 1);
}

template <int R>
static void core_R(const CoreCall &c) {
    if constexpr (R == 1) fail(GRASS_ERR_INVALID, "the core takes more than one column");
    else if (c.prec == GRASS_FP64) core_T<double, R>(c);
    else core_T<float, R>(c);
}

bool core_solve(grass_ctx_t ctx, grass_sparsifier_t S, int r, grass_prec prec, const void *Y, void *X,
                double tol, int maxit, unsigned long long *maxbits, int64_t its) {
    if (!core_wanted(S, r, prec, its) || !core_build(ctx, S)) return false;
    CoreCall c{ctx, S, prec, Y, X, tol, maxit, maxbits};
    GRASS_DISPATCH_R(r, core_R, c);
    return true;
}

}  // namespace grass
