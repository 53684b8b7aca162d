// cg.cuh -- device code of the r-column CG on the sparsifier, shared by the
// fused CG and PCG kernels (krylov.cu) and the CG on the sparsifier's core
// (core.cu).
#pragma once

#include "tree_solve.cuh"

namespace grass {

template <typename T>
struct CGArgs {
    int64_t n;
    const int32_t *sptr, *scol;
    const T *sw, *D;
    const T *Y;
    T *X, *Rv, *Z, *P, *Q;
    double tol;
    int maxit;
    double *part;                // [2][gridDim.x][32]
    double *iter_acc;            // += max over columns of the iterations; iter_acc[1] += 1
                                 // when a column reached the iteration cap
    unsigned long long *maxbits; // optional max |X|
    EulerKArgs eu;               // scan-form tree solve (r = 1, no D)
    // one column, scan form: perm != nullptr when the solve runs in another
    // numbering (X, Rv, Z, P, Q and the CSR indexed by k, vertex perm[k]); Y
    // is then read and the result written to Xout in vertex ids
    const int32_t *perm;
    T *Xout;
};

// The eliminated part of the sparsifier in a CG on its core (core.cu): one
// coordinate per column beside the core's vectors, in units of the column's
// eliminated right-hand side b1.  Shared memory; every block holds the same.
struct CoreScalars {
    double e1[32];     // b1' T11^{-1} b1
    double s1[32];     // |b1|^2
    double r[32], p[32], x[32];
};

// Per-block column sums of the thread partials v[e] (column c*EPT + e),
// written to out[0..R): lanes sharing c fold together (xor offsets >= TPR),
// then one thread per column adds the warps in order.
// TPR: lanes per group of columns (a thread of lane l holds columns
// (l mod TPR) * EPT ..), EPT = R / TPR.
template <int R, int TPR = Lay<R>::TPR>
__device__ __forceinline__ void block_cols(const double (&v)[R / TPR], int c,
                                           double (*s_red)[32], double *out) {
    constexpr int EPT = R / TPR;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        double x = v[e];
        for (int d = 16; d >= TPR; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
        if (lane < TPR) s_red[wid][lane * EPT + e] = x;
    }
    __syncthreads();
    if (threadIdx.x < R) {
        double s = 0.0;
        for (int w = 0; w < nw; ++w) s += s_red[w][threadIdx.x];
        out[threadIdx.x] = s;
    }
    __syncthreads();
}

template <int R, int TPR = Lay<R>::TPR, typename T>
__device__ __forceinline__ void block_cols(const Acc<T> (&a)[R / TPR], int c,
                                           double (*s_red)[32], double *out) {
    double v[R / TPR];
#pragma unroll
    for (int e = 0; e < R / TPR; ++e) v[e] = a[e].value();
    block_cols<R, TPR>(v, c, s_red, out);
}

// Column sums over all blocks' partials (same order in every block): warp j
// takes column j, lanes stride over the blocks, fixed xor tree.
// The loads of up to U x 32 blocks are issued before the first add (one
// round trip per U x 32 blocks instead of one per 32); the order of the
// adds is the plain one (lane, lane + 32, ...).
template <int R>
__device__ inline void grid_cols(const double *part, double *s_out) {
    constexpr int U = R == 1 ? 8 : 2;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int col = wid; col < R; col += (int)(blockDim.x >> 5)) {
        double s = 0.0;
        for (unsigned b0 = lane; b0 < gridDim.x; b0 += 32 * U) {
            double v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned b = b0 + 32 * u;
                v[u] = b < gridDim.x ? part[(int64_t)b * 32 + col] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (b0 + 32 * u < gridDim.x) s += v[u];
        }
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if (lane == 0) s_out[col] = s;
    }
    __syncthreads();
}

// threads of k_cg_persist: the scan form and r > 1 columns keep 1024
template <int R, bool EU>
__host__ __device__ constexpr int cg_max_threads() { return (EU || R > 1) ? kPersistMaxThreads : kFusedMaxThreads; }

// Laplacian rows of a CSR (off-diagonal weights w, columns col) applied to
// x with stride S: q[u] += w_j (xi[u] - x[col_j * S]) over the entries
// [jb[u], je[u]) of each row, in j order.  The first K entries of every row
// (indices and weights, then the gathers) are loaded before any arithmetic;
// a longer row goes on K entries at a time.
template <typename T, int U, int K, int S>
__device__ __forceinline__ void lap_rows(const int32_t *col, const T *w, const T *x, int32_t (&jb)[U],
                                         const int32_t (&je)[U], const T (&xi)[U], T (&q)[U]) {
    bool more = true;
    while (more) {
        int32_t cc[U][K];
        T wv[U][K], xc[U][K];
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int32_t j = jb[u] + k;
                const bool v = j < je[u];
                cc[u][k] = v ? col[j] : 0;
                wv[u][k] = v ? w[j] : (T)0;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int k = 0; k < K; ++k) xc[u][k] = jb[u] + k < je[u] ? x[(int64_t)cc[u][k] * S] : (T)0;
        }
        more = false;
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (jb[u] + k < je[u]) q[u] += wv[u][k] * (xi[u] - xc[u][k]);
            jb[u] += K;
            more = more || jb[u] < je[u];
        }
    }
}

// Two column sums at once: warps 0..R-1 reduce part0 and warps R..2R-1
// part1 (each the same order as grid_cols), when the block has 2R warps.
template <int R>
__device__ inline void grid_cols2(const double *part0, double *s_out0, const double *part1,
                                  double *s_out1) {
    if (2 * R > (int)(blockDim.x >> 5)) {
        grid_cols<R>(part0, s_out0);
        grid_cols<R>(part1, s_out1);
        return;
    }
    constexpr int U = R == 1 ? 8 : 2;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (wid < 2 * R) {
        const double *part = wid < R ? part0 : part1;
        const int col = wid < R ? wid : wid - R;
        double s = 0.0;
        for (unsigned b0 = lane; b0 < gridDim.x; b0 += 32 * U) {
            double v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned b = b0 + 32 * u;
                v[u] = b < gridDim.x ? part[(int64_t)b * 32 + col] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (b0 + 32 * u < gridDim.x) s += v[u];
        }
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if (lane == 0) (wid < R ? s_out0 : s_out1)[col] = s;
    }
    __syncthreads();
}

// The whole inner CG as a device function of a cooperative grid (used by
// k_cg_persist and inside the fused PCG).  Returns false when a barrier wait
// ran out (the caller must return).  Ends without a trailing grid barrier:
// every element of X is last written (and read by the max |X| pass) by the
// thread that owns it under the element mapping (one column: the chunks of
// for_chunks; else rows slot, slot + nslots, ... and columns c*EPT ..), so
// a caller with the same mapping
// reads X at once.  preset: the caller has already set X = 0, R = Z = Y and
// passed a grid barrier since.
// CORE (core.cu): the vectors are the core's; cs holds the eliminated
// part's coordinate of every column, dv the difference between the core's
// original and eliminated right-hand sides, so that |r|^2 of the whole
// sparsifier is |r + cs.r dv|^2 + cs.r^2 cs.s1.
template <typename T, int R, bool EU, bool UNITS, bool CORE = false>
__device__ __forceinline__ bool cg_dev(const CGArgs<T> &g, const TreeKArgs<T> &tk,
                                       unsigned int &epoch, T *ys, bool preset = false,
                                       CoreScalars *cs = nullptr, const T *dv = nullptr) {
    static_assert(!EU || R == 1, "the scan-form solve handles one column");
    static_assert(!CORE || R > 1, "one column takes the scan form");
    constexpr int TPR = Lay<R>::TPR, EPT = Lay<R>::EPT;
    __shared__ double s_red[32][32];
    __shared__ double s_rz[32], s_rr[32], s_yy[32], s_pq[32], s_new[32], s_al[32];
    __shared__ int s_act[32], s_brk[32], s_it[32], s_nact;
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = (int)(gt % TPR);
    const int64_t slot = gt / TPR, nslots = (int64_t)gridDim.x * blockDim.x / TPR;
    double *part0 = g.part, *part1 = g.part + (int64_t)gridDim.x * 32;
    double *mypart0 = part0 + (int64_t)blockIdx.x * 32, *mypart1 = part1 + (int64_t)blockIdx.x * 32;
    double mx = 0.0;
    // Element loops in chunks (for_chunks): one column (chunks of rows, the
    // mapping the fused PCG uses for the same vectors), or for FP32 and
    // r = 4, 8, 16, 32 the n x r array as flat 4-float chunks; the thread
    // count is a multiple of r / 4, so a thread's chunks all hold columns
    // c4 .. c4 + 3 (c4 = 4 (gt mod r/4)): NA sums per thread, laid out for
    // block_cols as groups of TPA lanes.
    constexpr bool CH1 = R == 1;
    constexpr bool CHR = sizeof(T) == 4 && (R == 4 || R == 8 || R == 16 || R == 32);
    constexpr bool CH = CH1 || CHR;
    constexpr int W = Chunk<T>::W;
    constexpr int NA = CHR ? 4 : EPT;
    constexpr int TPA = CHR ? R / 4 : TPR;
    const int64_t nel = CHR ? g.n * R : g.n;
    const int c4 = CHR ? (int)(gt % (R / 4)) * 4 : 0;
    Acc<T> acc0[NA], acc1[NA];

    if (!preset && CH) {
        for_chunks<T>(nel, gt, (int64_t)gridDim.x * blockDim.x, [&](int64_t i0, int cnt) {
            T y[W], zero[W] = {};
            bool gathered = false;
            if constexpr (EU) {
                if (g.perm) {
#pragma unroll
                    for (int w = 0; w < W; ++w) y[w] = w < cnt ? g.Y[g.perm[i0 + w]] : (T)0;
                    gathered = true;
                }
            }
            if (!gathered) ld_chunk(g.Y + i0, cnt, y);
            st_chunk(g.X + i0, cnt, zero);
            st_chunk(g.Rv + i0, cnt, y);
            st_chunk(g.Z + i0, cnt, y);
        });
        if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return false;
    } else if (!preset) {
        for (int64_t i = slot; i < g.n; i += nslots) {
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
                int64_t k = i * R + c * EPT + e;
                T y = g.Y[k];
                g.X[k] = (T)0;
                g.Rv[k] = y;
                g.Z[k] = y;
            }
        }
        if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return false;
    }
    if (threadIdx.x < R) {
        s_brk[threadIdx.x] = 0;
        s_it[threadIdx.x] = 0;
        if constexpr (CORE) {
            cs->r[threadIdx.x] = 1.0;
            cs->p[threadIdx.x] = cs->x[threadIdx.x] = 0.0;
        }
    }
    // Iteration `it` starts with Z = M^{-1} R (the only call site of the
    // tree solve), then P (it = 0: P = Z; else P = Z + beta P), then the
    // stop test (a column goes on while ||r|| > tol ||y||), the product and the
    // updates.  After the updates the test is looked at once more, so no
    // solve is spent when no column goes on.
    for (int it = 0;; ++it) {
        // the scan form writes Z with the element loops' own mapping (no
        // barrier); the elimination rounds write out of order
        if constexpr (EU) {
            if (!euler_solve_dev<T, true>(g.eu, g.Z, tk.bar, tk.budget, tk.err, epoch, mx)) return false;
        } else {
            if (!tree_solve_dev<T, R, false, UNITS>(tk, g.Z, epoch, mx, ys)) return false;
            if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return false;
        }
#pragma unroll
        for (int e = 0; e < NA; ++e) acc0[e] = acc1[e] = Acc<T>();
        if constexpr (CH) {
            for_chunks<T>(nel, gt, (int64_t)gridDim.x * blockDim.x, [&](int64_t i0, int cnt) {
                T z[W], rr[W], rf[W] = {};
                ld_chunk(g.Z + i0, cnt, z);
                ld_chunk(g.Rv + i0, cnt, rr);
                if (CORE && it == 0) ld_chunk(dv + i0, cnt, rf);
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    if (w >= cnt) break;
                    acc0[CHR ? w : 0].add_prod(rr[w], z[w]);
                    rf[w] += rr[w];
                    if (it == 0) acc1[CHR ? w : 0].add_prod(rf[w], rf[w]);
                }
                if (it == 0) st_chunk(g.P + i0, cnt, z);
            });
        } else {
        for (int64_t i = slot; i < g.n; i += nslots) {
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
                int64_t k = i * R + c * EPT + e;
                T z = g.Z[k], rr = g.Rv[k];
                acc0[e].add_prod(rr, z);
                if (it == 0) {
                    g.P[k] = z;
                    if constexpr (CORE) rr += dv[k];
                    acc1[e].add_prod(rr, rr);
                }
            }
        }
        }
        block_cols<R, TPA>(acc0, c, s_red, mypart0);
        if (it == 0) block_cols<R, TPA>(acc1, c, s_red, mypart1);
        if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return false;
        if (it == 0) {
            grid_cols2<R>(part0, s_rz, part1, s_rr);
            if constexpr (CORE) {
                if (threadIdx.x < R) {
                    const int j = threadIdx.x;
                    s_rz[j] += cs->e1[j];
                    s_rr[j] += cs->s1[j];
                    cs->p[j] = 1.0;
                }
                __syncthreads();
            }
            if (threadIdx.x < R) s_yy[threadIdx.x] = s_rr[threadIdx.x];
            __syncthreads();
        } else {
            grid_cols<R>(part0, s_new);
            if (threadIdx.x < R) {
                int j = threadIdx.x;
                if constexpr (CORE) s_new[j] += cs->r[j] * cs->r[j] * cs->e1[j];
                double beta = s_act[j] ? s_new[j] / s_rz[j] : 0.0;
                if (s_act[j]) s_rz[j] = s_new[j];
                if constexpr (CORE)
                    if (s_act[j]) cs->p[j] = cs->r[j] + beta * cs->p[j];
                s_al[j] = beta;
            }
            __syncthreads();
            if constexpr (CH1) {
                if (s_act[0]) {
                    const T be = (T)s_al[0];
                    for_chunks<T>(g.n, gt, (int64_t)gridDim.x * blockDim.x, [&](int64_t i0, int cnt) {
                        T z[W], pv[W];
                        ld_chunk(g.Z + i0, cnt, z);
                        ld_chunk(g.P + i0, cnt, pv);
#pragma unroll
                        for (int w = 0; w < W; ++w) pv[w] = z[w] + be * pv[w];
                        st_chunk(g.P + i0, cnt, pv);
                    });
                }
            } else if constexpr (CHR) {
                for_chunks<T>(nel, gt, (int64_t)gridDim.x * blockDim.x, [&](int64_t i0, int cnt) {
                    T z[W], pv[W];
                    ld_chunk(g.Z + i0, cnt, z);
                    ld_chunk(g.P + i0, cnt, pv);
#pragma unroll
                    for (int w = 0; w < W; ++w)
                        if (s_act[c4 + w]) pv[w] = z[w] + (T)s_al[c4 + w] * pv[w];
                    st_chunk(g.P + i0, cnt, pv);
                });
            } else {
            for (int64_t i = slot; i < g.n; i += nslots) {
#pragma unroll
                for (int e = 0; e < EPT; ++e) {
                    int j = c * EPT + e;
                    if (!s_act[j]) continue;
                    int64_t k = i * R + j;
                    g.P[k] = g.Z[k] + (T)s_al[j] * g.P[k];
                }
            }
            }
            if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return false;
        }
        if (it >= g.maxit) break;
        // stop test per column: a column goes on while ||r|| > tol ||y||
        if (threadIdx.x == 0) s_nact = 0;
        __syncthreads();
        if (threadIdx.x < R) {
            int j = threadIdx.x;
            int a = !s_brk[j] && sqrt(s_rr[j]) > g.tol * sqrt(s_yy[j]);
            s_act[j] = a;
            if (a) atomicAdd(&s_nact, 1);
        }
        __syncthreads();
        if (s_nact == 0) break;
        // Q = L_S P (+D), partial P.Q (row layout)
        Acc<T> accq[EPT];
#pragma unroll
        for (int e = 0; e < EPT; ++e) accq[e] = Acc<T>();
        if constexpr (EPT == 1 && (EU || cg_max_threads<R, EU>() <= kFusedMaxThreads)) {
            // two rows at a time, every load of both rows before the sums
            constexpr int K = 4;
            for (int64_t i0 = slot; i0 < g.n; i0 += 2 * nslots) {
                int32_t jb[2], je[2];
                T p0[2], q[2], dd[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int64_t i = i0 + u * nslots;
                    const bool ok = i < g.n;
                    p0[u] = ok ? g.P[i * R + c] : (T)0;
                    dd[u] = ok && g.D ? g.D[i] : (T)0;
                    jb[u] = ok ? g.sptr[i] : 0;
                    je[u] = ok ? g.sptr[i + 1] : 0;
                    q[u] = (T)0;
                }
                lap_rows<T, 2, K, R>(g.scol, g.sw, g.P + c, jb, je, p0, q);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int64_t i = i0 + u * nslots;
                    if (i >= g.n) break;
                    if (g.D) q[u] += dd[u] * p0[u];
                    g.Q[i * R + c] = q[u];
                    accq[0].add_prod(p0[u], q[u]);
                }
            }
        } else {
        for (int64_t i = slot; i < g.n; i += nslots) {
            T p0[EPT], q[EPT];
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
                p0[e] = g.P[i * R + c * EPT + e];
                q[e] = (T)0;
            }
            for (int32_t j = g.sptr[i]; j < g.sptr[i + 1]; ++j) {
                const T *pq = g.P + (int64_t)g.scol[j] * R + c * EPT;
                T w = g.sw[j];
#pragma unroll
                for (int e = 0; e < EPT; ++e) q[e] += w * (p0[e] - pq[e]);
            }
            if (g.D) {
                T dd = g.D[i];
#pragma unroll
                for (int e = 0; e < EPT; ++e) q[e] += dd * p0[e];
            }
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
                g.Q[i * R + c * EPT + e] = q[e];
                accq[e].add_prod(p0[e], q[e]);
            }
        }
        }
        block_cols<R>(accq, c, s_red, mypart0);
        if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return false;
        grid_cols<R>(part0, s_pq);
        if (threadIdx.x < R) {
            int j = threadIdx.x;
            double pq = s_pq[j];
            if constexpr (CORE) pq += cs->p[j] * cs->p[j] * cs->e1[j];
            if (s_act[j] && !(pq > 0.0)) {
                s_brk[j] = 1;
                s_act[j] = 0;
            }
            s_al[j] = s_act[j] ? s_rz[j] / pq : 0.0;
            if constexpr (CORE) {
                cs->x[j] += s_al[j] * cs->p[j];
                cs->r[j] -= s_al[j] * cs->p[j];
            }
            if (s_act[j]) s_it[j] += 1;
        }
        __syncthreads();
        // X += alpha P, R -= alpha Q, Z = R, partial R.R
#pragma unroll
        for (int e = 0; e < NA; ++e) acc1[e] = Acc<T>();
        if constexpr (CHR) {
            for_chunks<T>(nel, gt, (int64_t)gridDim.x * blockDim.x, [&](int64_t i0, int cnt) {
                T rr[W], xv[W], pv[W], qv[W];
                ld_chunk(g.Rv + i0, cnt, rr);
                ld_chunk(g.X + i0, cnt, xv);
                ld_chunk(g.P + i0, cnt, pv);
                ld_chunk(g.Q + i0, cnt, qv);
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const T a = (T)s_al[c4 + w];
                    if (a != (T)0) {
                        xv[w] += a * pv[w];
                        rr[w] -= a * qv[w];
                    }
                }
                st_chunk(g.X + i0, cnt, xv);
                st_chunk(g.Rv + i0, cnt, rr);
                st_chunk(g.Z + i0, cnt, rr);
                if constexpr (CORE) {
                    ld_chunk(dv + i0, cnt, qv);
#pragma unroll
                    for (int w = 0; w < W; ++w) rr[w] += (T)cs->r[c4 + w] * qv[w];
                }
#pragma unroll
                for (int w = 0; w < W; ++w) acc1[w].add_prod(rr[w], rr[w]);
            });
        } else if constexpr (CH1) {
            const T a = (T)s_al[0];
            for_chunks<T>(g.n, gt, (int64_t)gridDim.x * blockDim.x, [&](int64_t i0, int cnt) {
                T rr[W];
                ld_chunk(g.Rv + i0, cnt, rr);
                if (a != (T)0) {
                    T xv[W], pv[W], qv[W];
                    ld_chunk(g.X + i0, cnt, xv);
                    ld_chunk(g.P + i0, cnt, pv);
                    ld_chunk(g.Q + i0, cnt, qv);
#pragma unroll
                    for (int w = 0; w < W; ++w) {
                        xv[w] += a * pv[w];
                        rr[w] -= a * qv[w];
                    }
                    st_chunk(g.X + i0, cnt, xv);
                    st_chunk(g.Rv + i0, cnt, rr);
                }
                st_chunk(g.Z + i0, cnt, rr);
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    if (w >= cnt) break;
                    acc1[0].add_prod(rr[w], rr[w]);
                }
            });
        } else {
        for (int64_t i = slot; i < g.n; i += nslots) {
#pragma unroll
            for (int e = 0; e < EPT; ++e) {
                int64_t k = i * R + c * EPT + e;
                T a = (T)s_al[c * EPT + e];
                T rr = g.Rv[k];
                if (a != (T)0) {
                    g.X[k] += a * g.P[k];
                    rr -= a * g.Q[k];
                    g.Rv[k] = rr;
                }
                g.Z[k] = rr;
                if constexpr (CORE) rr += (T)cs->r[c * EPT + e] * dv[k];
                acc1[e].add_prod(rr, rr);
            }
        }
        }
        // look ahead: another iteration only if one is allowed and some
        // column passes the test
        if (it + 1 >= g.maxit) break;
        block_cols<R, TPA>(acc1, c, s_red, mypart1);
        if (!grid_sync(tk.bar, tk.budget, tk.err, epoch)) return false;
        grid_cols<R>(part1, s_rr);
        if constexpr (CORE) {
            if (threadIdx.x < R) s_rr[threadIdx.x] += cs->r[threadIdx.x] * cs->r[threadIdx.x] * cs->s1[threadIdx.x];
        }
        if (threadIdx.x == 0) s_nact = 0;
        __syncthreads();
        if (threadIdx.x < R) {
            int j = threadIdx.x;
            if (!s_brk[j] && sqrt(s_rr[j]) > g.tol * sqrt(s_yy[j])) atomicAdd(&s_nact, 1);
        }
        __syncthreads();
        if (s_nact == 0) break;
    }
    if (g.maxbits) {
        double m = 0.0;
        if constexpr (CH) {
            for_chunks<T>(nel, gt, (int64_t)gridDim.x * blockDim.x, [&](int64_t i0, int cnt) {
                T xv[W];
                ld_chunk(g.X + i0, cnt, xv);
#pragma unroll
                for (int w = 0; w < W; ++w) m = fmax(m, fabs((double)xv[w]));
            });
        } else {
        for (int64_t i = slot; i < g.n; i += nslots) {
#pragma unroll
            for (int e = 0; e < EPT; ++e) m = fmax(m, fabs((double)g.X[i * R + c * EPT + e]));
        }
        }
        block_atomic_max(g.maxbits, m);
    }
    if constexpr (CH1 && EU) {
        // back to vertex ids: each thread scatters the elements it owns
        if (g.perm) {
            for_chunks<T>(g.n, gt, (int64_t)gridDim.x * blockDim.x, [&](int64_t i0, int cnt) {
                T xv[W];
                ld_chunk(g.X + i0, cnt, xv);
#pragma unroll
                for (int w = 0; w < W; ++w)
                    if (w < cnt) g.Xout[g.perm[i0 + w]] = xv[w];
            });
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int mxit = 0;
        for (int j = 0; j < R; ++j) mxit = max(mxit, s_it[j]);
        *g.iter_acc += (double)mxit;
        if (mxit >= g.maxit) g.iter_acc[1] += 1.0;
    }
    return true;
}

}  // namespace grass
