// units.cuh -- device code of the unit form of the tree solve.
//
// The elimination rounds of tree.cu pass a grid barrier per round (about 9
// forward and 9 backward at a million vertices).  In the unit form the
// vertices, in a preorder that visits every vertex's largest subtree last,
// are cut into units of B consecutive positions; one block eliminates the
// inside of a unit in shared memory (rake and compress rounds separated by
// block barriers) down to the vertices that have a child in another unit
// and the few branching ones between them.  What survives is again a tree,
// about 3 vertices per unit, and is cut into units the same way until one
// unit is left (units.cu builds all of it).  A solve is then one grid phase
// per level forward, one block-local solve of the last level, and one grid
// phase per level backward: three phases and two barriers at a million
// vertices.
//
// Inside a unit: local indices 0 .. nel-1 are the eliminated vertices in
// elimination order, nel .. size-1 the survivors, size .. local-1 the
// vertices of earlier units that vertices of this one hang from.  A
// vertex's forward value is its right-hand side plus the multiplied values
// of the neighbours eliminated before it, gathered in elimination order
// when its own round comes; survivors and outside vertices gather the same
// way at the end and go out as the unit's exports, which the next level
// adds up per vertex in a fixed order.
//
// What bounds it: the block-local rounds' chains of dependent shared-memory
// reads and block barriers (0.2-0.5 us a round, 9-11 rounds a unit), then the
// rows' way in and out; FP64 with 8 columns and more is bound by the FP64
// pipe (about 80M operations at 16 columns).  1M vertices, 608 units of
// 1645, per call, back to back on the same buffers (the rounds form in
// brackets; on other buffers each call 16 FP32 columns 147): FP32 1 column 54 us (120; the
// kernel alone 29 and 121), 4 columns 68 (156), 16 columns 131 (234), FP64
// 1 column 85 (147), 8 columns 217 (268); 90,000 vertices FP32 41-54 (80-105).
#pragma once

#include "common.cuh"

namespace grass {

template <typename T>
struct PackT;
template <>
struct PackT<float> {
    using V2 = float2;
    using V4 = float4;
};
template <>
struct PackT<double> {
    using V2 = double2;
    using V4 = Dbl4;
};

constexpr int kUnitHeavy = 64;      // lists longer than this are summed by a warp

template <typename T>
struct UnitLevelArgs {
    int64_t n;
    int B, nu;
    const int32_t *ord;         // level 0: position -> vertex id; above, null: rows by position
    const int4 *meta;           // per unit {eliminated, local indices, rounds | long lists << 16, first export}
    const uint16_t *roff;       // per unit [kUnitRounds + 2] first position of every round
    const uint16_t *cbeg;       // per unit [unit_stride(B)] list starts by local index
    const uint16_t *clist;      // per unit [unit_stride(B)] contributor positions
    const T *cm;                // per unit [unit_stride(B)] their multipliers
    const int32_t *epos;        // next level's position of every export
    const int32_t *edst;        // its row in this level's export array
    const typename PackT<T>::V4 *coef;   // by position {1/d, w1/d, w2/d, n1 | n2 << 16}
    const int32_t *sptr;        // levels >= 1: [n + 1] the previous level's export rows by position
    T *V;                       // levels >= 1: the level's vector [n x R], by position
    T *exp;                     // exports of this level [nexp x R], grouped by the next level's position
};

template <typename T>
struct UnitArgs {
    int nl;                     // levels (0: no unit form)
    int groups;                 // units a block works on at once (1, 2 or 4 thread groups)
    int gbytes;                 // shared memory of one of them
    const T *rinv;              // 1 / pivot of the root (0: grounded)
    UnitLevelArgs<T> lv[kUnitLevels];
};

// Columns worked on at a time (CG; the last level, one block per column
// group: TG): rows of 64 bytes where they fit beside the lists.  Measured,
// 1M vertices: 16 FP32 columns at once 131 us a solve, 8 at a time (two
// units side by side) 143, 8 at a time with the next 8 loaded meanwhile 177;
// 8 FP64 columns at once 217 us, 4 at a time 325.
template <typename T, int R>
struct UnitCols {
    static constexpr int CG = sizeof(T) == 4 ? (R == 24 ? 8 : R > 16 ? 16 : R) : (R > 8 ? 8 : R);
    static constexpr int NG = R / CG;
    static constexpr int TG = sizeof(T) == 4 ? (R > 4 ? 4 : R) : 1;
};

// Shared memory of one unit: the forward pass's multipliers, contributors
// and list starts, or the backward pass's coefficients, in one region; then
// the rows.
template <typename T>
struct UnitSmem {
    T *y;
    typename PackT<T>::V4 *cf;
    T *cm;
    uint16_t *cl, *cb;
    __host__ __device__ static size_t up(size_t x) { return (x + 31) & ~size_t(31); }
    // the staged arrays are copied in whole 16-byte pieces: each is rounded up
    __host__ __device__ static size_t lists(int local, int elim) {
        const size_t f = up(2 * (size_t)elim * sizeof(T)) + up(2 * (size_t)elim * sizeof(uint16_t)) +
                         up(((size_t)local + 1) * sizeof(uint16_t));
        const size_t b = up((size_t)elim * sizeof(typename PackT<T>::V4));
        return f > b ? f : b;
    }
    __host__ __device__ static size_t rows(int local, int cg) {
        return up((size_t)local * cg * sizeof(T));
    }
    __device__ UnitSmem(void *p, int local, int elim) {
        char *q = reinterpret_cast<char *>(p);
        cf = reinterpret_cast<typename PackT<T>::V4 *>(q);
        cm = reinterpret_cast<T *>(q);
        size_t o = up(2 * (size_t)elim * sizeof(T));
        cl = reinterpret_cast<uint16_t *>(q + o);
        o = up(o + 2 * (size_t)elim * sizeof(uint16_t));
        cb = reinterpret_cast<uint16_t *>(q + o);
        y = reinterpret_cast<T *>(q + lists(local, elim));
    }
};

// Host side: thread groups and dynamic shared memory for R columns.  local,
// elim: the largest unit of the levels below the last; tlocal, telim: of the
// last.
template <typename T, int R>
inline size_t unit_shape(UnitArgs<T> &a, int local, int elim, int tlocal, int telim) {
    using C = UnitCols<T, R>;
    const size_t top = UnitSmem<T>::lists(tlocal, telim) + UnitSmem<T>::rows(tlocal, C::TG);
    const size_t one = elim > 0 ? UnitSmem<T>::lists(local, elim) + UnitSmem<T>::rows(local, C::CG)
                                : 32;
    a.groups = 4 * one <= kTailSmem ? 4 : 2 * one <= kTailSmem ? 2 : 1;
    a.gbytes = (int)one;
    const size_t all = one * a.groups;
    return all > top ? all : top;
}

// The threads that work on one unit: the whole block, or one of 2 or 4 equal
// parts of it with a barrier of its own.
struct UnitGroup {
    int tid, nt, id;
    __device__ __forceinline__ void sync() const {
        asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nt) : "memory");
    }
};

__device__ __forceinline__ uint32_t unit_nn(const float4 &c) { return __float_as_uint(c.w); }
__device__ __forceinline__ uint32_t unit_nn(const Dbl4 &c) {
    return (uint32_t)__double_as_longlong(c.w);
}

// V consecutive elements, by one vector access when `al` (the row pieces are
// 16-byte aligned), else one by one
template <typename T, int V>
__device__ __forceinline__ void uld(const T *p, bool al, T (&v)[V]) {
    if constexpr (V * sizeof(T) == 16) {
        if (al) {
            if constexpr (sizeof(T) == 4) {
                const float4 q = *reinterpret_cast<const float4 *>(p);
                v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
            } else {
                const double2 q = *reinterpret_cast<const double2 *>(p);
                v[0] = q.x, v[1] = q.y;
            }
            return;
        }
    }
#pragma unroll
    for (int e = 0; e < V; ++e) v[e] = p[e];
}
template <typename T, int V>
__device__ __forceinline__ void ust(T *p, bool al, const T (&v)[V]) {
    if constexpr (V * sizeof(T) == 16) {
        if (al) {
            if constexpr (sizeof(T) == 4)
                *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
            else *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
            return;
        }
    }
#pragma unroll
    for (int e = 0; e < V; ++e) p[e] = v[e];
}

template <typename T, int CG>
struct UnitVec {
    static constexpr int V = (CG * sizeof(T)) % 16 == 0 ? 16 / (int)sizeof(T) : 1;
    static constexpr int LP = CG / V;   // lanes per row
};

// Asynchronous copies into shared memory: a unit's rows, lists and
// coefficients (about 150 KB an SM) are all in flight at once and hold no
// registers (with 4 row pieces a thread in registers a unit's loads took
// 9.5 us of its 17 at 16 FP32 columns).
template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES)
                     : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the last N committed groups have arrived
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// bytes (rounded up to 16) from a 16-byte aligned array
__device__ __forceinline__ void unit_copy(const UnitGroup &g, void *dst, const void *src, int bytes) {
    char *d = static_cast<char *>(dst);
    const char *q = static_cast<const char *>(src);
    for (int o = g.tid * 16; o < bytes; o += g.nt * 16) cp_async<16>(d + o, q + o);
}

// Rows [p0, p1) of W (row ord[p], columns at W) into shared memory.
template <typename T, int R, int CG>
__device__ __forceinline__ void unit_rows(const UnitGroup &g, const UnitSmem<T> &s,
                                          const int32_t *ord, int p0, int p1, const T *W, bool al) {
    constexpr int V = UnitVec<T, CG>::V, LP = UnitVec<T, CG>::LP, NB = 4;
    const int end = p1 * LP;
    for (int i0 = p0 * LP + g.tid; i0 < end; i0 += NB * g.nt) {
        int32_t o[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int it = i0 + k * g.nt;
            o[k] = it >= end ? 0 : ord ? ord[it / LP] : it / LP;
        }
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int it = i0 + k * g.nt;
            if (it >= end) break;
            const T *q = W + (int64_t)o[k] * R + (it % LP) * V;
            T *d = s.y + it * V;
            if (V == 1 || al) {
                cp_async<V * sizeof(T)>(d, q);
            } else {
#pragma unroll
                for (int e = 0; e < V; ++e) cp_async<sizeof(T)>(d + e, q + e);
            }
        }
    }
}

// Calls f(p) for every p in [lo, hi) whose list len(p) is long, a warp at a
// time (all lanes call f together); warps scan 32 lengths per step.
template <typename LEN, typename F>
__device__ __forceinline__ void unit_heavy(const UnitGroup &g, int lo, int hi, LEN len, F f) {
    const int lane = g.tid & 31;
    for (int p0 = lo + (g.tid & ~31); p0 < hi; p0 += g.nt) {
        const int p = p0 + lane;
        unsigned mask = __ballot_sync(0xffffffffu, p < hi && len(p) > kUnitHeavy);
        for (; mask; mask &= mask - 1) f(p0 + __ffs(mask) - 1);
    }
}

// y[p] += sum of the contributions to local index p, p in [lo, hi), with SP
// lanes sharing a list: lane k takes entries k, k + SP, ... and a fixed xor
// tree adds the lanes.
template <typename T, int CG, int SP>
__device__ __forceinline__ void unit_gather_sp(const UnitGroup &g, const UnitSmem<T> &s, int lo,
                                               int hi) {
    constexpr int V = UnitVec<T, CG>::V, LP = UnitVec<T, CG>::LP;
    const int total = (hi - lo) * LP * SP;
    for (int i0 = g.tid & ~31; i0 < total; i0 += g.nt) {
        const int it = i0 + (g.tid & 31);
        const bool on = it < total;
        const int p = lo + it / (LP * SP), c = (it % LP) * V, k = (it / LP) % SP;
        const int b = on ? s.cb[p] : 0, e = on ? s.cb[p + 1] : 0;
        const bool mine = e > b && e - b <= kUnitHeavy;
        T acc[V];
#pragma unroll
        for (int x = 0; x < V; ++x) acc[x] = (T)0;
        if (mine && k == 0) uld<T, V>(s.y + p * CG + c, true, acc);
        if (mine) {
            // NB entries' loads before the first product
            constexpr int NB = SP == 1 ? 4 : 2;
            for (int j0 = b + k; j0 < e; j0 += NB * SP) {
                int v[NB];
                T m[NB], yv[NB][V];
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    const int j = min(j0 + q * SP, e - 1);
                    v[q] = s.cl[j];
                    m[q] = j0 + q * SP < e ? s.cm[j] : (T)0;
                }
#pragma unroll
                for (int q = 0; q < NB; ++q) uld<T, V>(s.y + v[q] * CG + c, true, yv[q]);
#pragma unroll
                for (int q = 0; q < NB; ++q) {
                    if (j0 + q * SP >= e) break;
#pragma unroll
                    for (int x = 0; x < V; ++x) acc[x] += m[q] * yv[q][x];
                }
            }
        }
#pragma unroll
        for (int d = LP; d < LP * SP; d <<= 1) {
#pragma unroll
            for (int x = 0; x < V; ++x) acc[x] += __shfl_xor_sync(0xffffffffu, acc[x], d);
        }
        if (mine && k == 0) ust<T, V>(s.y + p * CG + c, true, acc);
    }
}

// One forward round of a unit; ends with the group's barrier.  Late rounds
// have few vertices with long lists (a vertex collects from every round it
// has lived through), so the fewer the vertices the more lanes share a list;
// the split depends on the round's size alone, so results do not depend on
// the launch shape.
template <typename T, int CG>
__device__ __forceinline__ void unit_gather(const UnitGroup &g, const UnitSmem<T> &s, int lo, int hi,
                                            bool heavy) {
    const int work = (hi - lo) * UnitVec<T, CG>::LP;
    if (work > 192) unit_gather_sp<T, CG, 1>(g, s, lo, hi);
    else if (work > 48) unit_gather_sp<T, CG, 4>(g, s, lo, hi);
    else unit_gather_sp<T, CG, 8>(g, s, lo, hi);
    g.sync();
    if (!heavy) return;
    const int lane = g.tid & 31;
    unit_heavy(g, lo, hi, [&](int p) { return s.cb[p + 1] - s.cb[p]; }, [&](int p) {
        const int b = s.cb[p], e = s.cb[p + 1];
        for (int c = 0; c < CG; ++c) {
            T acc = (T)0;
            for (int j = b + lane; j < e; j += 32) acc += s.cm[j] * s.y[(int)s.cl[j] * CG + c];
            for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
            if (lane == 0) s.y[p * CG + c] += acc;
        }
    });
    g.sync();
}

// Stage a unit's lists and round offsets (asynchronous copies).
template <typename T>
__device__ __forceinline__ void unit_lists(const UnitGroup &g, const UnitLevelArgs<T> &L, int u,
                                           const int4 m, const UnitSmem<T> &s, uint16_t *s_roff) {
    const int64_t lo = (int64_t)u * unit_stride(L.B);
    const uint16_t *ro = L.roff + (int64_t)u * (kUnitRounds + 2);
    unit_copy(g, s.cb, L.cbeg + lo, (m.y + 1) * (int)sizeof(uint16_t));
    const int nc = L.cbeg[lo + m.y];
    unit_copy(g, s.cl, L.clist + lo, nc * (int)sizeof(uint16_t));
    unit_copy(g, s.cm, L.cm + lo, nc * (int)sizeof(T));
    for (int k = g.tid; k <= (m.z & 0xffff); k += g.nt) s_roff[k] = ro[k];
}

// Levels above 0: the unit's rows as the sums of the previous level's
// exports (a long list by a warp).  Ends with the group's barrier.
template <typename T, int R, int CG>
__device__ __forceinline__ void unit_sums(const UnitGroup &g, const UnitLevelArgs<T> &L, const T *E,
                                          int u, const UnitSmem<T> &s, int c0) {
    constexpr int V = UnitVec<T, CG>::V, LP = UnitVec<T, CG>::LP;
    const int64_t pos0 = (int64_t)u * L.B;
    const int size = (int)min((int64_t)L.B, L.n - pos0);
    for (int it = g.tid; it < size * LP; it += g.nt) {
        const int p = it / LP, c = (it % LP) * V;
        const int b = L.sptr[pos0 + p], e = L.sptr[pos0 + p + 1];
        T acc[V];
#pragma unroll
        for (int x = 0; x < V; ++x) acc[x] = (T)0;
        if (e - b <= kUnitHeavy) {
            for (int j = b; j < e; ++j) {
                T v[V];
                uld<T, V>(E + (int64_t)j * R + c0 + c, true, v);
#pragma unroll
                for (int x = 0; x < V; ++x) acc[x] += v[x];
            }
        }
        ust<T, V>(s.y + p * CG + c, true, acc);
    }
    g.sync();
    const int lane = g.tid & 31;
    unit_heavy(g, 0, size, [&](int p) { return L.sptr[pos0 + p + 1] - L.sptr[pos0 + p]; }, [&](int p) {
        const int b = L.sptr[pos0 + p], e = L.sptr[pos0 + p + 1];
        for (int c = 0; c < CG; ++c) {
            T acc = (T)0;
            for (int j = b + lane; j < e; j += 32) acc += E[(int64_t)j * R + c0 + c];
            for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
            if (lane == 0) s.y[p * CG + c] = acc;
        }
    });
    g.sync();
}

// Forward rounds and the exports' sums.
template <typename T, int CG>
__device__ __forceinline__ void unit_forward(const UnitGroup &g, const UnitSmem<T> &s, const int4 m,
                                             const uint16_t *s_roff) {
    const int rounds = m.z & 0xffff;
    const bool heavy = m.z >> 16;
    for (int k = 1; k < rounds; ++k) unit_gather<T, CG>(g, s, s_roff[k], s_roff[k + 1], heavy);
    unit_gather<T, CG>(g, s, m.x, m.y, heavy);
}

// The unit's coefficients into shared memory (over the forward lists).
template <typename T>
__device__ __forceinline__ void unit_coef(const UnitGroup &g, const UnitLevelArgs<T> &L, int u,
                                          const int4 m, const UnitSmem<T> &s) {
    unit_copy(g, s.cf, L.coef + (int64_t)u * L.B, m.x * (int)sizeof(typename PackT<T>::V4));
}

// Rows [p0, p1) of a unit from shared memory to their places in W.
template <typename T, int R, int CG>
__device__ __forceinline__ void unit_store(const UnitGroup &g, const UnitSmem<T> &s,
                                           const int32_t *ord, int p0, int p1, T *W, bool al) {
    constexpr int V = UnitVec<T, CG>::V, LP = UnitVec<T, CG>::LP, NB = 4;
    const int end = p1 * LP;
    for (int i0 = p0 * LP + g.tid; i0 < end; i0 += NB * g.nt) {
        int32_t o[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int it = i0 + k * g.nt;
            o[k] = it >= end ? 0 : ord ? ord[it / LP] : it / LP;
        }
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const int it = i0 + k * g.nt;
            if (it >= end) break;
            T v[V];
            uld<T, V>(s.y + it * V, true, v);
            ust<T, V>(W + (int64_t)o[k] * R + (it % LP) * V, al, v);
        }
    }
}

// Backward rounds of a unit in shared memory (x of the survivors and the
// outside vertices is there); ends with the group's barrier.
template <typename T, int CG>
__device__ __forceinline__ void unit_backward(const UnitGroup &g, const UnitSmem<T> &s,
                                              const uint16_t *roff, int rounds) {
    constexpr int V = UnitVec<T, CG>::V, LP = UnitVec<T, CG>::LP;
    for (int k = rounds - 1; k >= 0; --k) {
        const int lo = roff[k], hi = roff[k + 1];
        for (int it = g.tid; it < (hi - lo) * LP; it += g.nt) {
            const int p = lo + it / LP, c = (it % LP) * V;
            const auto cf = s.cf[p];
            const uint32_t nn = unit_nn(cf);
            const int n1 = nn & 0xffff, n2 = nn >> 16;
            T y[V], a[V], b[V];
            uld<T, V>(s.y + p * CG + c, true, y);
            uld<T, V>(s.y + n1 * CG + c, true, a);
#pragma unroll
            for (int x = 0; x < V; ++x) b[x] = (T)0;
            if (n2 != 0xffff) uld<T, V>(s.y + n2 * CG + c, true, b);
#pragma unroll
            for (int x = 0; x < V; ++x) y[x] = cf.x * y[x] + cf.y * a[x];
            if (n2 != 0xffff) {
#pragma unroll
                for (int x = 0; x < V; ++x) y[x] += cf.z * b[x];
            }
            ust<T, V>(s.y + p * CG + c, true, y);
        }
        g.sync();
    }
}

// Solve from B into Y (n x R; B may be Y) by every thread of a cooperative
// grid; false when a barrier wait ran out.  mx accumulates max |x| over what
// this thread wrote.  Ends without a trailing grid barrier.
// A block's thread groups take units side by side (the rounds of one unit
// are a chain of short dependent steps: two to four chains at a time hide
// each other's latency).  A task is a unit with `span` of its column groups:
// all of them when there are units enough for the grid (the lists are staged
// once), one when there are not.  A group takes its tasks of a level in
// order forward and in reverse backward, so the last column group it solved
// is still in shared memory when the backward pass starts, unless the
// block solved a column group of the last level in between (those go to the
// last blocks of the grid).
template <typename T, int R, bool TRACK>
__device__ __forceinline__ bool unit_solve_dev(const UnitArgs<T> &a, unsigned int *bar,
                                               long long budget, int *err, const T *B, T *Y,
                                               unsigned int &epoch, double &mx, T *ys) {
    constexpr int CG = UnitCols<T, R>::CG, NG = UnitCols<T, R>::NG;
    constexpr int TG = UnitCols<T, R>::TG, NT = R / TG;
    constexpr int V = UnitVec<T, CG>::V, LP = UnitVec<T, CG>::LP;
    __shared__ uint16_t s_roff_all[4][kUnitRounds + 2];
    const int G = (int)gridDim.x, me = (int)blockIdx.x;
    const bool al = (((uintptr_t)Y | (uintptr_t)B) & 15) == 0 && (R * sizeof(T)) % 16 == 0;
    const int top = a.nl - 1;
    UnitGroup g;
    int groups = a.groups;   // of whole warps
    while ((int)blockDim.x % (32 * groups)) groups >>= 1;
    g.nt = (int)blockDim.x / groups;
    const int gi = (int)threadIdx.x / g.nt;
    g.tid = (int)threadIdx.x - gi * g.nt;
    g.id = 1 + gi;
    const int GG = G * groups, mg = me + gi * G;
    uint16_t *s_roff = s_roff_all[gi];
    char *gsm = reinterpret_cast<char *>(ys) + (size_t)gi * a.gbytes;
    T tm = (T)0;
    __syncthreads();
    bool kept = false;
    for (int l = 0; l < top; ++l) {
        const UnitLevelArgs<T> &L = a.lv[l];
        const T *E = l > 0 ? a.lv[l - 1].exp : nullptr;
        const int span = L.nu >= GG ? NG : 1, parts = NG / span;
        for (int t = mg; t < L.nu * parts; t += GG) {
            const int u = t / parts, cg0 = (t % parts) * span;
            const int4 m = L.meta[u];
            const int size = (int)min((int64_t)L.B, L.n - (int64_t)u * L.B);
            const int32_t *ord = l == 0 ? L.ord + (int64_t)u * L.B : nullptr;
            const UnitSmem<T> s(gsm, m.y, m.x);
            unit_lists(g, L, u, m, s, s_roff);
            if (l == 0) unit_rows<T, R, CG>(g, s, ord, 0, size, B + cg0 * CG, al);
            cp_async_commit();
            for (int k = 0; k < span; ++k) {
                const int c0 = (cg0 + k) * CG;
                if (l == 0 && k > 0) {
                    unit_rows<T, R, CG>(g, s, ord, 0, size, B + c0, al);
                    cp_async_commit();
                }
                cp_async_wait<0>();
                for (int it = g.tid; it < (m.y - size) * CG; it += g.nt) s.y[size * CG + it] = (T)0;
                if (l == 0) g.sync();
                else unit_sums<T, R, CG>(g, L, E, u, s, c0);
                unit_forward<T, CG>(g, s, m, s_roff);
                for (int it = g.tid; it < (m.y - m.x) * LP; it += g.nt) {
                    const int j = it / LP, c = (it % LP) * V;
                    T v[V];
                    uld<T, V>(s.y + (m.x + j) * CG + c, true, v);
                    ust<T, V>(L.exp + (int64_t)L.edst[m.w + j] * R + c0 + c, true, v);
                }
                if (top == 1 && k + 1 == span && t + GG >= L.nu * parts && me < G - NT) {
                    kept = true;   // stays in shared memory
                    break;
                }
                T *W = l == 0 ? Y : L.V + (int64_t)u * L.B * R;
                // level 0's first round is as it was in B
                const int p0 = l == 0 && (m.z & 0xffff) > 0 ? s_roff[1] : 0;
                unit_store<T, R, CG>(g, s, ord, p0, m.x, W + c0, l == 0 ? al : true);
                g.sync();
            }
        }
        if (!grid_sync(bar, budget, err, epoch)) return false;
    }
    // the last level: one unit, a block per column group
    {
        constexpr int TV = UnitVec<T, TG>::V, TLP = UnitVec<T, TG>::LP;
        const UnitLevelArgs<T> &L = a.lv[top];
        T *W = top > 0 ? L.V : Y;
        const bool wal = top > 0 ? true : al;
        UnitGroup h;
        h.tid = (int)threadIdx.x;
        h.nt = (int)blockDim.x;
        h.id = 0;
        for (int t = G - 1 - me; t < NT; t += G) {
            const int c0 = t * TG;
            const int4 m = L.meta[0];
            const int rounds = m.z & 0xffff;
            const UnitSmem<T> s(ys, m.y, m.x);
            unit_lists(h, L, 0, m, s, s_roff_all[0]);
            if (top == 0) unit_rows<T, R, TG>(h, s, L.ord, 0, m.y, B + c0, al);
            cp_async_commit();
            if (top > 0) unit_sums<T, R, TG>(h, L, a.lv[top - 1].exp, 0, s, c0);
            cp_async_wait<0>();
            h.sync();
            unit_forward<T, TG>(h, s, m, s_roff_all[0]);
            unit_coef(h, L, 0, m, s);
            cp_async_commit();
            if (h.tid < TG) s.y[m.x * TG + h.tid] *= *a.rinv;
            cp_async_wait<0>();
            h.sync();
            unit_backward<T, TG>(h, s, s_roff_all[0], rounds);
            for (int it = h.tid; it < m.y * TLP; it += h.nt) {
                const int p = it / TLP, c = (it % TLP) * TV;
                T v[TV];
                uld<T, TV>(s.y + p * TG + c, true, v);
                ust<T, TV>(W + (int64_t)(top > 0 ? p : L.ord[p]) * R + c0 + c, wal, v);
                if (TRACK) {
#pragma unroll
                    for (int x = 0; x < TV; ++x) tm = fmax(tm, fabs(v[x]));
                }
            }
            h.sync();
        }
    }
    for (int l = top - 1; l >= 0; --l) {
        const UnitLevelArgs<T> &L = a.lv[l];
        const T *X = a.lv[l + 1].V;   // the next level's solution
        const bool wal = l == 0 ? al : true;
        const int span = L.nu >= GG ? NG : 1, parts = NG / span;
        const int ntask = L.nu * parts;
        const int last = mg < ntask ? mg + (ntask - 1 - mg) / GG * GG : -1;
        if (kept) {   // the coefficients do not wait for the last level
            const int u = last / parts;
            const int4 m = L.meta[u];
            const UnitSmem<T> s(gsm, m.y, m.x);
            g.sync();
            unit_coef(g, L, u, m, s);
            cp_async_commit();
        }
        if (!grid_sync(bar, budget, err, epoch)) {
            cp_async_wait<0>();   // the block ends with none of its copies in flight
            return false;
        }
        for (int t = last; t >= 0; t -= GG) {
            const int u = t / parts, cg0 = (t % parts) * span;
            const int4 m = L.meta[u];
            const int rounds = m.z & 0xffff;
            const int size = (int)min((int64_t)L.B, L.n - (int64_t)u * L.B);
            const int32_t *ord = l == 0 ? L.ord + (int64_t)u * L.B : nullptr;
            T *W = l == 0 ? Y : L.V + (int64_t)u * L.B * R;
            const UnitSmem<T> s(gsm, m.y, m.x);
            const bool keep = kept && t == last;
            int p1 = 0;
            if (!keep) {
                const uint16_t *ro = L.roff + (int64_t)u * (kUnitRounds + 2);
                for (int k = g.tid; k <= rounds; k += g.nt) s_roff[k] = ro[k];
                unit_coef(g, L, u, m, s);
                p1 = l == 0 && rounds > 0 ? ro[1] : 0;
            } else {
                p1 = rounds > 0 ? s_roff[1] : 0;
            }
            for (int k = span - 1; k >= 0; --k) {
                const int c0 = (cg0 + k) * CG;
                if (!keep || k + 1 < span) {
                    unit_rows<T, R, CG>(g, s, ord, 0, p1, B + c0, wal);
                    unit_rows<T, R, CG>(g, s, ord, p1, m.x, W + c0, wal);
                    cp_async_commit();
                }
                for (int it = g.tid; it < (m.y - m.x) * LP; it += g.nt) {
                    const int j = it / LP, c = (it % LP) * V;
                    T v[V];
                    uld<T, V>(X + (int64_t)L.epos[m.w + j] * R + c0 + c, true, v);
                    ust<T, V>(s.y + (m.x + j) * CG + c, true, v);
                }
                cp_async_wait<0>();
                g.sync();
                unit_backward<T, CG>(g, s, s_roff, rounds);
                unit_store<T, R, CG>(g, s, ord, 0, size, W + c0, wal);
                if (TRACK) {
                    for (int it = g.tid; it < size * CG; it += g.nt) tm = fmax(tm, fabs(s.y[it]));
                }
                g.sync();
            }
        }
    }
    if (TRACK) mx = fmax(mx, (double)tm);
    return true;
}

}  // namespace grass
