// units.cu -- builds the unit form of a single spanning tree (units.cuh):
// the preorder that visits every vertex's largest subtree last, the units of
// every level with their block-local elimination order and contribution
// lists, and the numeric coefficients.
//
// Why the largest subtree last: a unit is a stretch of B consecutive
// positions, and a vertex survives its unit when it has a child in another
// one.  At a cut between two units those are ancestors of the first
// vertex after the cut whose path there leaves through a child that is not
// the last one, so through a light edge (at most log2 n of them), or the one
// parent whose last child starts there.  With children in any order a long
// path with a late leaf at every vertex would make every vertex of a unit
// survive.
#include "units.cuh"

namespace grass {
namespace {

constexpr int kBuildThreads = 512;

// ---------------------------------------------------------------- preorder

// heavy[p] = max over p's children of (subtree size, smaller id first)
__global__ void k_un_heavy(int64_t n, const int32_t *ein, const int32_t *eout, const int32_t *par,
                           unsigned long long *heavy) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n || ein[v] < 0) return;
    const unsigned long long size = (unsigned long long)(eout[v] - ein[v] + 1) / 2;
    atomicMax(heavy + par[v], size << 32 | (0xffffffffull - (unsigned long long)v));
}

// A vertex's shift against its parent when the heavy child moves behind its
// siblings, placed at the tour's entry (+) and exit (-): the prefix sum at
// the entry is the shift of the whole root path.
__global__ void k_un_shift(int64_t n, int32_t root, const int32_t *ein, const int32_t *eout,
                           const int32_t *par, const int32_t *pre, const unsigned long long *heavy,
                           int64_t *d) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n || ein[v] < 0) return;
    const int32_t p = par[v];
    const int64_t h = (int64_t)(0xffffffffull - (heavy[p] & 0xffffffffull));
    const int64_t hs = (int64_t)(heavy[p] >> 32);
    const int64_t psize = p == root ? n : (eout[p] - ein[p] + 1) / 2;
    int64_t s = 0;
    if (v == h) s = (pre[p] + psize) - (pre[v] + hs);
    else if (pre[v] > pre[h]) s = -hs;
    d[ein[v]] = s;
    d[eout[v]] = -s;
}

__global__ void k_un_pos(int64_t n, const int32_t *ein, const int32_t *pre, const int64_t *d,
                         const int64_t *sum, int32_t *pos, int32_t *vid) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const int64_t e = ein[v];
    const int32_t k = (int32_t)(pre[v] + (e < 0 ? 0 : sum[e] + d[e]));
    pos[v] = k;
    vid[k] = (int32_t)v;
}

__global__ void k_un_level0(int64_t n, const int32_t *vid, const int32_t *pos, const int32_t *par,
                            const int32_t *ein, const double *pw, int32_t *parent, double *w) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int32_t v = vid[k];
    parent[k] = ein[v] < 0 ? -1 : pos[par[v]];
    w[k] = pw[v];
}

// ---------------------------------------------------------------- symbolic, per unit

// pin[p] = 1 for every vertex with a child in another unit (and the root)
__global__ void k_un_cross(int64_t n, int B, const int32_t *parent, uint8_t *pin) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t p = parent[i];
    if (p < 0) pin[i] = 1;
    else if (p / B != i / B) pin[p] = 1;
}

// exclusive block scan of one int per thread; *total = the block's sum
__device__ inline int un_scan(int v, int *total) {
    __shared__ int ws[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int s = lane < nw ? ws[lane] : 0;
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, d);
            if (lane >= d) s += y;
        }
        ws[lane] = s;
    }
    __syncthreads();
    const int before = wid > 0 ? ws[wid - 1] : 0;
    *total = ws[nw - 1];
    __syncthreads();
    return before + x - v;
}

struct UnitBuildArgs {
    int64_t n;
    int B;
    const int32_t *parent;
    const uint8_t *pin;
    const int32_t *vid;      // level 0: vertex id of a position; else null
    int32_t *ord, *lidx;     // unit order -> vertex id / index at this level
    uint32_t *nn;
    int4 *meta;
    uint16_t *roff, *cbeg, *clist;
    int32_t *halo;           // [nu * B] outside vertices of unit u from u * B on
    int32_t *up;             // [n] parent (index at this level) of every survivor
    int32_t *cnt;            // [2 nu] survivors and exports of every unit
    int *most;               // [0] local indices, [1] eliminated, over all units
};

// shared memory of the build: see the carve-up in the kernel
inline size_t unit_build_smem(int B) {
    return (size_t)B * (4 * 4 + 2 + 2 + 2 + 2 + 1 + 1) + (size_t)B * 2 * (4 + 4 + 2 + 2) + 256;
}

// One block contracts one unit (the rules of tree.cu on parent pointers, a
// vertex's children known by their number and the xor of their ids): leaves
// are raked, an independent set of vertices with one child compressed,
// pinned vertices and those hanging from another unit's vertex by a
// compressible chain included until nothing more can go.
__global__ void __launch_bounds__(kBuildThreads, 1) k_unit_build(UnitBuildArgs a) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int B = a.B, u = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int64_t base = (int64_t)u * B;
    const int size = (int)min((int64_t)B, a.n - base);
    int32_t *out = reinterpret_cast<int32_t *>(sm);   // outside parent, or -1
    int32_t *nch = out + B, *xch = nch + B, *par = xch + B;
    int32_t *cnt = par + B, *beg = cnt + 2 * B;       // per local index
    uint16_t *ent = reinterpret_cast<uint16_t *>(beg + 2 * B), *rcv = ent + 2 * B;
    uint16_t *n1 = rcv + 2 * B, *n2 = n1 + B, *pos = n2 + B, *own = pos + B;
    uint8_t *er = reinterpret_cast<uint8_t *>(own + B), *cls = er + B;
    __shared__ int s_best;
    constexpr int kNone = -1, kRoot = -2;
    for (int i = tid; i < size; i += nt) {
        const int32_t p = a.parent[base + i];
        out[i] = -1;
        par[i] = p < 0 ? kRoot : p >= base ? (int)(p - base) : kNone;
        if (p >= 0 && p < base) out[i] = p;
        nch[i] = xch[i] = 0;
        er[i] = 255;
    }
    __syncthreads();
    for (int i = tid; i < size; i += nt)
        if (par[i] >= 0) {
            atomicAdd(nch + par[i], 1);
            atomicXor(xch + par[i], i);
        }
    // number the distinct outside parents, largest first
    int nh = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_best = -1;
        __syncthreads();
        int b = -1;
        for (int i = tid; i < size; i += nt)
            if (par[i] == kNone) b = max(b, out[i]);
        for (int d = 16; d > 0; d >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, d));
        if ((tid & 31) == 0 && b >= 0) atomicMax(&s_best, b);
        __syncthreads();
        b = s_best;
        if (b < 0) break;
        for (int i = tid; i < size; i += nt)
            if (par[i] == kNone && out[i] == b) par[i] = size + nh;
        if (tid == 0) a.halo[base + nh] = b;
        ++nh;
    }
    const int local = size + nh;
    // contraction rounds
    int rounds = 0;
    for (; rounds < kUnitRounds; ++rounds) {
        for (int i = tid; i < size; i += nt) {
            uint8_t c = 0;
            if (er[i] == 255 && !a.pin[base + i] && par[i] >= 0)
                c = nch[i] == 0 ? 1 : nch[i] == 1 ? 2 : 0;
            cls[i] = c;
        }
        __syncthreads();
        int any = 0;
        for (int i = tid; i < size; i += nt) {
            if (cls[i] == 0) continue;
            bool take = cls[i] == 1;
            if (!take) {
                const int p = par[i], c = xch[i];
                take = cls[c] != 1;
                if (take && p < size && cls[p] == 2) take = prio_gt(base + i, base + p, rounds);
                if (take && cls[c] == 2) take = prio_gt(base + i, base + c, rounds);
            }
            if (take) {
                er[i] = (uint8_t)rounds;
                n1[i] = (uint16_t)par[i];
                n2[i] = cls[i] == 1 ? 0xffff : (uint16_t)xch[i];
                any = 1;
            }
        }
        if (!__syncthreads_or(any)) break;
        // a second pass over the chains: the candidates with no chosen
        // neighbour that beat their other such neighbours (0.43 instead of
        // 0.33 of a long chain a round: fewer rounds per solve)
        for (int i = tid; i < size; i += nt) {
            if (cls[i] != 2) continue;
            const int p = par[i], c = xch[i];
            const bool hit = er[i] == rounds || cls[c] == 1 || (p < size && er[p] == rounds) ||
                             er[c] == rounds;
            out[i] = hit ? 0 : 1;
        }
        __syncthreads();
        for (int i = tid; i < size; i += nt) {
            if (cls[i] != 2 || !out[i]) continue;
            const int p = par[i], c = xch[i];
            if (p < size && cls[p] == 2 && out[p] && !prio_gt(base + i, base + p, rounds)) continue;
            if (cls[c] == 2 && out[c] && !prio_gt(base + i, base + c, rounds)) continue;
            er[i] = (uint8_t)rounds;
            n1[i] = (uint16_t)p;
            n2[i] = (uint16_t)c;
        }
        __syncthreads();
        for (int i = tid; i < size; i += nt) {
            if (er[i] != rounds) continue;
            const int p = n1[i];
            if (n2[i] == 0xffff) {
                if (p < size) {
                    atomicSub(nch + p, 1);
                    atomicXor(xch + p, i);
                }
            } else {
                const int c = n2[i];
                par[c] = p;
                if (p < size) atomicXor(xch + p, i ^ c);
            }
        }
        __syncthreads();
    }
    // Order by (round, one or two neighbours, list length, position), the
    // survivors last: a warp's items of a round then run through the same
    // branches and list lengths (an FP64 instruction occupies its pipe for
    // the whole warp, however few lanes are on).  A bitonic sort of keys.
    for (int j = tid; j < local; j += nt) cnt[j] = 0;
    __syncthreads();
    for (int i = tid; i < size; i += nt) {
        if (er[i] == 255) continue;
        atomicAdd(cnt + n1[i], 1);
        if (n2[i] != 0xffff) atomicAdd(cnt + n2[i], 1);
    }
    __syncthreads();
    int P = 1;
    while (P < size) P <<= 1;
    for (int i = tid; i < P; i += nt) {
        uint32_t key = 0xffffffffu;
        if (i < size) {
            const uint32_t r = er[i];
            key = r << 24 | (r == 255 ? 0u : (n2[i] != 0xffff ? 1u : 0u) << 23 |
                                                 (uint32_t)min(cnt[i], 127) << 16) | (uint32_t)i;
        }
        beg[i] = (int32_t)key;
    }
    __syncthreads();
    for (int k = 2; k <= P; k <<= 1)
        for (int d = k >> 1; d > 0; d >>= 1) {
            for (int i = tid; i < P; i += nt) {
                const int x = i ^ d;
                if (x <= i) continue;
                const uint32_t a0 = (uint32_t)beg[i], a1 = (uint32_t)beg[x];
                if ((a0 > a1) == ((i & k) == 0)) {
                    beg[i] = (int32_t)a1;
                    beg[x] = (int32_t)a0;
                }
            }
            __syncthreads();
        }
    int nel = size;
    uint16_t *ro = a.roff + (int64_t)u * (kUnitRounds + 2);
    __shared__ int s_nel;
    if (tid == 0) s_nel = size;
    __syncthreads();
    for (int p = tid; p < size; p += nt) {
        const uint32_t key = (uint32_t)beg[p];
        const int i = (int)(key & 0xffffu), r = (int)(key >> 24);
        pos[i] = (uint16_t)p;
        own[p] = (uint16_t)i;
        if (p == 0 || (int)((uint32_t)beg[p - 1] >> 24) != r) {
            if (r == 255) s_nel = p;
            else ro[r] = (uint16_t)p;
        }
    }
    __syncthreads();
    nel = s_nel;
    if (tid == 0) ro[rounds] = (uint16_t)nel;
    auto ref = [&](int x) { return x < size ? (int)pos[x] : x; };
    for (int p = tid; p < size; p += nt) {
        const int i = own[p];
        a.lidx[base + p] = (int32_t)(base + i);
        a.ord[base + p] = a.vid ? a.vid[base + i] : (int32_t)(base + i);
        if (p < nel) {
            const uint32_t x = (uint32_t)ref(n1[i]);
            const uint32_t y = n2[i] == 0xffff ? 0xffffu : (uint32_t)ref(n2[i]);
            a.nn[base + p] = x | y << 16;
        } else {
            const int q = par[i];
            a.up[base + i] = q == kRoot ? -1
                             : q < size ? (int32_t)(base + q)
                                        : a.halo[base + (q - size)];
        }
    }
    // contribution lists, sorted by contributor
    for (int j = tid; j < local; j += nt) cnt[j] = 0;
    __syncthreads();
    for (int p = tid; p < nel; p += nt) {
        const int i = own[p];
        atomicAdd(cnt + ref(n1[i]), 1);
        if (n2[i] != 0xffff) atomicAdd(cnt + ref(n2[i]), 1);
    }
    __syncthreads();
    uint16_t *cb = a.cbeg + (int64_t)u * unit_stride(B);
    int tot = 0;
    for (int j0 = 0; j0 < local; j0 += nt) {
        const int j = j0 + tid;
        int t;
        const int at = tot + un_scan(j < local ? cnt[j] : 0, &t);
        if (j < local) {
            beg[j] = at;
            cb[j] = (uint16_t)at;
        }
        tot += t;
    }
    __syncthreads();
    if (tid == 0) cb[local] = (uint16_t)tot;
    for (int j = tid; j < local; j += nt) cnt[j] = beg[j];
    __syncthreads();
    for (int p = tid; p < nel; p += nt) {
        const int i = own[p];
        const int r1 = ref(n1[i]);
        int k = atomicAdd(cnt + r1, 1);
        ent[k] = (uint16_t)(2 * p);
        rcv[k] = (uint16_t)r1;
        if (n2[i] != 0xffff) {
            const int r2 = ref(n2[i]);
            k = atomicAdd(cnt + r2, 1);
            ent[k] = (uint16_t)(2 * p + 1);
            rcv[k] = (uint16_t)r2;
        }
    }
    __syncthreads();
    uint16_t *cl = a.clist + (int64_t)u * unit_stride(B);
    int heavy = 0;
    for (int k = tid; k < tot; k += nt) {
        const int r = rcv[k], b = beg[r], e = cnt[r];
        const uint16_t x = ent[k];
        int rank = 0;
        for (int j = b; j < e; ++j) rank += ent[j] < x;
        cl[b + rank] = x;
        heavy |= e - b > kUnitHeavy;
    }
    heavy = __syncthreads_or(heavy);
    if (tid == 0) {
        a.meta[u] = make_int4(nel, local, rounds | (heavy ? 1 << 16 : 0), 0);
        a.cnt[2 * u] = size - nel;
        a.cnt[2 * u + 1] = local - nel;
        atomicMax(a.most, local);
        atomicMax(a.most + 1, nel);
    }
}

// One block: exclusive sums of the units' survivors and exports; totals to
// tot[0], tot[1], the first export into meta.
__global__ void k_un_offsets(int nu, const int32_t *cnt, int32_t *soff, int4 *meta, int *tot) {
    int rs = 0, re = 0;
    for (int u0 = 0; u0 < nu; u0 += blockDim.x) {
        const int u = u0 + threadIdx.x;
        int t0, t1;
        const int s = un_scan(u < nu ? cnt[2 * u] : 0, &t0);
        const int e = un_scan(u < nu ? cnt[2 * u + 1] : 0, &t1);
        if (u < nu) {
            soff[u] = rs + s;
            meta[u].w = re + e;
        }
        rs += t0;
        re += t1;
    }
    if (threadIdx.x == 0) {
        tot[0] = rs;
        tot[1] = re;
    }
}

// next level's index of every survivor
__global__ void k_un_core(int64_t n, int B, const int4 *meta, const int32_t *lidx,
                          const int32_t *soff, int32_t *core) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int u = (int)(k / B), p = (int)(k % B);
    if (p >= meta[u].x) core[lidx[k]] = soff[u] + p - meta[u].x;
}

// exports' indices and the next level's parents
__global__ void k_un_link(int64_t n, int B, int nu, const int4 *meta, const int32_t *lidx,
                          const int32_t *halo, const int32_t *up, const int32_t *core,
                          int32_t *ecore, int32_t *next_parent, int32_t *scnt) {
    const int u = blockIdx.x;
    const int4 m = meta[u];
    const int64_t base = (int64_t)u * B;
    const int size = (int)min((int64_t)B, n - base);
    for (int j = m.x + threadIdx.x; j < m.y; j += blockDim.x) {
        const int32_t i = j < size ? lidx[base + j] : halo[base + j - size];
        const int32_t c = core[i];
        ecore[m.w + j - m.x] = c;
        atomicAdd(scnt + c, 1);
        if (j < size) next_parent[c] = up[i] < 0 ? -1 : core[up[i]];
    }
}

// Per position of a level: how many of the previous level's exports make it
// up, their exclusive sums and cursors.  One block, 1,024 entries a step: a few
// thousand in a tree's own levels, up to n / 4 for a core.
__global__ void k_un_sptr(int n1, const int32_t *lidx, const int32_t *scnt, int32_t *sptr,
                          int32_t *cur, int32_t *pos_of) {
    int run = 0;
    for (int p0 = 0; p0 < n1; p0 += blockDim.x) {
        const int p = p0 + threadIdx.x;
        const int i = p < n1 && lidx ? lidx[p] : p;
        int t;
        const int s = run + un_scan(p < n1 ? scnt[i] : 0, &t);
        if (p < n1) {
            sptr[p] = cur[p] = s;
            pos_of[i] = p;
        }
        run += t;
    }
    if (threadIdx.x == 0) sptr[n1] = run;
}

__global__ void k_un_sfill(int64_t nexp, const int32_t *ecore, const int32_t *pos_of, int32_t *cur,
                           int32_t *raw, int32_t *epos) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nexp) return;
    const int32_t p = pos_of[ecore[k]];
    epos[k] = p;
    raw[atomicAdd(cur + p, 1)] = (int32_t)k;
}

// rows in export order within a position
__global__ void k_un_ssort(int64_t nexp, const int32_t *epos, const int32_t *sptr,
                           const int32_t *raw, int32_t *edst) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nexp) return;
    const int32_t x = raw[k], p = epos[x];
    int rank = 0;
    for (int32_t j = sptr[p]; j < sptr[p + 1]; ++j) rank += raw[j] < x;
    edst[x] = sptr[p] + rank;
}

// ---------------------------------------------------------------- numeric

struct UnitFactorArgs {
    int64_t n;
    int B;
    const int4 *meta;
    const uint16_t *roff, *cbeg, *clist;   // clist: contributor * 2 + side
    uint16_t *cpos;                        // contributor alone, in the same order
    double *m64;                           // its multiplier
    float *m32;
    const uint32_t *nn;
    const int32_t *lidx, *ord;
    const double *w;               // [n] weight to the parent
    const double *D;               // level 0: [vertices] diagonal load, or null (L_T alone)
    const double *dexp;            // levels >= 1: the previous level's load exports, or null
    const int32_t *sptr;
    const int32_t *ecore, *edst;
    double *next_w, *dout;         // next level's weights, this level's load exports
    Dbl4 *c64;
    float4 *c32;
    double *rinv64;                // the last level: 1 / pivot of the root
    float *rinv32;
    int last;
};

inline size_t unit_factor_smem(int local, int elim) {
    return sizeof(double) * (2 * (size_t)local + 2 * (size_t)elim) + 64;
}

// Round by round the pivots d = load + weights, the coefficients and the
// series weights; loads gathered like a forward solve.  FP64.
__global__ void __launch_bounds__(kBuildThreads, 1) k_unit_factor(UnitFactorArgs a) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int B = a.B, u = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int64_t base = (int64_t)u * B;
    const int size = (int)min((int64_t)B, a.n - base);
    const int4 m = a.meta[u];
    double *w = reinterpret_cast<double *>(sm), *dp = w + m.y, *b1 = dp + m.y, *b2 = b1 + m.x;
    const uint16_t *ro = a.roff + (int64_t)u * (kUnitRounds + 2);
    const uint16_t *cb = a.cbeg + (int64_t)u * unit_stride(B), *cl = a.clist + (int64_t)u * unit_stride(B);
    const bool load = a.D || a.dexp;
    for (int p = tid; p < m.y; p += nt) {
        double d = 0.0;
        if (p < size) {
            const int32_t i = a.lidx[base + p];
            w[p] = a.w[i];
            if (a.D) d = a.D[a.ord[base + p]];
            else if (a.dexp)
                for (int32_t j = a.sptr[base + p]; j < a.sptr[base + p + 1]; ++j) d += a.dexp[j];
        }
        dp[p] = d;
    }
    __syncthreads();
    auto gather = [&](int p) {
        double d = dp[p];
        for (int j = cb[p]; j < cb[p + 1]; ++j) {
            const int c = cl[j], v = c >> 1;
            d += ((c & 1) ? b2[v] : b1[v]) * dp[v];
        }
        dp[p] = d;
        return d;
    };
    const int rounds = m.z & 0xffff;
    for (int k = 0; k < rounds; ++k) {
        for (int p = ro[k] + tid; p < ro[k + 1]; p += nt) {
            const double load_p = load ? gather(p) : 0.0;
            const uint32_t nn = a.nn[base + p];
            const int c = nn >> 16;
            const double w1 = w[p], w2 = c != 0xffff ? w[c] : 0.0;
            const double d = load_p + w1 + w2;
            const Dbl4 q{1.0 / d, w1 / d, w2 / d, __longlong_as_double((long long)nn)};
            b1[p] = q.y;
            b2[p] = q.z;
            if (c != 0xffff) w[c] = w1 * w2 / d;
            a.c64[base + p] = q;
            a.c32[base + p] = make_float4((float)q.x, (float)q.y, (float)q.z, __uint_as_float(nn));
        }
        __syncthreads();
    }
    for (int j = tid; j < cb[m.y]; j += nt) {
        const int c = cl[j];
        const double x = (c & 1) ? b2[c >> 1] : b1[c >> 1];
        a.cpos[(int64_t)u * unit_stride(B) + j] = (uint16_t)(c >> 1);
        a.m64[(int64_t)u * unit_stride(B) + j] = x;
        a.m32[(int64_t)u * unit_stride(B) + j] = (float)x;
    }
    for (int j = m.x + tid; j < m.y; j += nt) {
        const double d = load ? gather(j) : 0.0;
        if (a.last) {
            const double r = d > 0.0 ? 1.0 / d : 0.0;   // no load: grounded, x = 0
            *a.rinv64 = r;
            *a.rinv32 = (float)r;
        } else {
            a.dout[a.edst[m.w + j - m.x]] = d;
            if (j < size) a.next_w[a.ecore[m.w + j - m.x]] = w[j];
        }
    }
}

int unit_size(int64_t n, int sms) {
    // as few units per SM as shared memory allows, of equal size
    const int64_t waves = cdiv(n, (int64_t)sms * kUnitMax);
    return (int)std::max<int64_t>(kUnitMin, cdiv(n, (int64_t)sms * waves));
}

}  // namespace

void unit_group(grass_ctx_t ctx, UnitTree &U, UnitLevel &P, int64_t n1, const int32_t *lidx,
                const int32_t *scnt, Arena &tmp, int32_t *sptr) {
    P.epos = U.arena.get<int32_t>(P.nexp);
    P.edst = U.arena.get<int32_t>(P.nexp);
    auto *cur = tmp.get<int32_t>(n1);
    auto *pos_of = tmp.get<int32_t>(n1);
    auto *raw = tmp.get<int32_t>(P.nexp);
    launch(ctx, k_un_sptr, 1, 1024, 0, (int)n1, lidx, scnt, sptr, cur, pos_of);
    launch(ctx, k_un_sfill, cdiv(P.nexp, kBlock), kBlock, 0, P.nexp, (const int32_t *)P.ecore,
           (const int32_t *)pos_of, cur, raw, P.epos);
    launch(ctx, k_un_ssort, cdiv(P.nexp, kBlock), kBlock, 0, P.nexp, (const int32_t *)P.epos,
           (const int32_t *)sptr, (const int32_t *)raw, P.edst);
}

bool unit_levels(grass_ctx_t ctx, int64_t n, int32_t *parent, const int32_t *vid,
                 const uint8_t *pin_in, Arena &tmp, UnitTree &U, int32_t *core, int32_t **scnt_out,
                 int64_t *n_next) {
    GCK(cudaFuncSetAttribute((const void *)k_unit_build, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)unit_build_smem(kUnitTop)));
    GCK(cudaFuncSetAttribute((const void *)k_unit_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kTailSmem));
    auto *up = tmp.get<int32_t>(n);
    auto *halo = tmp.get<int32_t>(n + kUnitTop);
    auto *pin = tmp.get<uint8_t>(n);
    auto *tot = tmp.get<int>(8);
    int64_t nl = n;
    int32_t *scnt = nullptr;
    U.lv.clear();
    U.built = false;
    U.open = pin_in != nullptr;
    for (int l = 0; l < kUnitLevels; ++l) {
        U.lv.emplace_back();
        UnitLevel &L = U.lv.back();
        L.n = nl;
        L.B = nl <= kUnitTop && !U.open ? (int)nl : unit_size(nl, ctx->num_sms);
        L.nu = (int)cdiv(nl, L.B);
        const int B = L.B, nu = L.nu;
        L.ord = U.arena.get<int32_t>(nl);
        L.lidx = U.arena.get<int32_t>(nl);
        L.nn = U.arena.get<uint32_t>(nl);
        L.meta = U.arena.get<int4>(nu);
        L.roff = U.arena.get<uint16_t>((size_t)nu * (kUnitRounds + 2));
        L.cbeg = U.arena.get<uint16_t>((size_t)nu * unit_stride(B));
        L.clist = U.arena.get<uint16_t>((size_t)nu * unit_stride(B));
        L.cpos = U.arena.get<uint16_t>((size_t)nu * unit_stride(B));
        auto *cnt = tmp.get<int32_t>(2 * (size_t)nu);
        auto *soff = tmp.get<int32_t>(nu);
        if (pin_in) copy_d(ctx, pin, pin_in, nl);
        else memset_d(ctx, pin, 0, nl);
        memset_d(ctx, tot, 0, 8 * sizeof(int));
        launch(ctx, k_un_cross, cdiv(nl, kBlock), kBlock, 0, nl, B, (const int32_t *)parent, pin);
        UnitBuildArgs a{nl, B, parent, pin, l == 0 ? vid : nullptr, L.ord, L.lidx, L.nn, L.meta,
                        L.roff, L.cbeg, L.clist, halo, up, cnt, tot + 2};
        launch(ctx, k_unit_build, nu, kBuildThreads, unit_build_smem(B), a);
        launch(ctx, k_un_offsets, 1, 1024, 0, nu, (const int32_t *)cnt, soff, L.meta, tot);
        if (l > 0) {
            L.sptr = U.arena.get<int32_t>(nl + 1);
            unit_group(ctx, U, U.lv[l - 1], nl, L.lidx, scnt, tmp, L.sptr);
        }
        int h[4];
        d2h(ctx, h, tot, sizeof(h));
        const int64_t n1 = h[0];
        L.nexp = h[1];
        L.local = h[2];
        L.elim = h[3];
        if (nu == 1 && !U.open) {
            if (n1 != 1) return false;   // the round limit: keep the elimination rounds
            U.built = true;
            break;
        }
        // the widest column groups of a unit must fit shared memory
        if (n1 > nl / 2 ||
            UnitSmem<double>::lists(L.local, L.elim) + UnitSmem<double>::rows(L.local, 8) > kTailSmem)
            return false;
        if (!U.open) L.exp = U.arena.get<char>((size_t)L.nexp * 32 * sizeof(double));
        L.dexp = U.arena.get<double>(L.nexp);
        L.ecore = U.arena.get<int32_t>(L.nexp);
        scnt = tmp.get<int32_t>(n1);
        memset_d(ctx, scnt, 0, n1 * sizeof(int32_t));
        launch(ctx, k_un_core, cdiv(nl, kBlock), kBlock, 0, nl, B, (const int4 *)L.meta,
               (const int32_t *)L.lidx, (const int32_t *)soff, core);
        launch(ctx, k_un_link, nu, 128, 0, nl, B, nu, (const int4 *)L.meta, (const int32_t *)L.lidx,
               (const int32_t *)halo, (const int32_t *)up, (const int32_t *)core, L.ecore, parent,
               scnt);
        nl = n1;
        if (U.open) {
            U.built = true;
            break;
        }
    }
    if (!U.built) return false;
    for (size_t l = 1; l < U.lv.size(); ++l) {
        UnitLevel &L = U.lv[l];
        L.V = U.arena.get<char>((size_t)L.n * 32 * sizeof(double));
        L.w = U.arena.get<double>(L.n);
    }
    *scnt_out = scnt;
    *n_next = nl;
    return true;
}

bool unit_build(grass_ctx_t ctx, grass_tree_t T, UnitTree &U) {
    const EulerTour &E = T->euler;
    const int64_t n = T->g.n;
    U.built = false;
    if (!E.built || T->batch || T->nroots != 1 || ctx->num_sms <= 0 || n < 2) return false;
    U.arena.chunk_min = (size_t)n * 52 + ((size_t)1 << 20);
    Arena &tmp = ctx->build_tmp;
    // preorder with the heavy child last
    auto *heavy = tmp.get<unsigned long long>(n);
    auto *shift = tmp.get<int64_t>(E.L + 1);
    auto *sum = tmp.get<int64_t>(E.L + 1);
    auto *parent = tmp.get<int32_t>(n);
    auto *core = tmp.get<int32_t>(n);
    U.pos = U.arena.get<int32_t>(n);
    U.vid = U.arena.get<int32_t>(n);
    U.parent = U.arena.get<int32_t>(n);
    U.w0 = U.arena.get<double>(n);
    memset_d(ctx, heavy, 0, n * sizeof(unsigned long long));
    launch(ctx, k_un_heavy, cdiv(n, kBlock), kBlock, 0, n, (const int32_t *)E.ein.p,
           (const int32_t *)E.eout.p, (const int32_t *)E.par.p, heavy);
    launch(ctx, k_un_shift, cdiv(n, kBlock), kBlock, 0, n, T->ground, (const int32_t *)E.ein.p,
           (const int32_t *)E.eout.p, (const int32_t *)E.par.p, (const int32_t *)E.pre.p,
           (const unsigned long long *)heavy, shift);
    scan_i64(ctx, shift, sum, E.L, nullptr);
    launch(ctx, k_un_pos, cdiv(n, kBlock), kBlock, 0, n, (const int32_t *)E.ein.p,
           (const int32_t *)E.pre.p, (const int64_t *)shift, (const int64_t *)sum, U.pos, U.vid);
    launch(ctx, k_un_level0, cdiv(n, kBlock), kBlock, 0, n, (const int32_t *)U.vid,
           (const int32_t *)U.pos, (const int32_t *)E.par.p, (const int32_t *)E.ein.p,
           (const double *)E.pw.p, U.parent, U.w0);
    copy_d(ctx, parent, U.parent, n * sizeof(int32_t));
    int32_t *scnt = nullptr;
    int64_t n1 = 0;
    if (!unit_levels(ctx, n, parent, U.vid, nullptr, tmp, U, core, &scnt, &n1)) return false;
    return true;
}

void unit_factor(grass_ctx_t ctx, const UnitTree &U, const double *D, UnitFactor &f,
                 double *next_w) {
    f.arena.chunk_min = (size_t)U.lv[0].n * 76 + ((size_t)1 << 16);
    f.arena.reset();
    f.c64.clear();
    f.c32.clear();
    f.m64.clear();
    f.m32.clear();
    f.rinv64 = f.arena.get<double>(1);
    f.rinv32 = f.arena.get<float>(1);
    for (size_t l = 0; l < U.lv.size(); ++l) {
        const UnitLevel &L = U.lv[l];
        f.c64.push_back(f.arena.get<Dbl4>(L.n));
        f.c32.push_back(f.arena.get<float4>(L.n));
        f.m64.push_back(f.arena.get<double>((size_t)L.nu * unit_stride(L.B)));
        f.m32.push_back(f.arena.get<float>((size_t)L.nu * unit_stride(L.B)));
        const bool end = l + 1 == U.lv.size(), last = end && !U.open;
        UnitFactorArgs a{L.n, L.B, L.meta, L.roff, L.cbeg, L.clist, L.cpos, f.m64[l], f.m32[l], L.nn, L.lidx, L.ord,
                         l == 0 ? U.w0 : L.w, l == 0 ? D : nullptr,
                         l > 0 && D ? U.lv[l - 1].dexp : nullptr, L.sptr, L.ecore, L.edst,
                         end ? next_w : U.lv[l + 1].w, L.dexp, f.c64[l], f.c32[l], f.rinv64,
                         f.rinv32, last ? 1 : 0};
        launch(ctx, k_unit_factor, L.nu, kBuildThreads, unit_factor_smem(L.local, L.elim), a);
    }
}

}  // namespace grass
