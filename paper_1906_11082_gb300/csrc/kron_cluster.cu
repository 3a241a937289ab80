// Float semi-iteration steps on clusters of four rows (CHEB, CHEB_FILT).
//
// One step x_{k+1} = x_{k-1} + om (x_k - x_{k-1} + D^-1 (w - A x_k) / theta) of
// A = M_rho (x) I_3 (or the pressure matrix) gathers every stored neighbour's
// record of R x b floats: row by row 27 records of 384 bytes per row at
// b = 32, 4 GB through L1 per step of the 1.15M-dof planet, bound by the
// latency of those gathers and the instructions around them (DRAM at 28%, L2
// at 52%, no unit saturated). Rows of a P2 mesh share neighbours: four rows
// chosen inside a window of 64 (Morton) rows to share most store half as many
// distinct columns as entries (0.50 on the planet; four consecutive rows
// 0.59). A lane takes four columns of all R components of such a cluster, so
// one 16-byte gather serves four rows; twice the multiply-adds (packed
// f32x2), half the gathered bytes.
//
// Layout: S lane groups of L = (columns / 4) lanes split a cluster's entries,
// U = 3 entries' records are in flight per lane, entries are padded to a
// multiple of six (S U for two groups; four groups skip what lies past the end).
// Warps walk clusters with a grid stride (one wave), the next cluster's header
// and first columns being fetched during the current one, so no chain of
// dependent loads is exposed between clusters; the epilogue's streams are
// prefetched to L2 when the cluster begins. 128 registers, four CTAs of four
// warps per SM: at 96 registers and five CTAs the compiler spills and the step
// takes 345 us; keeping the loads rolling over trips and clusters 272 us;
// staging tiles of 20 rows in shared memory 439 us (the copies and the tile's
// serial phases), per-thread cp.async rings 349 us.
//
// Per step, 1.15M dof, before (one row per warp, 16-byte lane groups) and now:
// b = 32: 298 -> 239 us, pressure rows (82k) 46 -> 23 us in a chain of steps (34
// us with cold caches). 199k dof: b = 16 55 -> 23 us, b = 64 199 -> 89 us (were
// per-lane scalar gathers). The clusters are built on the host at the first
// float or mixed call: with the float copies 11 ms at 199k dof, 52 ms at 1.15M.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <new>
#include <vector>

#include "kernels.h"
#include "nm_internal.h"
#include "dependent.cuh"

namespace nm {

namespace {

constexpr int kThreads = 128;
constexpr int kMaxRows = 64;         // consecutive rows a cluster is chosen from
constexpr int kPad = 6;              // a cluster's entries are padded to a multiple of this (2 groups x 3)

__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

struct F4 {
    unsigned long long lo, hi;
};
// NC: by the read-only path
template <bool NC>
__device__ __forceinline__ F4 ldg4(const float* p) {
    if constexpr (NC) {
        F4 r;
        asm("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(r.lo), "=l"(r.hi) : "l"(p));
        return r;
    } else {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
        return {t.x, t.y};
    }
}
__device__ __forceinline__ float4 f4(const F4& v) {
    const float2 a = unpack2(v.lo), b = unpack2(v.hi);
    return make_float4(a.x, a.y, b.x, b.y);
}

}  // namespace

// L: 16-byte columns of a column group (grid y); DENSE: the gathered block is
// exactly one group wide. Lane (cluster cw of the warp, split sp, column q).
template <int R, int L, int MODE, int S, int U, bool DENSE, bool DEP, int MINB>
__global__ void __launch_bounds__(kThreads, MINB) kron_cluster_kernel(const KronArgs<float> a) {
    constexpr int LC = S * L;                 // lanes of a cluster
    constexpr int CW = 32 / LC;               // clusters of a warp
    constexpr int RPL = 4 / S;                // rows a lane finishes
    const int grp = DENSE ? 0 : blockIdx.y;
    const int c0 = grp * 4 * L;               // first column of the group
    const int nq = DENSE ? L : min(L, a.b / 4 - grp * L);
    const int64_t ld = DENSE ? 4 * L : a.ldx;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cw = lane / LC, rl = lane - cw * LC, sp = rl / L, q = rl - sp * L;
    const int qc = DENSE ? q : min(q, nq - 1);
    const float* const X = a.X + c0 + 4 * qc;
    const int stride = gridDim.x * (kThreads / 32) * CW;
    int cl = (blockIdx.x * (kThreads / 32) + warp) * CW + (cw < CW ? cw : 0);
    const int last = a.cl.n - 1;
    // header and first columns of the next cluster are fetched during this one
    int e = __ldg(a.cl.ptr + min(cl, last)), e1 = __ldg(a.cl.ptr + min(cl, last) + 1);
    int4 rows = __ldg(a.cl.rows + min(cl, last));
    int c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = __ldg(a.cl.col + min(e + sp + u * S, e1 - 1));
    // DEP: started while the previous step drains. What is loaded above is
    // matrix data; the blocks are read after this wait, and by plain loads.
    if constexpr (DEP) dep_sync();
    for (int first = (blockIdx.x * (kThreads / 32) + warp) * CW; first <= last; first += stride) {
        const bool on = cw < CW && cl <= last && q < nq;
        const int cn = min(cl + stride, last);
        const int en = __ldg(a.cl.ptr + cn), en1 = __ldg(a.cl.ptr + cn + 1);
        const int4 rowsn = __ldg(a.cl.rows + cn);
        F4 acc[4][R];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int k = 0; k < R; ++k) acc[r][k].lo = acc[r][k].hi = 0ull;
        const float4* pv = a.cl.val + e + sp;
        const int* pc = a.cl.col + e + sp;
        int left = e1 - e - sp;               // entries from this lane group's first on
        // the epilogue's streams, on their way to L2 during the gather
        if (on && (q & 7) == 0) {
#pragma unroll
            for (int i = 0; i < RPL; ++i) {
                const int f = sp * RPL + i, row = f == 0 ? rows.x : f == 1 ? rows.y : f == 2 ? rows.z : rows.w;
                if (row >= 0) {
#pragma unroll
                    for (int k = 0; k < R; ++k) {
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.W + ((int64_t)R * row + k) * a.ldw + c0));
                        if (a.Xp) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.Xp + ((int64_t)R * row + k) * a.ldp + c0));
                    }
                }
            }
        }
        while (left > 0) {
            F4 x[U][R];
            float4 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float* p = X + c[u] * (R * ld);
#pragma unroll
                for (int k = 0; k < R; ++k) x[u][k] = ldg4<!DEP>(p + k * ld);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (S * U == kPad || u * S < left)
                    v[u] = __ldg(pv + u * S);
                else
                    v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            pv += U * S;
            pc += U * S;
            left -= U * S;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (S * U == kPad ? left > 0 : u * S < left) c[u] = __ldg(pc + u * S);
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float vr = r == 0 ? v[u].x : r == 1 ? v[u].y : r == 2 ? v[u].z : v[u].w;
                    const unsigned long long vv = pack2(vr, vr);
#pragma unroll
                    for (int k = 0; k < R; ++k) {
                        fma2(acc[r][k].lo, vv, x[u][k].lo);
                        fma2(acc[r][k].hi, vv, x[u][k].hi);
                    }
                }
        }
        int row[RPL];
        float pd[RPL];
        float4 pw[RPL][R], pp[RPL][R];
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
            const int f = sp * RPL + i;
            row[i] = f == 0 ? rows.x : f == 1 ? rows.y : f == 2 ? rows.z : rows.w;
            if (!on) row[i] = -1;
            pd[i] = 0.f;
#pragma unroll
            for (int k = 0; k < R; ++k) pw[i][k] = pp[i][k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row[i] >= 0) {
                pd[i] = __ldg(a.dinv + row[i]);
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const int64_t r = (int64_t)R * row[i] + k;
                    pw[i][k] = __ldcs(reinterpret_cast<const float4*>(a.W + r * a.ldw + c0 + 4 * q));
                    if (a.Xp) pp[i][k] = __ldcs(reinterpret_cast<const float4*>(a.Xp + r * a.ldp + c0 + 4 * q));
                }
            }
        }
        e = en;
        e1 = en1;
        rows = rowsn;
        cl += stride;
#pragma unroll
        for (int u = 0; u < U; ++u) c[u] = __ldg(a.cl.col + min(e + sp + u * S, e1 - 1));
        // sum the splits; a lane keeps the rows sp * RPL .. + RPL - 1
        float4 sum[RPL][R];
        if constexpr (S == 1) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int k = 0; k < R; ++k) sum[i][k] = f4(acc[i][k]);
        } else {
            const int up = S == 2 ? sp : sp >> 1;                 // upper pair of rows
            const int peer = lane + (up ? -1 : 1) * (S == 2 ? L : 2 * L);
            float4 half[2][R];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const float4 mine = f4(up ? acc[2 + i][k] : acc[i][k]), give = f4(up ? acc[i][k] : acc[2 + i][k]);
                    half[i][k].x = mine.x + __shfl_sync(0xffffffffu, give.x, peer);
                    half[i][k].y = mine.y + __shfl_sync(0xffffffffu, give.y, peer);
                    half[i][k].z = mine.z + __shfl_sync(0xffffffffu, give.z, peer);
                    half[i][k].w = mine.w + __shfl_sync(0xffffffffu, give.w, peer);
                }
            if constexpr (S == 2) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int k = 0; k < R; ++k) sum[i][k] = half[i][k];
            } else {
                const int odd = sp & 1;
                const int peer1 = lane + (odd ? -L : L);
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const float4 mine = odd ? half[1][k] : half[0][k], give = odd ? half[0][k] : half[1][k];
                    sum[0][k].x = mine.x + __shfl_sync(0xffffffffu, give.x, peer1);
                    sum[0][k].y = mine.y + __shfl_sync(0xffffffffu, give.y, peer1);
                    sum[0][k].z = mine.z + __shfl_sync(0xffffffffu, give.z, peer1);
                    sum[0][k].w = mine.w + __shfl_sync(0xffffffffu, give.w, peer1);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
            if (row[i] < 0) continue;
            const float dd = pd[i] * a.inv_theta;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const float4* px = reinterpret_cast<const float4*>(X + ((int64_t)R * row[i] + k) * ld);
                const float4 xk = DEP ? *px : __ldg(px);
                const float4 xp = pp[i][k], w = pw[i][k];
                float4 sm = sum[i][k];
                // a non-finite record times a zero value of another row: the row's own entries decide
                const float t = sm.x + sm.y + sm.z + sm.w;
                if (t != t) {
                    sm = make_float4(0.f, 0.f, 0.f, 0.f);
                    for (int j = __ldg(a.rowptr + row[i]); j < __ldg(a.rowptr + row[i] + 1); ++j) {
                        const float vj = __ldg(a.val + j);
                        const float4 xj = f4(ldg4<!DEP>(X + ((int64_t)R * __ldg(a.col + j) + k) * ld));
                        sm.x = fmaf(vj, xj.x, sm.x);
                        sm.y = fmaf(vj, xj.y, sm.y);
                        sm.z = fmaf(vj, xj.z, sm.z);
                        sm.w = fmaf(vj, xj.w, sm.w);
                    }
                }
                float4 xn;
                xn.x = xp.x + a.om * (xk.x - xp.x + dd * (w.x - sm.x));
                xn.y = xp.y + a.om * (xk.y - xp.y + dd * (w.y - sm.y));
                xn.z = xp.z + a.om * (xk.z - xp.z + dd * (w.z - sm.z));
                xn.w = xp.w + a.om * (xk.w - xp.w + dd * (w.w - sm.w));
                const int64_t r = (int64_t)R * row[i] + k;
                const int cc = c0 + 4 * q;
                if constexpr (MODE == KRON_CHEB) {
                    *reinterpret_cast<float4*>(a.Xn + r * a.ldn + cc) = xn;
                } else {   // the outer Chebyshev update on x_{k_M}
                    const float4 tk = *reinterpret_cast<const float4*>(a.Tk + r * a.ldtk + cc);
                    float4 tp = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (a.Tp) tp = *reinterpret_cast<const float4*>(a.Tp + r * a.ldtp + cc);
                    float4 tn;
                    tn.x = a.a1 * (xn.x - a.cshift * tk.x) - a.a2 * tp.x;
                    tn.y = a.a1 * (xn.y - a.cshift * tk.y) - a.a2 * tp.y;
                    tn.z = a.a1 * (xn.z - a.cshift * tk.z) - a.a2 * tp.z;
                    tn.w = a.a1 * (xn.w - a.cshift * tk.w) - a.a2 * tp.w;
                    *reinterpret_cast<float4*>(a.Tn + r * a.ldtn + cc) = tn;
                    if (a.Z) {   // Z is the caller's: any alignment
                        float* z = a.Z + r * a.ldz + cc;
                        z[0] += (a.gam_tab ? (float)a.gam_tab[cc / a.gam_group] : a.gam) * tn.x;
                        z[1] += (a.gam_tab ? (float)a.gam_tab[(cc + 1) / a.gam_group] : a.gam) * tn.y;
                        z[2] += (a.gam_tab ? (float)a.gam_tab[(cc + 2) / a.gam_group] : a.gam) * tn.z;
                        z[3] += (a.gam_tab ? (float)a.gam_tab[(cc + 3) / a.gam_group] : a.gam) * tn.w;
                    }
                }
            }
        }
    }
}

template <int R, int L, int MODE, int S, int U, int MINB>
static int cluster_go(const KronArgs<float>& a, int ng, cudaStream_t s) {
    const int64_t per = 32 / (S * L) * (kThreads / 32);
    const unsigned grid = (unsigned)std::min<int64_t>((a.cl.n + per - 1) / per, (int64_t)a.cl.sms * MINB);
    if (a.ldx == 4 * L && ng == 1) {
        // Steps of less than about 20 warps per SM start while their
        // predecessor drains (803 clusters, 24 columns: a filter of 1,200
        // steps 10.9 -> 8.0 ms; 16.6k clusters, 16 columns 16.6 -> 15.6 ms);
        // above, the early CTAs and the plain loads cost more than the gap
        // (96k clusters, 32 columns 100.9 -> 104.0 ms).
        if ((int64_t)a.cl.n * L < 640 * (int64_t)a.cl.sms)
            return launch_dependent(kron_cluster_kernel<R, L, MODE, S, U, true, true, MINB>, dim3(grid), kThreads, s, a);
        kron_cluster_kernel<R, L, MODE, S, U, true, false, MINB><<<grid, kThreads, 0, s>>>(a);
    } else {
        kron_cluster_kernel<R, L, MODE, S, U, false, false, MINB><<<dim3(grid, ng), kThreads, 0, s>>>(a);
    }
    count_launch();
    NM_CUDA(cudaGetLastError());
    return NM_OK;
}

// Two lane groups per cluster fill the chip from 16 warps per SM on (b = 32:
// 234 us against 243 us with four); below that, and for at most 16 columns
// (24.3 us against 23.3 us) or one component (27 us against 26 us), four
// shorten a cluster's chain of trips.
template <int R, int L, int MODE>
static int cluster_launch(const KronArgs<float>& a, int ng, cudaStream_t s) {
    if constexpr (R == 3 && L > 4) {
        const int64_t warps = (int64_t)a.cl.n * ng * (2 * L) / 32;
        if (warps >= 16 * (int64_t)a.cl.sms) return cluster_go<R, L, MODE, 2, 3, 4>(a, ng, s);
    }
    if constexpr (R == 1)
        return cluster_go<R, L, MODE, 4, 3, 6>(a, ng, s);
    else
        return cluster_go<R, L, MODE, 4, 3, 4>(a, ng, s);
}

template <int R, int MODE>
static int cluster_width(const KronArgs<float>& a, cudaStream_t s) {
    const int lanes = a.b / 4, ng = (lanes + 7) / 8;
    switch ((lanes + ng - 1) / ng) {
        case 1: return cluster_launch<R, 1, MODE>(a, ng, s);
        case 2: return cluster_launch<R, 2, MODE>(a, ng, s);
        case 3: return cluster_launch<R, 3, MODE>(a, ng, s);
        case 4: return cluster_launch<R, 4, MODE>(a, ng, s);
        case 5: return cluster_launch<R, 5, MODE>(a, ng, s);
        case 6: return cluster_launch<R, 6, MODE>(a, ng, s);
        case 7: return cluster_launch<R, 7, MODE>(a, ng, s);
        default: return cluster_launch<R, 8, MODE>(a, ng, s);
    }
}

bool kron_cluster_ok(int R, int mode, const KronArgs<float>& a) {
    if (a.cl.n <= 0 || a.b % 4 != 0 || a.ldx % 4 != 0 || a.ldw % 4 != 0) return false;
    uintptr_t p = (uintptr_t)a.X | (uintptr_t)a.W | (uintptr_t)a.Xp;
    if (a.Xp && a.ldp % 4 != 0) return false;
    if (mode == KRON_CHEB) return (R == 1 || R == 3) && a.ldn % 4 == 0 && ((p | (uintptr_t)a.Xn) & 15) == 0;
    if (mode != KRON_CHEB_FILT || R != 3) return false;
    p |= (uintptr_t)a.Tk | (uintptr_t)a.Tp | (uintptr_t)a.Tn;
    return a.ldtk % 4 == 0 && (!a.Tp || a.ldtp % 4 == 0) && a.ldtn % 4 == 0 && (p & 15) == 0;
}

int launch_kron_cluster(int R, int mode, const KronArgs<float>& a, cudaStream_t s) {
    if (R == 1) return cluster_width<1, KRON_CHEB>(a, s);
    return mode == KRON_CHEB ? cluster_width<3, KRON_CHEB>(a, s) : cluster_width<3, KRON_CHEB_FILT>(a, s);
}

// Cluster values from the matrix values.
__global__ void cluster_values_kernel(int64_t n4, const int* at, const float* val, float* out) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n4; t += (int64_t)gridDim.x * blockDim.x)
        out[t] = at[t] < 0 ? 0.f : val[at[t]];
}

// Clusters inside windows of kMaxRows consecutive (Morton) rows, greedily: the
// undone row with most entries takes the three rows that add fewest new
// columns for the columns they share.
static int make_clusters(DevCSR& A, cudaStream_t s) {
    const int64_t N = A.nrows;
    if (N < 1 || A.nnz < 1) return NM_OK;
    const int64_t nwin = (N + kMaxRows - 1) / kMaxRows;
    constexpr int kPer = kMaxRows / 4;
    const int64_t ncl = (nwin - 1) * kPer + (N - (nwin - 1) * kMaxRows + 3) / 4;
    std::vector<int> ptr(ncl + 1, 0), rows(4 * ncl, -1);
    struct Win {
        std::vector<int> col, at;
    };
    std::vector<Win> win(nwin);
    const int* rp = A.h_rowptr.data();
    const int* col = A.h_col.data();
    std::atomic<bool> no_memory{false};   // an exception must not leave the parallel region
#pragma omp parallel
    {
        std::vector<int> cols, pos;
        std::vector<uint64_t> bits, cur;
#pragma omp for schedule(dynamic, 32)
        for (int64_t w = 0; w < nwin; ++w) {
            try {
                const int r0 = (int)(w * kMaxRows), n = (int)std::min<int64_t>(kMaxRows, N - r0);
                cols.assign(col + rp[r0], col + rp[r0 + n]);
                std::sort(cols.begin(), cols.end());
                cols.erase(std::unique(cols.begin(), cols.end()), cols.end());
                const int U = (int)cols.size(), words = (U + 63) / 64;
                bits.assign((size_t)n * words, 0);
                cur.assign(words, 0);
                pos.assign((size_t)n * U, -1);
                for (int i = 0; i < n; ++i)
                    for (int e = rp[r0 + i]; e < rp[r0 + i + 1]; ++e) {
                        const int l = (int)(std::lower_bound(cols.begin(), cols.end(), col[e]) - cols.begin());
                        bits[(size_t)i * words + l / 64] |= 1ull << (l % 64);
                        pos[(size_t)i * U + l] = e;
                    }
                int ord[kMaxRows];
                bool done[kMaxRows] = {};
                for (int i = 0; i < n; ++i) ord[i] = i;
                std::sort(ord, ord + n, [&](int x, int y) {
                    const int dx = rp[r0 + x + 1] - rp[r0 + x], dy = rp[r0 + y + 1] - rp[r0 + y];
                    return dx != dy ? dx > dy : x < y;
                });
                int64_t c = w * kPer;
                for (int o = 0; o < n; ++o) {
                    const int seed = ord[o];
                    if (done[seed]) continue;
                    int m[4] = {seed, -1, -1, -1};
                    done[seed] = true;
                    for (int k = 0; k < words; ++k) cur[k] = bits[(size_t)seed * words + k];
                    for (int f = 1; f < 4; ++f) {
                        int best = -1, bs = 1 << 30;
                        for (int i = 0; i < n; ++i) {
                            if (done[i]) continue;
                            int grow = 0, shared = 0;
                            for (int k = 0; k < words; ++k) {
                                const uint64_t b = bits[(size_t)i * words + k];
                                grow += __builtin_popcountll(b & ~cur[k]);
                                shared += __builtin_popcountll(b & cur[k]);
                            }
                            if (2 * grow - shared < bs) {
                                bs = 2 * grow - shared;
                                best = i;
                            }
                        }
                        if (best < 0) break;
                        m[f] = best;
                        done[best] = true;
                        for (int k = 0; k < words; ++k) cur[k] |= bits[(size_t)best * words + k];
                    }
                    int u = 0;
                    for (int l = 0; l < U; ++l) {
                        if (!((cur[l / 64] >> (l % 64)) & 1)) continue;
                        for (int f = 0; f < 4; ++f) win[w].at.push_back(m[f] < 0 ? -1 : pos[(size_t)m[f] * U + l]);
                        win[w].col.push_back(cols[l]);
                        ++u;
                    }
                    for (; u % kPad; ++u) {
                        for (int f = 0; f < 4; ++f) win[w].at.push_back(-1);
                        win[w].col.push_back(win[w].col.back());
                    }
                    for (int f = 0; f < 4; ++f) rows[4 * c + f] = m[f] < 0 ? -1 : r0 + m[f];
                    ptr[++c] = u;
                }
            } catch (const std::bad_alloc&) {
                no_memory = true;
            }
        }
    }
    if (no_memory) throw std::bad_alloc();
    int64_t ne = 0;
    for (int64_t c = 0; c < ncl; ++c) {
        ne += ptr[c + 1];
        if (ne > INT32_MAX / 4) return NM_OK;
        ptr[c + 1] = (int)ne;
    }
    std::vector<int> fc(ne), fa(4 * ne);
#pragma omp parallel for schedule(static)
    for (int64_t w = 0; w < nwin; ++w) {
        std::copy(win[w].col.begin(), win[w].col.end(), fc.begin() + ptr[w * kPer]);
        std::copy(win[w].at.begin(), win[w].at.end(), fa.begin() + 4 * (int64_t)ptr[w * kPer]);
    }
    DevBuf at;
    auto up = [&](DevBuf& b, const void* src, size_t bytes) -> int {
        NM_TRY(b.alloc(bytes));
        return copy_in(b.p, src, bytes, s);
    };
    NM_TRY(up(at, fa.data(), fa.size() * sizeof(int)));
    NM_TRY(up(A.cl_ptr, ptr.data(), ptr.size() * sizeof(int)));
    NM_TRY(up(A.cl_col, fc.data(), fc.size() * sizeof(int)));
    NM_TRY(up(A.cl_rows, rows.data(), rows.size() * sizeof(int)));
    NM_TRY(A.cl_val.alloc(fa.size() * sizeof(float)));
    cluster_values_kernel<<<(unsigned)std::min<int64_t>((4 * ne + 255) / 256 + 1, 4864), 256, 0, s>>>(
        4 * ne, at.as<int>(), A.val32.as<float>(), A.cl_val.as<float>());
    count_launch();
    NM_CUDA(cudaGetLastError());
    NM_CUDA(cudaStreamSynchronize(s));   // the positions are released here, later calls may come on another stream
    int dev = 0;
    NM_CUDA(cudaGetDevice(&dev));
    NM_CUDA(cudaDeviceGetAttribute(&A.cl.sms, cudaDevAttrMultiProcessorCount, dev));
    A.cl.n = (int)ncl;
    A.cl.ptr = A.cl_ptr.as<int>();
    A.cl.col = A.cl_col.as<int>();
    A.cl.val = A.cl_val.as<float4>();
    A.cl.rows = A.cl_rows.as<int4>();
    A.cl_state = 1;
    return NM_OK;
}

// State -1 only for matrices without clusters: a call that finds no memory
// fails, and the next one tries again.
int build_clusters(DevCSR& A, cudaStream_t s) {
    if (A.cl_state) return NM_OK;
    int rc;
    try {
        rc = make_clusters(A, s);
    } catch (const std::bad_alloc&) {
        rc = fail(NM_ENOMEM, "host allocation failed");
    }
    if (rc == NM_OK && A.cl_state == 0) A.cl_state = -1;
    return rc;
}

}  // namespace nm
