// Sparse products row by row (any type, width and leading dimension): the
// scalar matrix (x) I_R with the semi-iteration epilogues, the 3x3-block K_eff
// product and the 1x3-block E_G^T product.
//
// What bounds them: in double, the FP64 units (2 multiply-adds per clock and
// SM) once the rows fill the chip; on small meshes and narrow blocks the chain
// of dependent loads row -> columns -> records, and the launch. So:
//  - a row's entries are split over S lane groups and U entries per group are
//    in flight together: a 27-entry row is fetched in one or two round trips;
//    S falls to 1 as the rows fill the chip, since every doubling adds FP64
//    additions;
//  - an FP64 instruction holds its SM's pipe for 16 cycles however few lanes
//    are active: the groups' sums are scattered, not broadcast, and the
//    epilogue is spread over the groups with them;
//  - rows are taken in order of length inside windows of 64 (descriptors row,
//    first entry, end), so that the rows of one warp end together: unsorted,
//    a warp of eight rows runs as long as its 65-entry vertex row while the
//    mean is 27;
//  - CTAs of two warps: with four, 1124 CTAs of equal speed left 60 for a
//    second, nearly empty wave (the step's SMs were active 61% of the time);
//  - kernels of a chain start while their predecessor drains (programmatic
//    dependent launch): descriptors, columns and values do not depend on it
//    and are loaded before the wait.
// A lane group per row walking its entries one by one (the form before)
// against now, per semi-iteration step in double at 8 columns: 633 rows
// 26 -> 6.4 us, 17,977 rows 49 -> 40 us (FP64 floor 20 us).
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <initializer_list>
#include <vector>

#include "kernels.h"
#include "nm_internal.h"
#include "dependent.cuh"

namespace nm {

namespace {

constexpr int kThreads = 64;
constexpr int kWindow = 64;

// VW consecutive values of a row of which n exist. PAIR: two-value accesses
// (even widths and strides, aligned operands).
template <typename T, int VW>
struct Vec {
    T v[VW];
};
template <typename T>
struct Pair;
template <>
struct Pair<double> {
    using type = double2;
};
template <>
struct Pair<float> {
    using type = float2;
};
template <bool PAIR, typename T, int VW>
__device__ __forceinline__ Vec<T, VW> ld(const T* p, int n) {
    Vec<T, VW> r;
    if constexpr (PAIR) {
        using P = typename Pair<T>::type;
#pragma unroll
        for (int i = 0; i < VW; i += 2) {
            P t;
            t.x = t.y = T(0);
            if (i < n) t = *reinterpret_cast<const P*>(p + i);
            r.v[i] = t.x, r.v[i + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < VW; ++i) r.v[i] = i < n ? p[i] : T(0);
    }
    return r;
}
template <bool PAIR, typename T, int VW>
__device__ __forceinline__ void st(T* p, const Vec<T, VW>& r, int n) {
    if constexpr (PAIR) {
        using P = typename Pair<T>::type;
#pragma unroll
        for (int i = 0; i < VW; i += 2) {
            P t;
            t.x = r.v[i], t.y = r.v[i + 1];
            if (i < n) *reinterpret_cast<P*>(p + i) = t;
        }
    } else {
#pragma unroll
        for (int i = 0; i < VW; ++i)
            if (i < n) p[i] = r.v[i];
    }
}
template <typename T, int VW>
__device__ __forceinline__ Vec<T, VW> zero() {
    Vec<T, VW> r;
#pragma unroll
    for (int i = 0; i < VW; ++i) r.v[i] = T(0);
    return r;
}

// Sums N values over the S lane groups (tl lanes each) of a row. Every step
// halves the values a lane keeps (a group gives away the half it drops), so
// that S groups cost about N additions, not N log2 S, and what follows the
// sum is spread over the groups: on return v[0 .. cnt) holds the sums of the
// values base .. base + cnt - 1. An FP64 instruction holds its SM's pipe for
// 16 cycles however few lanes are active.
template <typename T, int N, int S>
struct Scatter {
    // values a lane keeps at most
    static constexpr int kept(int n, int s) { return s == 1 || n == 1 ? n : kept((n + 1) / 2, s / 2); }
    static constexpr int kKeep = kept(N, S);
    int base = 0, cnt = N;
    __device__ __forceinline__ explicit Scatter(int sp) {
        int n = N;
#pragma unroll
        for (int m = 1; m < S; m *= 2) {
            const bool up = sp & m;
            if (n == 1) {
                if (up) cnt = 0;
            } else {
                const int h = (n + 1) / 2;
                base += up ? h : 0;
                cnt = up ? max(cnt - h, 0) : min(cnt, h);
                n = h;
            }
        }
    }
    __device__ __forceinline__ void sum(T (&v)[N], int sp, int tl) const {
        int n = N;
#pragma unroll
        for (int m = 1; m < S; m *= 2) {
            const bool up = sp & m;
            if (n == 1) {
                v[0] += __shfl_xor_sync(0xffffffffu, v[0], m * tl);
            } else {
                const int h = (n + 1) / 2;
#pragma unroll
                for (int i = 0; i < (N + 1) / 2; ++i) {
                    if (i < h) {
                        const T hi = h + i < n ? v[h + i < N ? h + i : 0] : T(0);
                        const T give = up ? v[i] : hi, keep = up ? hi : v[i];
                        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, m * tl);
                    }
                }
                n = h;
            }
        }
    }
};

// Where a lane works: split sp of a row, columns c .. c + n - 1 (n = 0: no
// row). L lanes cover the columns; with splits L is a power of two.
struct Place {
    int sp, c, n;
    int4 d;   // row, first entry, end
};
template <int VW, int S>
__device__ __forceinline__ Place place(const int4* desc, int nrows, int b, int L) {
    Place p;
    const int lane = threadIdx.x & 31, lc = L * S, per = 32 / lc;
    const int cw = lane / lc, rl = lane - cw * lc;
    p.sp = rl / L;
    p.c = VW * (rl - p.sp * L + blockIdx.y * L);
    const int slot = (blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * per + cw;
    const bool on = cw < per && slot < nrows && p.c < b;
    p.d = __ldg(desc + (on ? slot : 0));
    p.n = on ? min(VW, b - p.c) : 0;
    if (!on) p.c = 0, p.d.z = p.d.y;   // no entries
    return p;
}

}  // namespace

// ----------------------------------------------------------------- A (x) I_R
template <typename T, int R, int MODE, int VW, bool PAIR, int S, int U>
__global__ void __launch_bounds__(kThreads) kron_rows_kernel(const KronArgs<T> a, int L) {
    const Place p = place<VW, S>(a.desc, a.nrows, a.b, L);
    const int c = p.c;
    const int64_t row = p.d.x;
    T acc[R * VW];
#pragma unroll
    for (int i = 0; i < R * VW; ++i) acc[i] = T(0);
    const T* const X = a.X + c;
    const int64_t RL = (int64_t)R * a.ldx;
    int e = p.d.y + p.sp;
    int j[U];
    T v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const bool ok = e + u * S < p.d.z;
        j[u] = ok ? __ldg(a.col + e + u * S) : -1;
        v[u] = ok ? __ldg(a.val + e + u * S) : T(0);
    }
    constexpr bool kCheb = MODE == KRON_CHEB || MODE == KRON_CHEB_FILT;
    const T dd = kCheb ? __ldg(a.dinv + row) * a.inv_theta : T(0);
    dep_sync();
    constexpr int N = R * VW;
    // CORI mixes the components: its lanes keep all of them
    constexpr int SS = MODE == KRON_CORI ? 1 : S;
    const Scatter<T, N, SS> sc(p.sp);
    constexpr int K = Scatter<T, N, SS>::kKeep;
    const int cnt = p.n ? sc.cnt : 0;
    // a lane's own values of a block: whole vectors, or single ones when the
    // row's sums are scattered over its lane groups
    auto own = [&](const T* base, int64_t l, T (&o)[K]) {
        if constexpr (SS == 1) {
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const Vec<T, VW> t = ld<PAIR, T, VW>(base + (R * row + k) * l + c, p.n);
#pragma unroll
                for (int i = 0; i < VW; ++i) o[k * VW + i] = t.v[i];
            }
        } else {
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const int t = sc.base + i;
                o[i] = i < cnt ? base[(R * row + t / VW) * l + c + t % VW] : T(0);
            }
        }
    };
    auto put = [&](T* base, int64_t l, const T (&o)[K]) {
        if constexpr (SS == 1) {
            if (S == 1 || p.sp == 0)
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    Vec<T, VW> t;
#pragma unroll
                    for (int i = 0; i < VW; ++i) t.v[i] = o[k * VW + i];
                    st<PAIR, T, VW>(base + (R * row + k) * l + c, t, p.n);
                }
        } else {
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const int t = sc.base + i;
                if (i < cnt) base[(R * row + t / VW) * l + c + t % VW] = o[i];
            }
        }
    };
    T xk[K], w[K], xp[K];
    if (kCheb) {
        own(a.X, a.ldx, xk);
        own(a.W, a.ldw, w);
#pragma unroll
        for (int i = 0; i < K; ++i) xp[i] = T(0);
        if (a.Xp) own(a.Xp, a.ldp, xp);
    }
    while (e < p.d.z) {
        Vec<T, VW> x[U][R];
        T vc[U];
        bool in[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            in[u] = j[u] >= 0;
            vc[u] = v[u];
#pragma unroll
            for (int k = 0; k < R; ++k) x[u][k] = in[u] ? ld<PAIR, T, VW>(X + j[u] * RL + k * a.ldx, p.n) : zero<T, VW>();
        }
        e += U * S;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool ok = e + u * S < p.d.z;
            j[u] = ok ? __ldg(a.col + e + u * S) : -1;
            v[u] = ok ? __ldg(a.val + e + u * S) : T(0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (in[u]) {
#pragma unroll
                for (int k = 0; k < R; ++k)
#pragma unroll
                    for (int i = 0; i < VW; ++i) acc[k * VW + i] = fma(vc[u], x[u][k].v[i], acc[k * VW + i]);
            }
    }
    if constexpr (SS == S) {
        sc.sum(acc, p.sp, L);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int m = 1; m < S; m *= 2) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], m * L);
    }
    T o[K];
    if (MODE == KRON_PLAIN) {
#pragma unroll
        for (int i = 0; i < K; ++i) o[i] = acc[i];
        put(a.Y, a.ldy, o);
    } else if constexpr (MODE == KRON_CORI) {
#pragma unroll
        for (int m = 0; m < R; ++m)
#pragma unroll
            for (int i = 0; i < VW; ++i) {
                T y = T(0);
#pragma unroll
                for (int k = 0; k < R; ++k) y += a.sk[m * 3 + k] * acc[k * VW + i];
                o[m * VW + i] = y;
            }
        put(a.Y, a.ldy, o);
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) o[i] = xp[i] + a.om * (xk[i] - xp[i] + dd * (w[i] - acc[i]));
        if (MODE == KRON_CHEB) {
            put(a.Xn, a.ldn, o);
        } else {
            T tk[K], tp[K];
            own(a.Tk, a.ldtk, tk);
#pragma unroll
            for (int i = 0; i < K; ++i) tp[i] = T(0);
            if (a.Tp) own(a.Tp, a.ldtp, tp);
#pragma unroll
            for (int i = 0; i < K; ++i) o[i] = a.a1 * (o[i] - a.cshift * tk[i]) - a.a2 * tp[i];
            put(a.Tn, a.ldtn, o);
            if (a.Z) {
                T z[K];
                own(a.Z, a.ldz, z);
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    const int cc = c + (SS == 1 ? i : sc.base + i) % VW;
                    z[i] += (a.gam_tab && cc < a.b ? (T)a.gam_tab[cc / a.gam_group] : a.gam) * o[i];
                }
                put(a.Z, a.ldz, z);
            }
        }
    }
}

// ----------------------------------------------------------------- 3x3 BSR (+ E S)
template <typename T, int VW, bool PAIR, int S, int U>
__global__ void __launch_bounds__(kThreads) bsr33_rows_kernel(const Bsr33Args<T> a, int L) {
    const Place p = place<VW, S>(a.desc, a.nrows, a.b, L);
    const int c = p.c;
    const int64_t row = p.d.x;
    const int f0 = a.e_rowptr && p.n ? __ldg(a.e_rowptr + row) : 0, f1 = a.e_rowptr && p.n ? __ldg(a.e_rowptr + row + 1) : 0;
    constexpr int N = 3 * VW;
    T acc[N];
#pragma unroll
    for (int i = 0; i < N; ++i) acc[i] = T(0);
    const T* const X = a.X + c;
    int e = p.d.y + p.sp;
    int j[U];
#pragma unroll
    for (int u = 0; u < U; ++u) j[u] = e + u * S < p.d.z ? __ldg(a.col + e + u * S) : -1;
    dep_sync();
    while (e < p.d.z) {
        Vec<T, VW> x[U][3];
        T kv[U][9];
        bool in[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            in[u] = j[u] >= 0;
#pragma unroll
            for (int k = 0; k < 3; ++k)
                x[u][k] = in[u] ? ld<PAIR, T, VW>(X + (3 * (int64_t)j[u] + k) * a.ldx, p.n) : zero<T, VW>();
#pragma unroll
            for (int t = 0; t < 9; ++t) kv[u][t] = in[u] ? __ldg(a.val + 9 * (int64_t)(e + u * S) + t) : T(0);
        }
        e += U * S;
#pragma unroll
        for (int u = 0; u < U; ++u) j[u] = e + u * S < p.d.z ? __ldg(a.col + e + u * S) : -1;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (in[u]) {
#pragma unroll
                for (int m = 0; m < 3; ++m)
#pragma unroll
                    for (int k = 0; k < 3; ++k)
#pragma unroll
                        for (int i = 0; i < VW; ++i)
                            acc[m * VW + i] = fma(kv[u][3 * m + k], x[u][k].v[i], acc[m * VW + i]);
            }
    }
#pragma unroll 2
    for (int f = f0 + p.sp; f < f1; f += S) {
        const Vec<T, VW> sv = ld<PAIR, T, VW>(a.S + (int64_t)__ldg(a.e_col + f) * a.lds + c, p.n);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const T ev = __ldg(a.e_val + 3 * (int64_t)f + m);
#pragma unroll
            for (int i = 0; i < VW; ++i) acc[m * VW + i] = fma(ev, sv.v[i], acc[m * VW + i]);
        }
    }
    const Scatter<T, N, S> sc(p.sp);
    constexpr int K = Scatter<T, N, S>::kKeep;
    sc.sum(acc, p.sp, L);
    if (!p.n) return;
    const T d = a.X1 ? __ldg(a.dinv + row) * a.inv_theta : T(0);
    if constexpr (S == 1) {
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            Vec<T, VW> t;
#pragma unroll
            for (int i = 0; i < VW; ++i) t.v[i] = acc[m * VW + i];
            st<PAIR, T, VW>(a.W + (3 * row + m) * a.ldw + c, t, p.n);
            if (a.X1) {
#pragma unroll
                for (int i = 0; i < VW; ++i) t.v[i] *= d;
                st<PAIR, T, VW>(a.X1 + (3 * row + m) * a.ldx1 + c, t, p.n);
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) {
            if (i >= sc.cnt) break;
            const int t = sc.base + i;
            a.W[(3 * row + t / VW) * a.ldw + c + t % VW] = acc[i];
            if (a.X1) a.X1[(3 * row + t / VW) * a.ldx1 + c + t % VW] = d * acc[i];
        }
    }
}

// ----------------------------------------------------------------- 1x3 BSR
template <typename T, int VW, bool PAIR, int S, int U>
__global__ void __launch_bounds__(kThreads) bsr13_rows_kernel(const Bsr13Args<T> a, int L) {
    const Place p = place<VW, S>(a.desc, a.nrows, a.b, L);
    const int c = p.c;
    const int64_t row = p.d.x;
    T acc[VW];
#pragma unroll
    for (int i = 0; i < VW; ++i) acc[i] = T(0);
    const T* const X = a.X + c;
    int e = p.d.y + p.sp;
    int j[U];
    T v[U][3];
    auto fetch = [&]() {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool ok = e + u * S < p.d.z;
            j[u] = ok ? __ldg(a.col + e + u * S) : -1;
#pragma unroll
            for (int k = 0; k < 3; ++k) v[u][k] = ok ? __ldg(a.val + 3 * (int64_t)(e + u * S) + k) : T(0);
        }
    };
    fetch();
    dep_sync();
    while (e < p.d.z) {
        Vec<T, VW> x[U][3];
        T vc[U][3];
        bool in[U];
#pragma unroll
        for (int u = 0; u < U; ++u) in[u] = j[u] >= 0;
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                x[u][k] = in[u] ? ld<PAIR, T, VW>(X + (3 * (int64_t)j[u] + k) * a.ldx, p.n) : zero<T, VW>();
                vc[u][k] = v[u][k];
            }
        e += U * S;
        fetch();
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (in[u]) {
#pragma unroll
                for (int k = 0; k < 3; ++k)
#pragma unroll
                    for (int i = 0; i < VW; ++i) acc[i] = fma(vc[u][k], x[u][k].v[i], acc[i]);
            }
    }
    const Scatter<T, VW, S> sc(p.sp);
    constexpr int K = Scatter<T, VW, S>::kKeep;
    sc.sum(acc, p.sp, L);
    if (!p.n) return;
    const T d = a.S1 ? __ldg(a.dinv + row) * a.inv_theta : T(0);
#pragma unroll
    for (int i = 0; i < K; ++i) {
        if (i >= min(sc.cnt, S == 1 ? p.n : VW)) break;
        a.Q[row * a.ldq + c + sc.base + i] = acc[i];
        if (a.S1) a.S1[row * a.lds1 + c + sc.base + i] = d * acc[i];
    }
}

// ----------------------------------------------------------------- launches
namespace {

int sm_count() {
    static std::atomic<int> n{0};
    int v = n.load(std::memory_order_relaxed);
    if (v == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1)
            v = 148;
        n.store(v, std::memory_order_relaxed);
    }
    return v;
}

struct Shape {
    int vw, L, splits;
    dim3 grid;
};

// Columns per lane and lanes per row. While the rows leave the chip below 16
// warps per SM the splits double (a double filter at 17,977 rows and 8 columns:
// 16.6 / 15.1 / 11.7 / 12.1 ms with 4 / 8 / 16 / 32 warps); L is then a power
// of two and the lanes hold pairs where the operands allow. Unsplit, the FP64
// pipe bounds, and the columns per lane (1 .. 4) are those that leave fewest
// lanes of a warp idle: 24 columns as 5 rows of 6 lanes, not 2 of 12.
template <typename T>
Shape shape(int nrows, int b, bool pair) {
    Shape h;
    h.vw = pair ? 2 : 1;
    int lanes = (b + h.vw - 1) / h.vw, shift = 0;
    while (shift < 5 && (1 << shift) < lanes) ++shift;
    h.L = 1 << shift;
    int ny = (lanes + h.L - 1) >> shift;
    h.splits = 1;
    while (h.splits < 8 && h.splits * h.L < 32 && (int64_t)nrows * ny * h.splits * h.L / 32 < 16 * (int64_t)sm_count())
        h.splits *= 2;
    if (h.splits == 1 && sizeof(T) == 8) {
        double best = 0;
        for (int vw : {2, 4, 1, 3}) {
            const int n = (b + vw - 1) / vw, y = (n + 31) / 32, L = (n + y - 1) / y;
            const double use = (double)(32 / L) * b / vw / (32.0 * y);
            if (use > best + 0.01) {
                best = use;
                h.vw = vw, h.L = L, ny = y;
            }
        }
    }
    const int64_t per = 32 / (h.L * h.splits) * (kThreads / 32);
    h.grid = dim3((unsigned)((nrows + per - 1) / per), (unsigned)ny);
    return h;
}

// two-value accesses need even widths and strides and aligned operands
template <typename T>
bool pairs(int b, std::initializer_list<int64_t> lds, std::initializer_list<const void*> ptrs) {
    if (b % 2) return false;
    for (int64_t l : lds)
        if (l % 2) return false;
    uintptr_t p = 0;
    for (const void* q : ptrs) p |= (uintptr_t)q;
    return (p & (2 * sizeof(T) - 1)) == 0;
}

// One kernel per columns per lane, splits and kind of access.
#define NM_ROWS(K)                                                                       \
    if (h.splits == 1) {                                                                 \
        switch (h.vw) {                                                                  \
            case 1: return launch_dependent(K(1, false, 1), h.grid, kThreads, s, a, h.L);                         \
            case 2: return pair ? launch_dependent(K(2, true, 1), h.grid, kThreads, s, a, h.L) : launch_dependent(K(2, false, 1), h.grid, kThreads, s, a, h.L); \
            case 3: return launch_dependent(K(3, false, 1), h.grid, kThreads, s, a, h.L);                         \
            default: return pair ? launch_dependent(K(4, true, 1), h.grid, kThreads, s, a, h.L) : launch_dependent(K(4, false, 1), h.grid, kThreads, s, a, h.L); \
        }                                                                                \
    }                                                                                    \
    switch (h.splits) {                                                                  \
        case 2: return pair ? launch_dependent(K(2, true, 2), h.grid, kThreads, s, a, h.L) : launch_dependent(K(1, false, 2), h.grid, kThreads, s, a, h.L); \
        case 4: return pair ? launch_dependent(K(2, true, 4), h.grid, kThreads, s, a, h.L) : launch_dependent(K(1, false, 4), h.grid, kThreads, s, a, h.L); \
        default: return pair ? launch_dependent(K(2, true, 8), h.grid, kThreads, s, a, h.L) : launch_dependent(K(1, false, 8), h.grid, kThreads, s, a, h.L); \
    }

template <typename T, int R, int MODE>
int kron_rows_mode(const KronArgs<T>& a, cudaStream_t s) {
    if (a.nrows == 0) return NM_OK;
    bool pair;
    if (MODE == KRON_PLAIN || MODE == KRON_CORI)
        pair = pairs<T>(a.b, {a.ldx, a.ldy}, {a.X, a.Y});
    else if (MODE == KRON_CHEB)
        pair = pairs<T>(a.b, {a.ldx, a.ldw, a.ldp, a.ldn}, {a.X, a.W, a.Xp, a.Xn});
    else
        pair = pairs<T>(a.b, {a.ldx, a.ldw, a.ldp, a.ldtk, a.ldtp, a.ldtn, a.ldz}, {a.X, a.W, a.Xp, a.Tk, a.Tp, a.Tn, a.Z});
    const Shape h = shape<T>(a.nrows, a.b, pair);
#define NM_K(VW, PAIR, S) kron_rows_kernel<T, R, MODE, VW, PAIR, S, (VW > 2 && R == 3 ? 2 : 4)>
    NM_ROWS(NM_K)
#undef NM_K
}

template <typename T>
int bsr33_rows(const Bsr33Args<T>& a, cudaStream_t s) {
    const bool pair = pairs<T>(a.b, {a.ldx, a.ldw, a.lds, a.ldx1}, {a.X, a.W, a.S, a.X1});
    const Shape h = shape<T>(a.nrows, a.b, pair);
#define NM_K(VW, PAIR, S) bsr33_rows_kernel<T, VW, PAIR, S, 2>
    NM_ROWS(NM_K)
#undef NM_K
}

template <typename T>
int bsr13_rows(const Bsr13Args<T>& a, cudaStream_t s) {
    const bool pair = pairs<T>(a.b, {a.ldx, a.ldq, a.lds1}, {a.X, a.Q, a.S1});
    const Shape h = shape<T>(a.nrows, a.b, pair);
#define NM_K(VW, PAIR, S) bsr13_rows_kernel<T, VW, PAIR, S, (VW > 2 ? 2 : 4)>
    NM_ROWS(NM_K)
#undef NM_K
}
#undef NM_ROWS

}  // namespace

template <typename T>
int launch_kron_rows(int R, int mode, const KronArgs<T>& a, cudaStream_t s) {
    if (R == 3) {
        switch (mode) {
            case KRON_PLAIN: return kron_rows_mode<T, 3, KRON_PLAIN>(a, s);
            case KRON_CHEB: return kron_rows_mode<T, 3, KRON_CHEB>(a, s);
            case KRON_CHEB_FILT: return kron_rows_mode<T, 3, KRON_CHEB_FILT>(a, s);
            case KRON_CORI: return kron_rows_mode<T, 3, KRON_CORI>(a, s);
        }
    } else if (R == 1) {
        switch (mode) {
            case KRON_PLAIN: return kron_rows_mode<T, 1, KRON_PLAIN>(a, s);
            case KRON_CHEB: return kron_rows_mode<T, 1, KRON_CHEB>(a, s);
            default: break;
        }
    }
    return fail(NM_EINVAL, "unsupported kron mode");
}

template <typename T>
int launch_bsr33(const Bsr33Args<T>& a, cudaStream_t s) {
    if (a.b < 1 || a.b > 64) return fail(NM_EINVAL, "block width must be in 1..64");
    if (a.nrows == 0) return NM_OK;
    return bsr33_rows<T>(a, s);
}

template <typename T>
int launch_bsr13(const Bsr13Args<T>& a, cudaStream_t s) {
    if (a.b < 1 || a.b > 64) return fail(NM_EINVAL, "block width must be in 1..64");
    if (a.nrows == 0) return NM_OK;
    return bsr13_rows<T>(a, s);
}

// Row descriptors: rows of each window of 64 in order of decreasing length.
int build_row_desc(DevCSR& A, cudaStream_t s) {
    const int64_t N = A.nrows;
    std::vector<int4> d(std::max<int64_t>(N, 1));
    const int32_t* rp = A.h_rowptr.data();
#pragma omp parallel for schedule(static)
    for (int64_t w = 0; w < (N + kWindow - 1) / kWindow; ++w) {
        const int64_t r0 = w * kWindow, r1 = std::min<int64_t>(N, r0 + kWindow);
        for (int64_t r = r0; r < r1; ++r) d[r] = make_int4((int)r, rp[r], rp[r + 1], 0);
        std::stable_sort(d.begin() + r0, d.begin() + r1, [](const int4& x, const int4& y) { return x.z - x.y > y.z - y.y; });
    }
    NM_TRY(A.desc.alloc(d.size() * sizeof(int4)));
    return copy_in(A.desc.p, d.data(), d.size() * sizeof(int4), s);
}

template int launch_kron_rows<double>(int, int, const KronArgs<double>&, cudaStream_t);
template int launch_kron_rows<float>(int, int, const KronArgs<float>&, cudaStream_t);
template int launch_bsr33<double>(const Bsr33Args<double>&, cudaStream_t);
template int launch_bsr33<float>(const Bsr33Args<float>&, cudaStream_t);
template int launch_bsr13<double>(const Bsr13Args<double>&, cudaStream_t);
template int launch_bsr13<float>(const Bsr13Args<float>&, cudaStream_t);

}  // namespace nm
