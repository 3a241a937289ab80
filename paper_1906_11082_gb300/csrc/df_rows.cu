// Double-float sparse products, row by row, any width: the K_eff block SpMM
// of the mixed form and the refinement residuals.
//
// Values and vectors are exact pairs of floats (hi + lo); a sum is a running
// float and the errors of everything added to it, collected in a second one
// (Dot2 of Ogita, Rump and Oishi): 12 float operations a term. (Adding the
// unrounded product by one fused multiply-add saves three of them and loses
// the error's low bits when the sum cancels: 5e-9 instead of 8e-15.)
//
// What bounds the K_eff SpMM: the float pipe. 1.15M dof, 32 columns: 3.0e9
// terms x 12 = 3.6e10 lane operations, 0.97 ms at 128 lanes x 152 SMs x 1.92
// GHz; the fluid rows' E_G S in double adds 0.23e9 multiply-adds, 0.40 ms of
// the FP64 pipe (2 per clock and SM). A row's entries are split over S = 4
// groups of L = columns / 4 lanes (two groups round sums of twice the length:
// 1.5e-14 against 9e-15 relative); rows come in order of length (rows.cu); the
// sums are scattered over the groups, so that E_G S uses every lane. 64
// registers and 32 warps per SM: 1.84 ms; the same with packed pairs and the
// records loaded ahead at 128 registers 1.98 ms.
// Against one lane per column (the form before, other widths than 32), 199k
// dof: 16 columns 320 -> 214 us, 64 columns 861 -> 610 us; 9.6k dof, 21
// columns 75 -> 36 us.
// The residuals are bound by their gathers (three entries in flight): 1.15M
// dof, 32 columns 723 -> 662 us, 199k dof, 64 columns 332 -> 236 us. They take
// w as a pair of floats (48 bits): subtracting in double held the FP64 pipe for
// 0.3 ms, and taking w exactly (three floats) changes no error: solves, products
// and filters of 4k to 1.15M dof at 18 to 40 inner steps within 1% of each other.
#include <algorithm>
#include <cstdint>

#include "kernels.h"
#include "nm_internal.h"
#include "df_convert.cuh"

namespace nm {

namespace {

constexpr int kThreads = 64;
using u64 = unsigned long long;

__device__ __forceinline__ u64 pack2(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(u64 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 neg2(u64 a) { return a ^ 0x8000000080000000ull; }
constexpr u64 kMinus1 = 0xBF800000BF800000ull;

// a - b, exactly as a subtraction rounds
__device__ __forceinline__ u64 sub2(u64 a, u64 b) { return fma2(b, kMinus1, a); }

// (s, l) += (ah + al) x, two columns at a time.
__device__ __forceinline__ void df_acc2(u64& s, u64& l, u64 ah, u64 al, u64 x) {
    const u64 p = mul2(ah, x);
    u64 t = fma2(al, x, fma2(ah, x, neg2(p)));
    const u64 sn = add2(s, p);
    const u64 nz = sub2(s, sn);
    t = add2(t, sub2(s, add2(sn, nz)));
    t = add2(t, add2(p, nz));
    l = add2(l, t);
    s = sn;
}

// (sh, sl) += (ah + al)(xh + xl).
__device__ __forceinline__ void df_acc(float& sh, float& sl, float ah, float al, float xh, float xl) {
    const float p = __fmul_rn(ah, xh);
    const float e = __fmaf_rn(ah, xh, -p);
    const float t = __fmaf_rn(ah, xl, __fmaf_rn(al, xh, e));
    const float s = __fadd_rn(sh, p);
    const float bp = __fadd_rn(s, -sh);
    const float err = __fadd_rn(__fadd_rn(sh, -__fadd_rn(s, -bp)), __fadd_rn(p, -bp));
    sh = s;
    sl = __fadd_rn(sl, __fadd_rn(err, t));
}

// (sh, sl) += (h2, l2) for two such sums.
__device__ __forceinline__ void df_merge(float& sh, float& sl, float h2, float l2) {
    const float s = __fadd_rn(sh, h2);
    const float bp = __fadd_rn(s, -sh);
    const float err = __fadd_rn(__fadd_rn(sh, -__fadd_rn(s, -bp)), __fadd_rn(h2, -bp));
    sh = s;
    sl = __fadd_rn(sl, __fadd_rn(err, l2));
}

// values a lane keeps of n when they are scattered over S groups
template <int N, int S>
struct Kept {
    static constexpr int n = Kept<(N + 1) / 2, S / 2>::n;
};
template <int N>
struct Kept<N, 1> {
    static constexpr int n = N;
};

// Sums N pairs over S lane groups (L lanes apart); every step halves what a
// lane keeps: on return h, l [0 .. cnt) are the sums of values base ..
template <int N, int S, int L>
__device__ __forceinline__ void df_scatter(float (&h)[N], float (&l)[N], int lane, int sp, int& base, int& cnt) {
    int n = N;
    base = 0;
    cnt = N;
#pragma unroll
    for (int m = 1; m < S; m *= 2) {
        const bool up = sp & m;
        const int peer = lane + (up ? -m : m) * L;
        if (n == 1) {
            df_merge(h[0], l[0], __shfl_sync(0xffffffffu, h[0], peer), __shfl_sync(0xffffffffu, l[0], peer));
            if (up) cnt = 0;
        } else {
            const int k = (n + 1) / 2;
#pragma unroll
            for (int i = 0; i < (N + 1) / 2; ++i) {
                if (i < k) {
                    const bool has = k + i < n;
                    const float hh = has ? h[k + i < N ? k + i : 0] : 0.f, hl = has ? l[k + i < N ? k + i : 0] : 0.f;
                    const float gh = up ? h[i] : hh, gl = up ? l[i] : hl;
                    h[i] = up ? hh : h[i];
                    l[i] = up ? hl : l[i];
                    df_merge(h[i], l[i], __shfl_sync(0xffffffffu, gh, peer), __shfl_sync(0xffffffffu, gl, peer));
                }
            }
            base += up ? k : 0;
            cnt = up ? max(cnt - k, 0) : min(cnt, k);
            n = k;
        }
    }
}

struct Lane {
    int sp, q;
    bool on;
    int4 d;
};
template <int L, int S>
__device__ __forceinline__ Lane place(const int4* desc, int nrows, int blk) {
    constexpr int LC = S * L, CW = 32 / LC;
    const int lane = threadIdx.x & 31;
    const int cw = lane / LC, rl = lane - cw * LC;
    Lane p;
    p.sp = rl / L;
    p.q = rl - p.sp * L;
    const int slot = (blk * (kThreads / 32) + (threadIdx.x >> 5)) * CW + cw;
    p.on = cw < CW && slot < nrows;
    p.d = __ldg(desc + (p.on ? slot : 0));
    if (!p.on) p.d.z = p.d.y;
    return p;
}

}  // namespace

// ----------------------------------------------------------------- K_eff
template <int L, int S>
__global__ void __launch_bounds__(kThreads, 16) bsr33_df_rows_kernel(const Bsr33DfArgs a, int ng) {
    const int blk = blockIdx.x / ng, c0 = (blockIdx.x - blk * ng) * 4 * L;   // column group
    const Lane p = place<L, S>(a.desc, a.nrows, blk);
    const int64_t row = p.d.x;
    const float* const Xh = a.Xh + c0 + 4 * p.q;
    const float* const Xl = a.Xl + c0 + 4 * p.q;
    float sh[12], sl[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) sh[i] = sl[i] = 0.f;
    for (int e = p.d.y + p.sp; e < p.d.z; e += S) {
        const int64_t j = 3 * (int64_t)__ldg(a.col + e);
        const float* v = reinterpret_cast<const float*>(a.vhl + 5 * (int64_t)e);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float4 xh = __ldg(reinterpret_cast<const float4*>(Xh + (j + k) * a.ldx));
            const float4 xl = __ldg(reinterpret_cast<const float4*>(Xl + (j + k) * a.ldx));
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const float ah = __ldg(v + 3 * m + k), al = __ldg(v + 9 + 3 * m + k);
                df_acc(sh[4 * m + 0], sl[4 * m + 0], ah, al, xh.x, xl.x);
                df_acc(sh[4 * m + 1], sl[4 * m + 1], ah, al, xh.y, xl.y);
                df_acc(sh[4 * m + 2], sl[4 * m + 2], ah, al, xh.z, xl.z);
                df_acc(sh[4 * m + 3], sl[4 * m + 3], ah, al, xh.w, xl.w);
            }
        }
    }
    int base, cnt;
    df_scatter<12, S, L>(sh, sl, threadIdx.x & 31, p.sp, base, cnt);
    if (!p.on) return;
    constexpr int K = Kept<12, S>::n;
    double acc[K];
    int cc[K], mm[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        const int t = base + i;
        mm[i] = t >> 2;
        cc[i] = c0 + 4 * p.q + (t & 3);
        if (i >= cnt || cc[i] >= a.b) cc[i] = -1;
        acc[i] = widen(sh[i]) + widen(sl[i]);
    }
    if (a.e_rowptr) {
        const int f1 = __ldg(a.e_rowptr + row + 1);
        constexpr int V = K > 3 ? 2 : 4;   // couplings in flight
        for (int f = __ldg(a.e_rowptr + row); f < f1; f += V) {
            int pc[V];
#pragma unroll
            for (int v = 0; v < V; ++v) pc[v] = f + v < f1 ? __ldg(a.e_col + f + v) : -1;
            double ev[V][K], sv[V][K];
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int i = 0; i < K; ++i) {
                    const bool ok = pc[v] >= 0 && cc[i] >= 0;
                    ev[v][i] = ok ? __ldg(a.e_val + 3 * (int64_t)(f + v) + mm[i]) : 0.0;
                    sv[v][i] = ok ? __ldg(a.S + (int64_t)pc[v] * a.lds + cc[i]) : 0.0;
                }
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (pc[v] >= 0) {
#pragma unroll
                    for (int i = 0; i < K; ++i) acc[i] = fma(ev[v][i], sv[v][i], acc[i]);
                }
        }
    }
#pragma unroll
    for (int i = 0; i < K; ++i)
        if (cc[i] >= 0) a.W[(3 * row + mm[i]) * a.ldw + cc[i]] = acc[i];
}

// ----------------------------------------------------------------- residuals
// r = w - (A (x) I_R) x with w as the pair (wh, wl), all blocks dense (4 L
// wide); x1 = inv_theta D^-1 r. wh may be r (a lane reads what it writes).
template <int R, int L, int S, int U>
__global__ void __launch_bounds__(kThreads) resid_df_rows_kernel(const ResidDfArgs a) {
    constexpr int ld = 4 * L;
    const Lane p = place<L, S>(a.desc, a.nrows, blockIdx.x);
    const int64_t row = p.d.x;
    const float* const X = a.x + 4 * p.q;
    u64 s[R][2], l[R][2];
#pragma unroll
    for (int k = 0; k < R; ++k) s[k][0] = s[k][1] = l[k][0] = l[k][1] = 0ull;
    int e = p.d.y + p.sp;
    int j[U];
#pragma unroll
    for (int u = 0; u < U; ++u) j[u] = e + u * S < p.d.z ? __ldg(a.col + e + u * S) : -1;
    while (e < p.d.z) {
        float4 x[U][R];
        float vh[U], vl[U];
        bool in[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            in[u] = j[u] >= 0;
#pragma unroll
            for (int k = 0; k < R; ++k)
                x[u][k] = in[u] ? __ldg(reinterpret_cast<const float4*>(X + ((int64_t)R * j[u] + k) * ld))
                                : make_float4(0.f, 0.f, 0.f, 0.f);
            vh[u] = in[u] ? __ldg(a.vh + e + u * S) : 0.f;
            vl[u] = in[u] ? __ldg(a.vl + e + u * S) : 0.f;
        }
        e += U * S;
#pragma unroll
        for (int u = 0; u < U; ++u) j[u] = e + u * S < p.d.z ? __ldg(a.col + e + u * S) : -1;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (in[u]) {
                const u64 ah = pack2(vh[u], vh[u]), al = pack2(vl[u], vl[u]);
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    df_acc2(s[k][0], l[k][0], ah, al, pack2(x[u][k].x, x[u][k].y));
                    df_acc2(s[k][1], l[k][1], ah, al, pack2(x[u][k].z, x[u][k].w));
                }
            }
    }
    constexpr int N = 4 * R;
    float sh[N], sl[N];
#pragma unroll
    for (int k = 0; k < R; ++k)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float2 h = unpack2(s[k][i]), t = unpack2(l[k][i]);
            sh[4 * k + 2 * i] = h.x, sh[4 * k + 2 * i + 1] = h.y;
            sl[4 * k + 2 * i] = t.x, sl[4 * k + 2 * i + 1] = t.y;
        }
    int base, cnt;
    df_scatter<N, S, L>(sh, sl, threadIdx.x & 31, p.sp, base, cnt);
    if (!p.on) return;
    const float d = a.x1 ? __ldg(a.dinv + row) * a.inv_theta : 0.f;
    constexpr int K = Kept<N, S>::n;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        if (i >= cnt) break;
        const int t = base + i;
        const int64_t at = (R * row + (t >> 2)) * ld + 4 * p.q + (t & 3);
        float h = a.wh[at], lo = a.wl[at];
        df_merge(h, lo, -sh[i], -sl[i]);
        const float r = __fadd_rn(h, lo);
        a.r[at] = r;
        if (a.x1) a.x1[at] = d * r;
    }
}

// ----------------------------------------------------------------- launches
namespace {

template <int L, int S>
unsigned blocks(int nrows) {
    constexpr int per = 32 / (S * L) * (kThreads / 32);
    return (unsigned)((nrows + per - 1) / per);
}

template <int L>
int bsr33_go(const Bsr33DfArgs& a, int ng, cudaStream_t s) {
    bsr33_df_rows_kernel<L, 4><<<blocks<L, 4>(a.nrows) * ng, kThreads, 0, s>>>(a, ng);
    count_launch();
    NM_CUDA(cudaGetLastError());
    return NM_OK;
}

template <int R, int L>
int resid_go(const ResidDfArgs& a, cudaStream_t s) {
    resid_df_rows_kernel<R, L, 4, R == 3 ? 3 : 4><<<blocks<L, 4>(a.nrows), kThreads, 0, s>>>(a);
    count_launch();
    NM_CUDA(cudaGetLastError());
    return NM_OK;
}

}  // namespace

int launch_bsr33_df(const Bsr33DfArgs& a, cudaStream_t s) {
    if (a.b < 1 || a.b > 64) return fail(NM_EINVAL, "block width must be in 1..64");
    if (a.nrows == 0) return NM_OK;
    int ng, bg;
    cluster_groups(a.b, &ng, &bg);
    if (a.ldx != ng * bg) return fail(NM_EINVAL, "split block of another width");
    switch (bg / 4) {
        case 1: return bsr33_go<1>(a, ng, s);
        case 2: return bsr33_go<2>(a, ng, s);
        case 3: return bsr33_go<3>(a, ng, s);
        case 4: return bsr33_go<4>(a, ng, s);
        case 5: return bsr33_go<5>(a, ng, s);
        case 6: return bsr33_go<6>(a, ng, s);
        case 7: return bsr33_go<7>(a, ng, s);
        default: return bsr33_go<8>(a, ng, s);
    }
}

int launch_resid_df(int R, const ResidDfArgs& a, int b, cudaStream_t s) {
    if (b < 4 || b > 32 || b % 4) return fail(NM_EINVAL, "residual blocks are 4 .. 32 columns wide");
    if (a.nrows == 0) return NM_OK;
#define NM_RS(N) \
    case N: return R == 3 ? resid_go<3, N>(a, s) : resid_go<1, N>(a, s);
    switch (b / 4) {
        NM_RS(1) NM_RS(2) NM_RS(3) NM_RS(4) NM_RS(5) NM_RS(6) NM_RS(7) NM_RS(8)
    }
#undef NM_RS
    return fail(NM_EINVAL, "unsupported width");
}

// 80-byte records of the blocks of A: nine high parts, nine low parts.
__global__ void df_records_kernel(int64_t n, const double* val, float4* out) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        float v[20];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const double d = val[9 * t + i];
            v[i] = __double2float_rn(d);
            v[9 + i] = __double2float_rn(d - (double)v[i]);
        }
        v[18] = v[19] = 0.f;
#pragma unroll
        for (int i = 0; i < 5; ++i) out[5 * t + i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
}

int launch_df_records(int64_t n, const double* val, float4* out, cudaStream_t s) {
    if (n == 0) return NM_OK;
    df_records_kernel<<<(unsigned)std::min<int64_t>((n + 127) / 128, 1 << 16), 128, 0, s>>>(n, val, out);
    count_launch();
    NM_CUDA(cudaGetLastError());
    return NM_OK;
}

}  // namespace nm
