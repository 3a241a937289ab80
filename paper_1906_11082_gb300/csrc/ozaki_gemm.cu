// FP64-accurate dense products on the tensor cores by operand splitting.
//
// The dense algebra of the filtered block Lanczos (Sec. 6.2) is two product
// shapes over the basis V (n rows, n ~ 1e6):
//   TN:  C (I x J) = alpha X^T Y + beta C,  X: n x I, Y: n x J  (the block
//        Gram-Schmidt coefficients V^T M W, the Ritz projections V^T K V,
//        V^T M V and the Coriolis projection X^T R X, Sec. 7);
//   NN:  D (n x J) = alpha X Y + beta D,    X: n x I, Y: I x J  (W -= V C,
//        the Ritz vectors X = V S).
// GB300's FP64 units run at 1/64 of its float units and its tensor cores
// take no FP64 here, so both run as fp16 tensor-core products of exact
// operand pieces (the error-free splitting of Ozaki, Ogita, Oishi and Rump,
// 2012):
//  - within a contraction chunk of 64 terms, every row i of X and column j
//    of Y gets the exponent E_i (F_j) of its largest entry; an entry becomes
//    the integer N = x 2^(1076 - E) truncated, |N| < 2^54, and N its seven
//    base-256 digits d_0 .. d_6 in [-128, 127] (the bytes of N plus 128 at
//    every digit, less 128: two's complement needs no carry chain);
//  - a digit is exact in fp16, a product of two at most 2^14, and the sum
//    over the chunk of the at most seven digit pairs of one diagonal p + q
//    is below 7 * 64 * 2^14 < 2^24, so the float accumulation of the tensor
//    cores (mma.sync m16n8k16, fp16 in, f32 out) is exact;
//  - the chunk's sum over the diagonals 0 .. 7 (34 products; the diagonals
//    from 8 on weigh 2^-64 of a leading product) is put together in 64-bit
//    integers and added in FP64 with one conversion and one multiply-add.
// The result carries FP64-level error relative to the products of each row's
// and column's largest entries.
// TN splits the long contraction over CTAs into a fixed number of parts
// summed in order by a second kernel, so every result is deterministic.
//
// What bounds it: the FP64 pipe and the splitting before; now the latency of
// cutting operands between products with two warps per scheduler (234 to 254
// registers), not yet the mma.sync rate. With eight 7-bit pieces combined in FP64 per diagonal
// (about 12 FP64 operations per output and chunk) and the splitting redone by
// every warp for every 16 output columns, V^T W at n = 1.15M, 576 x 32 took
// 22.0 ms and V C 23.5 ms. Now a warp holds 16 rows by 32 columns: an X entry
// is cut once (about 20 integer instructions, packed fp16 conversion), a Y
// entry once per CTA into shared memory in fragment order, raw chunks arrive
// by cp.async one chunk ahead: 6.8 ms and 6.0 ms, the mma.sync pipe busy 39 to
// 40% of the time (its limit 2.5 ms each; 10.9 GB for both would take 1.6 ms).
#include <algorithm>
#include <cstdint>

#include <cuda_fp16.h>

#include "kernels.h"
#include "nm_internal.h"

namespace nm {

namespace {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
constexpr int kTileI = 16 * kWarps;    // output rows per CTA (16 per warp)
constexpr int kChunk = 64;             // contraction terms per exact accumulation
constexpr int kDigits = 7;
constexpr int kDiag = 8;               // kept diagonals p + q = 0..7
// shared row strides of the raw chunks (doubles), chosen so that the four
// (k) by eight (row) lanes of a fragment load fall into distinct banks
constexpr int kLdXT = kTileI + 2;      // TN: [k][i]
constexpr int kLdXN = kChunk + 8;      // NN: [i][k]
constexpr int kLdYN = kChunk + 2;      // NN: [j][k]

// Magnitude bits of a double's exponent field for alignment (subnormals and
// zero count as 1), from its high word.
__device__ __forceinline__ int exp_of_hi(int hi) {
    const int e = (hi >> 20) & 0x7FF;
    return e == 0 ? 1 : e;
}

// N + 128 (256^0 + .. + 256^6) of v aligned to exponent E (E >= that of v):
// byte 6 - p is digit p plus 128.
__device__ __forceinline__ uint2 digits_of(double v, int E) {
    const int hi = __double2hiint(v);
    const unsigned lo = (unsigned)__double2loint(v);
    const int e = (hi >> 20) & 0x7FF;
    unsigned mh = (unsigned)hi & 0xFFFFFu;
    if (e != 0) mh |= 0x100000u;
    const int sh = min(E - max(e, 1), 63);
    unsigned long long m = (((unsigned long long)mh << 32) | lo) << 1 >> sh;
    const long long sg = (long long)(hi >> 31);
    m = (m ^ (unsigned long long)sg) - (unsigned long long)sg + 0x80808080808080ull;
    return make_uint2((unsigned)m, (unsigned)(m >> 32));
}

// fp16 pair of digit p of two entries (first entry in the low half).
template <int P>
__device__ __forceinline__ uint32_t digit_pair(const uint2& a, const uint2& b) {
    constexpr unsigned byte = (6 - P) & 3;
    constexpr unsigned sel = byte | (byte << 4) | ((4 + byte) << 8) | ((4 + byte) << 12);
    const unsigned w = P <= 2 ? __byte_perm(a.y, b.y, sel) : __byte_perm(a.x, b.x, sel);
    const unsigned h = (w & 0x00FF00FFu) | 0x64006400u;   // 1024 + byte
    const __half2 d = __hadd2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half((unsigned short)0xE480)));
    return *reinterpret_cast<const uint32_t*>(&d);        // - 1152
}

__device__ __forceinline__ void mma_f16(float* c, const uint32_t* a, const uint2& b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// 16 (or two times 8) bytes global -> shared, zeros where !ok.
__device__ __forceinline__ void copy2(double* dst, const double* src, bool wide, bool ok0, bool ok1) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (wide && ok0 == ok1) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok0 ? 16 : 0));
    } else {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(ok0 ? 8 : 0));
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d + 8), "l"(src + 1), "r"(ok1 ? 8 : 0));
    }
}

struct Shape {
    // X(i, k) = NN ? X[i * ldx + k] : X[k * ldx + i]
    // Y(k, j) = NN ? Y[k + j * ldy] : Y[k * ldy + j]
    const double* X;
    int64_t ldx;
    const double* Y;
    int64_t ldy;
    int64_t I, J, K;       // output rows, columns, contraction length
    int64_t chunks_per_part;   // 64-term chunks summed into one part
    int64_t parts_per_cta;     // consecutive parts of one CTA (grid z)
    int widex, widey;      // 16-byte copies allowed (alignment of base and stride)
    // output: part p of TN writes P[p][i + j * I]; NN writes D
    double* P;
    double* D;
    int64_t ldd;
    double alpha, beta;
};

template <bool NN, int NJ>
constexpr size_t ozaki_smem() {
    const size_t x = NN ? kTileI * kLdXN : kChunk * kLdXT;
    const size_t y = NN ? 8 * NJ * kLdYN : kChunk * 8 * NJ;
    return 2 * (x + y) * 8 + (size_t)kDigits * (kChunk / 16) * NJ * 32 * 8 + (8 + 1) * 8 * NJ * 4;
}

// One CTA: output rows i0 .. i0 + 127, columns j0 .. j0 + 8 NJ - 1,
// contraction terms [k_begin, k_end) in chunks of 64.
template <bool NN, int NJ>
__global__ void __launch_bounds__(kThreads, 1) ozaki_kernel(const Shape sh) {
    constexpr int JT = 8 * NJ;
    constexpr int XS = NN ? kTileI * kLdXN : kChunk * kLdXT;
    constexpr int YS = NN ? JT * kLdYN : kChunk * JT;
    extern __shared__ double oz_smem[];
    double* const xs = oz_smem;                                   // [2][XS]
    double* const ys = xs + 2 * XS;                               // [2][YS]
    uint2* const bs = reinterpret_cast<uint2*>(ys + 2 * YS);      // [digit][k16][n8][lane]
    int* const fpart = reinterpret_cast<int*>(bs + kDigits * (kChunk / 16) * NJ * 32);   // [8][JT]
    int* const Fy = fpart + 8 * JT;                               // [JT]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int gid = lane >> 2, tig = lane & 3;
    const int64_t i0 = (int64_t)blockIdx.x * kTileI;
    const int64_t j0 = (int64_t)blockIdx.y * JT;
    const int64_t k_cta = sh.parts_per_cta * sh.chunks_per_part * kChunk;
    const int64_t k_begin = blockIdx.z * k_cta;
    const int64_t k_end = sh.K < k_begin + k_cta ? sh.K : k_begin + k_cta;
    int64_t part = blockIdx.z * sh.parts_per_cta;
    int left = (int)sh.chunks_per_part;                    // chunks until the part is written
    const int nchunk = (int)((k_end - k_begin + kChunk - 1) / kChunk);

    auto fetch = [&](int ch) {
        const int64_t k0 = k_begin + (int64_t)ch * kChunk;
        double* x = xs + (ch & 1) * XS;
        double* y = ys + (ch & 1) * YS;
        if (NN) {
#pragma unroll 4
            for (int t = tid; t < kTileI * (kChunk / 2); t += kThreads) {
                const int i = t / (kChunk / 2), k = 2 * (t % (kChunk / 2));
                const int64_t gi = i0 + i, gk = k0 + k;
                const bool r = gi < sh.I, ok0 = r && gk < k_end, ok1 = r && gk + 1 < k_end;
                copy2(x + i * kLdXN + k, ok0 ? sh.X + gi * sh.ldx + gk : sh.X, sh.widex, ok0, ok1);
            }
            for (int t = tid; t < JT * (kChunk / 2); t += kThreads) {
                const int j = t / (kChunk / 2), k = 2 * (t % (kChunk / 2));
                const int64_t gj = j0 + j, gk = k0 + k;
                const bool r = gj < sh.J, ok0 = r && gk < k_end, ok1 = r && gk + 1 < k_end;
                copy2(y + j * kLdYN + k, ok0 ? sh.Y + gj * sh.ldy + gk : sh.Y, sh.widey, ok0, ok1);
            }
        } else {
#pragma unroll 4
            for (int t = tid; t < kChunk * (kTileI / 2); t += kThreads) {
                const int k = t / (kTileI / 2), i = 2 * (t % (kTileI / 2));
                const int64_t gk = k0 + k, gi = i0 + i;
                const bool r = gk < k_end, ok0 = r && gi < sh.I, ok1 = r && gi + 1 < sh.I;
                copy2(x + k * kLdXT + i, ok0 ? sh.X + gk * sh.ldx + gi : sh.X, sh.widex, ok0, ok1);
            }
            for (int t = tid; t < kChunk * (JT / 2); t += kThreads) {
                const int k = t / (JT / 2), j = 2 * (t % (JT / 2));
                const int64_t gk = k0 + k, gj = j0 + j;
                const bool r = gk < k_end, ok0 = r && gj < sh.J, ok1 = r && gj + 1 < sh.J;
                copy2(y + k * JT + j, ok0 ? sh.Y + gk * sh.ldy + gj : sh.Y, sh.widey, ok0, ok1);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    double out[NJ][4];
#pragma unroll
    for (int n = 0; n < NJ; ++n)
#pragma unroll
        for (int r = 0; r < 4; ++r) out[n][r] = 0.0;
    const int ra = 16 * warp + gid;                        // this lane's rows ra, ra + 8
    const bool busy = i0 + 16 * warp < sh.I;               // the warp has rows at all
    if (nchunk > 0) fetch(0);
    for (int ch = 0; ch < nchunk; ++ch) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                                   // chunk ch is here, chunk ch - 1 is consumed
        if (ch + 1 < nchunk) fetch(ch + 1);
        const double* x = xs + (ch & 1) * XS;
        const double* y = ys + (ch & 1) * YS;
        auto yat = [&](int k, int j) { return NN ? y[j * kLdYN + k] : y[k * JT + j]; };
        // largest exponents of the columns of Y: eight runs of eight terms
        for (int t = tid; t < 8 * JT; t += kThreads) {
            const int j = t % JT, r = t / JT;
            int m = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) m = max(m, __double2hiint(yat(8 * r + k, j)) & 0x7FFFFFFF);
            fpart[r * JT + j] = exp_of_hi(m);
        }
        // ... and of this lane's two rows of X (over the four lanes of a row)
        auto xat = [&](int r, int k) { return NN ? x[r * kLdXN + k] : x[k * kLdXT + r]; };
        int Ea = 0, Eb = 0;
        if (busy) {
#pragma unroll 4
            for (int s = 0; s < kChunk / 4; ++s) {
                const int k = 16 * (s >> 2) + 8 * ((s >> 1) & 1) + 2 * tig + (s & 1);
                Ea = max(Ea, __double2hiint(xat(ra, k)) & 0x7FFFFFFF);
                Eb = max(Eb, __double2hiint(xat(ra + 8, k)) & 0x7FFFFFFF);
            }
#pragma unroll
            for (int o = 1; o <= 2; o *= 2) {
                Ea = max(Ea, __shfl_xor_sync(0xffffffffu, Ea, o));
                Eb = max(Eb, __shfl_xor_sync(0xffffffffu, Eb, o));
            }
        }
        Ea = exp_of_hi(Ea);
        Eb = exp_of_hi(Eb);
        __syncthreads();
        // digits of Y in fragment order: word (k pair, column) of digit q
        for (int t = tid; t < JT * (kChunk / 2); t += kThreads) {
            const int j = t % JT, kp = t / JT;
            int F = fpart[j];
#pragma unroll
            for (int r = 1; r < 8; ++r) F = max(F, fpart[r * JT + j]);
            if (kp == 0) Fy[j] = F;
            const uint2 a = digits_of(yat(2 * kp, j), F), b = digits_of(yat(2 * kp + 1, j), F);
            const int ks = kp >> 3, half = (kp >> 2) & 1, ln = (j & 7) * 4 + (kp & 3);
            uint32_t* w = reinterpret_cast<uint32_t*>(bs + (ks * NJ + (j >> 3)) * 32 + ln) + half;
            constexpr int q = 2 * (kChunk / 16) * NJ * 32;   // words per digit
            w[0 * q] = digit_pair<0>(a, b);
            w[1 * q] = digit_pair<1>(a, b);
            w[2 * q] = digit_pair<2>(a, b);
            w[3 * q] = digit_pair<3>(a, b);
            w[4 * q] = digit_pair<4>(a, b);
            w[5 * q] = digit_pair<5>(a, b);
            w[6 * q] = digit_pair<6>(a, b);
        }
        __syncthreads();
        if (!busy) continue;
        float acc[kDiag][NJ][4];
#pragma unroll
        for (int d = 0; d < kDiag; ++d)
#pragma unroll
            for (int n = 0; n < NJ; ++n)
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[d][n][r] = 0.f;
#pragma unroll 1
        for (int ks = 0; ks < kChunk / 16; ++ks) {
            // A fragments of the digits: rows (ra, ra + 8), k = 16 ks + 2 tig + {0, 1} (+ 8)
            uint32_t a[kDigits][4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int r = ra + ((h & 1) ? 8 : 0), E = (h & 1) ? Eb : Ea;
                const int k = 16 * ks + 2 * tig + ((h & 2) ? 8 : 0);
                const uint2 d0 = digits_of(xat(r, k), E), d1 = digits_of(xat(r, k + 1), E);
                a[0][h] = digit_pair<0>(d0, d1);
                a[1][h] = digit_pair<1>(d0, d1);
                a[2][h] = digit_pair<2>(d0, d1);
                a[3][h] = digit_pair<3>(d0, d1);
                a[4][h] = digit_pair<4>(d0, d1);
                a[5][h] = digit_pair<5>(d0, d1);
                a[6][h] = digit_pair<6>(d0, d1);
            }
#pragma unroll
            for (int n = 0; n < NJ; ++n) {
                uint2 b[kDigits];
#pragma unroll
                for (int q = 0; q < kDigits; ++q) b[q] = bs[((q * (kChunk / 16) + ks) * NJ + n) * 32 + lane];
#pragma unroll
                for (int q = 0; q < kDigits; ++q)
#pragma unroll
                    for (int p = 0; p < kDigits; ++p)
                        if (p + q < kDiag) mma_f16(acc[p + q][n], a[p], b[q]);
            }
        }
        // exact chunk sums: diagonal d weighs 2^(96 - 8 d) in units of
        // 2^(E + F - 2152); v counts units of 2^52 of those, rounded (a floor
        // here biases every chunk: relative error 1.7e-15 at 65,536 normal terms)
#pragma unroll
        for (int n = 0; n < NJ; ++n)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                auto D = [&](int d) { return (long long)__float2int_rn(acc[d][n][r]); };
                const long long top = (((D(0) * 256 + D(1)) * 256 + D(2)) * 256) + D(3);
                const long long low = (((D(4) * 256 + D(5)) * 256 + D(6)) * 256) + D(7);
                const double v = (double)(top * (1 << 20) + ((low + 2048) >> 12));
                const int e = ((r < 2) ? Ea : Eb) + Fy[8 * n + 2 * tig + (r & 1)] - 2100;
                if (e > -1023 && e < 1024)
                    out[n][r] = fma(v, __hiloint2double((e + 1023) << 20, 0), out[n][r]);
                else
                    out[n][r] += ldexp(v, e);
            }
        // TN: a finished part goes to the workspace
        if (!NN && (--left == 0 || ch + 1 == nchunk)) {
#pragma unroll
            for (int n = 0; n < NJ; ++n)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int64_t i = i0 + ra + ((r >= 2) ? 8 : 0);
                    const int64_t j = j0 + 8 * n + 2 * tig + (r & 1);
                    if (i < sh.I && j < sh.J) sh.P[part * sh.I * sh.J + i + j * sh.I] = out[n][r];
                    out[n][r] = 0.0;
                }
            ++part;
            left = (int)sh.chunks_per_part;
        }
    }
    // NN: D (alpha, beta applied)
    if constexpr (NN) {
#pragma unroll
        for (int n = 0; n < NJ; ++n)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int64_t i = i0 + ra + ((r >= 2) ? 8 : 0);
                const int64_t j = j0 + 8 * n + 2 * tig + (r & 1);
                if (i >= sh.I || j >= sh.J) continue;
                double* d = sh.D + i * sh.ldd + j;
                *d = sh.alpha * out[n][r] + (sh.beta == 0.0 ? 0.0 : sh.beta * *d);
            }
    }
}

// C[i + j ldc] = alpha sum_p P[p][i + j I] + beta C, in a fixed order: runs of
// 16 parts, then the runs.
__global__ void ozaki_reduce_kernel(int64_t I, int64_t J, int parts, const double* P, double alpha, double beta,
                                    double* C, int64_t ldc) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < I * J; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t % I, j = t / I;
        double s = 0.0;
        for (int p0 = 0; p0 < parts; p0 += 16) {
            double v[16], r = 0.0;
#pragma unroll
            for (int p = 0; p < 16; ++p) v[p] = p0 + p < parts ? P[(int64_t)(p0 + p) * I * J + t] : 0.0;
#pragma unroll
            for (int p = 0; p < 16; ++p) r += v[p];
            s += r;
        }
        double* c = C + i + j * ldc;
        *c = alpha * s + (beta == 0.0 ? 0.0 : beta * *c);
    }
}

int g_sms = 0;

int sm_count() {
    if (!g_sms) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            g_sms = 148;
    }
    return g_sms;
}

int wide(const void* p, int64_t ld) { return ((uintptr_t)p & 15) == 0 && ld % 2 == 0; }

template <bool NN, int NJ>
int ozaki_go(const Shape& sh, int64_t ti, int64_t nz, cudaStream_t s) {
    const int64_t tj = (sh.J + 8 * NJ - 1) / (8 * NJ);
    if (ti > 0x7FFFFFFF || tj > 65535) return fail(NM_EINVAL, "product too large for one launch");
    constexpr size_t smem = ozaki_smem<NN, NJ>();
    NM_CUDA(cudaFuncSetAttribute(ozaki_kernel<NN, NJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    ozaki_kernel<NN, NJ><<<dim3((unsigned)ti, (unsigned)tj, (unsigned)nz), kThreads, smem, s>>>(sh);
    count_launch();
    NM_CUDA(cudaGetLastError());
    return NM_OK;
}

// Column tile: as narrow as the product (8 or 16 columns), else 32.
template <bool NN>
int ozaki_launch(const Shape& sh, int64_t ti, int64_t nz, cudaStream_t s) {
    if (sh.J <= 8) return ozaki_go<NN, 1>(sh, ti, nz, s);
    if (sh.J <= 16) return ozaki_go<NN, 2>(sh, ti, nz, s);
    return ozaki_go<NN, 4>(sh, ti, nz, s);
}

}  // namespace

// C (I x J, column-major, ldc) = alpha X^T Y + beta C with X: K x I and Y:
// K x J row-major (ldx, ldy). The workspace of the split parts belongs to
// the context (grown on demand, reused).
int ozaki_gemm_tn(nm_ctx* ctx, cudaStream_t s, int64_t I, int64_t J, int64_t K, double alpha, const double* X,
                  int64_t ldx, const double* Y, int64_t ldy, double beta, double* C, int64_t ldc) {
    if (I <= 0 || J <= 0) return NM_OK;
    const int jt = J <= 8 ? 8 : J <= 16 ? 16 : 32;
    const int64_t ti = (I + kTileI - 1) / kTileI, tj = (J + jt - 1) / jt;
    const int64_t chunks = std::max<int64_t>((K + kChunk - 1) / kChunk, 1);
    // One CTA per SM in all. A CTA's terms are summed in parts of at most 32
    // chunks, since one running FP64 sum over all of them rounds once per
    // chunk; longer parts where the workspace would pass 64 MB.
    const int64_t ctas = std::max<int64_t>(1, std::min<int64_t>(chunks, sm_count() / (ti * tj)));
    const int64_t per_cta = (chunks + ctas - 1) / ctas;
    const int64_t room = std::max<int64_t>(1, (64ll << 20) / (8 * I * J * ctas));
    const int64_t ppc = std::min<int64_t>((per_cta + 31) / 32, room), cpp = (per_cta + ppc - 1) / ppc;
    const int64_t nz = (chunks + ppc * cpp - 1) / (ppc * cpp);
    const int64_t parts = std::max<int64_t>(1, (chunks + cpp - 1) / cpp);
    const size_t need = (size_t)parts * I * J * sizeof(double);
    if (ctx->gemm_ws.bytes < need) NM_TRY(ctx->gemm_ws.alloc(need));
    Shape sh{X, ldx, Y, ldy, I, J, K, cpp, ppc, wide(X, ldx), wide(Y, ldy), ctx->gemm_ws.as<double>(), nullptr, 0, 1.0, 0.0};
    if (K > 0) {
        NM_TRY(ozaki_launch<false>(sh, ti, nz, s));
    } else {
        NM_CUDA(cudaMemsetAsync(ctx->gemm_ws.p, 0, need, s));
    }
    const int64_t tot = I * J;
    ozaki_reduce_kernel<<<(unsigned)std::min<int64_t>((tot + 255) / 256, 4096), 256, 0, s>>>(
        I, J, (int)parts, ctx->gemm_ws.as<double>(), alpha, beta, C, ldc);
    count_launch();
    NM_CUDA(cudaGetLastError());
    return NM_OK;
}

// D (I x J, row-major, ldd) = alpha X Y + beta D with X: I x K row-major
// (ldx) and Y: K x J column-major (ldy).
int ozaki_gemm_nn(cudaStream_t s, int64_t I, int64_t J, int64_t K, double alpha, const double* X, int64_t ldx,
                  const double* Y, int64_t ldy, double beta, double* D, int64_t ldd) {
    if (I <= 0 || J <= 0) return NM_OK;
    Shape sh{X, ldx, Y, ldy, I, J, K, (K + kChunk - 1) / kChunk + 1, 1, wide(X, ldx), wide(Y, ldy), nullptr, D, ldd, alpha, beta};
    return ozaki_launch<true>(sh, (I + kTileI - 1) / kTileI, 1, s);
}

}  // namespace nm
