// iso_frame.cu -- the frame-space ISO-Merger of one weight matrix (App. E)
// on one GPU.
//
// Given the thin SVDs W_0 = U_0 S_0 V_0^T (base) and W_i = U_i S_i V_i^T
// (experts, i = 1..K; their spectra are not used), the merge is
//   s_ik   = sign(<u_0k, u_ik>), sign(0) := 1                  (Sign canonicalization)
//   xi_Fi  = Pi_{F_0}(s_i F_i - F_0) D_keep,  F in {U, V}       (Stiefel tangent projection,
//            Pi_{F_0}(X) = X - F_0 sym(F_0^T X)                  Top-k_keep masking)
//   g_i    = xi_Ui S_0 V_0^T + U_0 S_0 xi_Vi^T, Gamma_ij = <g_i, g_j>_F
//   c*     = clip((Gamma + ridge I)^-1 diag Gamma)              (Retention coefficients)
//   xi_F*  = Pi_{F_0}(sum_i c*_i xi_Fi),  F* = polar(F_0 + xi_F*) (Retraction and
//   W*     = U* S_0 V*^T                                          reconstruction)
//
// How it is computed here (every identity below is pinned against the binary64
// oracle of the same definitions):
// * Nothing of size m x n is formed but the output.  With A_i = F_0^T dF_i
//   (dF_i = s_i F_i - F_0), Sym_i = sym(A_i), Kw_i = A_i - Sym_i:
//     F_0^T xi_Fi = Kw_i D,
//     (xi_Fi^T xi_Fj)_kk = D_k [(dF_i^T dF_j)_kk - (A_i^T Sym_j)_kk - (Sym_i A_j)_kk + (Sym_i Sym_j)_kk],
//     Gamma_ij = sum_k s_k^2 [(xi_Ui^T xi_Uj)_kk + (xi_Vi^T xi_Vj)_kk]
//                - sum_kl s_k s_l D_k D_l (KwU_i KwV_j + KwU_j KwV_i)[k, l],
//     xi_F* = D dF_c - F_0 Y,  dF_c = sum_i c*_i dF_i,
//     Y = (sum_i c*_i Sym_i) D + sym((sum_i c*_i Kw_i) D).
// * polar(F_0 + xi) = (F_0 + xi)(I + xi^T xi)^(-1/2), since F_0^T xi is skew;
//   the inverse square root comes from the coupled Newton-Schulz iteration
//   written in differences from the identity (Y = I + y, Z = I + z), so that
//   every product is of small matrices, scaled when ||xi^T xi||_F >= 0.9.
// * W* = W_0 + [E_U S_0 | U_0 S_0] [V* | E_V]^T with E_F = F* - F_0: the
//   difference form keeps the low-precision products on the small motion;
//   W_0 itself (the caller's matrix) replaces U_0 S_0 V_0^T.
// * Precision.  A_i = F_0^T dF_i to binary64: on dense spectra the frames
//   rotate far inside near-degenerate singular subspaces while the proxies
//   stay small, so Gamma is a difference of terms up to thousands of times
//   larger than itself (the paper takes the merge in binary64 throughout).
//   It runs on the tensor cores all the same, from exact 8-bit slices of the
//   columns (k_oz_gemm), as the optimizer step's F^T F does.  The other large
//   contractions (F_0 Y, xi*^T xi*, the Newton-Schulz products,
//   (F_0 + xi*) R and the reconstruction) are three tf32 products per pair
//   (hi hi + hi lo + lo hi, x = hi + lo split in binary64; k_gemm_x3) with
//   binary32 accumulation, about 2^-22 relative per product; what they feed
//   is the merged frame, whose error reaches W* only through products with
//   the small motion.  Everything else is binary64 on the CUDA cores.
#include "iso_gemm.cuh"
#include "iso_internal.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <vector>

namespace iso {

namespace {

constexpr int FR_PAD = 128;        // operand arrays padded to whole GEMM tiles
constexpr int FR_MAX_NS = 64;      // Newton-Schulz iteration limit
constexpr int FR_DEFAULT_NS = 16;
constexpr double FR_NS_TOL = 1e-9; // max |y + z + z y| at which the iteration has converged

long long pad_up(long long x) { return (x + FR_PAD - 1) / FR_PAD * FR_PAD; }

struct FrameHeader {
    int32_t status;
    int32_t conv[2];                // per side: the Newton-Schulz iteration has converged
    int32_t pad;
    double nu2[2];                  // per side: ||xi^T xi||_F^2
    double cs[2];                   // per side: the scaling of I + xi^T xi
    uint32_t wmax[2][FR_MAX_NS];    // per side and iteration: max |w| as binary32 bits
};

// Conversions between binary64 and binary32 / tf32 in integer arithmetic: the
// conversion instructions run at the binary64 rate, a thirtieth of the integer
// rate here, and the element-wise kernels below were bound by them.
// binary32 -> binary64
__device__ __forceinline__ double widen(float x) {
    if (!(fabsf(x) <= 3.402823466e38f)) return (double)x;
    const bool sub = fabsf(x) < 1.17549435e-38f;                     // scaled into the normal range first
    const uint32_t u = __float_as_uint(sub ? x * 0x1p64f : x), m = u & 0x7FFFFFFFu;
    const uint32_t h = m ? (m >> 3) + (sub ? 0x38000000u - (64u << 20) : 0x38000000u) : 0u;
    return __hiloint2double((int)((u & 0x80000000u) | h), (int)(m << 29));
}
// binary64 -> (hi, lo) with hi a tf32 value (x to binary32, nearest even, then
// to nearest, ties away) and lo the tf32 value nearest to the rest, so that
// hi + lo = x to about 2^-22 |x|.  From 2^-73 to 2^127 the two roundings are
// integer operations on the high word (the first one matters only where it
// carries into it, from a low word of 0xF0000000 on), and lo, a multiple of
// x's last place, is zero or a normal number; everything else takes the
// conversions themselves.
__device__ __forceinline__ uint32_t tf32_high(double x) {            // the magnitude's high word; the low one is 0
    return (((uint32_t)__double2hiint(x) & 0x7FFFFFFFu) + 0x200u + ((uint32_t)__double2loint(x) >= 0xF0000000u ? 1u : 0u)) & ~0x3FFu;
}
__device__ __forceinline__ float tf32_cvt(double x) {
    float f;
    asm("{\n\t.reg .b32 t;\n\tcvt.rna.tf32.f32 t, %1;\n\tmov.b32 %0, t;\n\t}" : "=f"(f) : "f"((float)x));
    return f;
}
__device__ __forceinline__ void split_tf32(double x, float& hi, float& lo) {
    const uint32_t hx = (uint32_t)__double2hiint(x), m = hx & 0x7FFFFFFFu, sx = hx & 0x80000000u;
    if (m - 0x3B600000u < 0x47E00000u - 0x3B600000u) {
        const uint32_t r = tf32_high(x);
        hi = __uint_as_float(sx | (r - 0x38000000u) << 3);
        const double rest = x - __hiloint2double((int)(sx | r), 0);
        const uint32_t l = tf32_high(rest);
        lo = __uint_as_float(((uint32_t)__double2hiint(rest) & 0x80000000u) | (l ? (l - 0x38000000u) << 3 : 0u));
    } else if ((m | (uint32_t)__double2loint(x)) == 0) {
        hi = lo = 0.0f;
    } else {
        hi = tf32_cvt(x);
        lo = tf32_cvt(x - (double)hi);
    }
}

// The same three steps for the Newton-Schulz iterates, which are differences
// from the identity: what lies below 2^-126 there is far below the rounding of
// the products it enters, and becomes 0 without a branch (the iteration of a
// 3584 x 18944 merge 9.5 ms, 11.0 ms with the exact forms above).
__device__ __forceinline__ double ns_widen(float x) {
    const uint32_t u = __float_as_uint(x), m = u & 0x7FFFFFFFu;
    if (m >= 0x7F800000u) return (double)x;
    const uint32_t h = m < 0x00800000u ? 0u : (m >> 3) + 0x38000000u;
    return __hiloint2double((int)((u & 0x80000000u) | h), m < 0x00800000u ? 0 : (int)(m << 29));
}
__device__ __forceinline__ double halve(double x) {
    const uint32_t h = (uint32_t)__double2hiint(x), m = h & 0x7FFFFFFFu;
    if (m >= 0x7FF00000u) return x;
    return m < 0x00200000u ? 0.0 : __hiloint2double((int)(h - 0x00100000u), __double2loint(x));
}
__device__ __forceinline__ float ns_tf32(double x, uint32_t& hw_out) {
    const uint32_t hx = (uint32_t)__double2hiint(x), sx = hx & 0x80000000u;
    uint32_t r = tf32_high(x);
    r = r < 0x38100000u ? 0u : r;
    hw_out = sx | r;
    if (r >= 0x47F00000u) return __uint_as_float(sx | ((hx & 0x7FFFFFFFu) > 0x7FF00000u ? 0x7FC00000u : 0x7F800000u));
    return __uint_as_float(sx | (r ? (r - 0x38000000u) << 3 : 0u));
}

// An operand row of contraction length L (padded) is stored as two segments [hi | lo].
__device__ __forceinline__ void put_split(float* row, long long L, long long k, double x) {
    float hi, lo;
    split_tf32(x, hi, lo);
    row[k] = hi;
    row[L + k] = lo;
}

struct Frames {                     // one side (U: d = m; V: d = n), d x q row-major binary64
    const double* F0;
    const double* F[MAXK];
    int K;
    long long d, q;
};

// ---------------------------------------------------------------------------
// layout helpers
// ---------------------------------------------------------------------------
// out (C x R) = in (R x C)^T, binary64, 32 x 32 tiles
__global__ void __launch_bounds__(256) k_fr_transpose(const double* in, double* out, long long R, long long C) {
    pdl_enter();
    __shared__ double t[32][33];
    const long long r0 = (long long)blockIdx.y * 32, c0 = (long long)blockIdx.x * 32;
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long r = r0 + y, c = c0 + threadIdx.x;
        t[y][threadIdx.x] = (r < R && c < C) ? in[r * C + c] : 0.0;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long c = c0 + y, r = r0 + threadIdx.x;
        if (c < C && r < R) out[c * R + r] = t[threadIdx.x][y];
    }
}

// s_ik = sign(<u_0k, u_ik>): the column dot products (U side), summed into dots[i][k]
__global__ void __launch_bounds__(256) k_fr_signdots(Frames f, double* dots, int row_chunks) {
    pdl_enter();
    __shared__ double red[8][33];
    const long long k = (long long)blockIdx.x * 32 + threadIdx.x;
    const int i = blockIdx.y;
    const long long per = (f.d + row_chunks - 1) / row_chunks;
    const long long r0 = (long long)blockIdx.z * per, r1 = min(f.d, r0 + per);
    double acc = 0.0;
    if (k < f.q)
        for (long long r = r0 + threadIdx.y; r < r1; r += 8) acc = fma(f.F0[r * f.q + k], f.F[i][r * f.q + k], acc);
    red[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y == 0 && k < f.q) {
        double s = 0.0;
        for (int y = 0; y < 8; ++y) s += red[y][threadIdx.x];
        atomicAdd(&dots[(long long)i * f.q + k], s);
    }
}

__device__ __forceinline__ double sign_of(const double* dots, long long q, int i, long long k) {
    return dots[(long long)i * q + k] < 0.0 ? -1.0 : 1.0;
}

// (dF_i^T dF_j)_kk for i <= j, summed into cd[i][j][k]; KC >= K is the
// compile-time bound (a bound of 8 for any K spent 36 products a row: 6.1 ms
// for three experts of a 3584 x 18944 matrix)
template <int KC>
__global__ void __launch_bounds__(256) k_fr_coldots(Frames f, const double* dots, double* cd, int row_chunks) {
    pdl_enter();
    __shared__ double red[8][33];
    const long long k = (long long)blockIdx.x * 32 + threadIdx.x;
    const int K = f.K;
    const long long per = (f.d + row_chunks - 1) / row_chunks;
    const long long r0 = (long long)blockIdx.y * per, r1 = min(f.d, r0 + per);
    double acc[KC * (KC + 1) / 2];
#pragma unroll
    for (int p = 0; p < KC * (KC + 1) / 2; ++p) acc[p] = 0.0;
    double sg[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) sg[i] = (i < K && k < f.q) ? sign_of(dots, f.q, i, k) : 0.0;
    if (k < f.q) {
#pragma unroll 2
        for (long long r = r0 + threadIdx.y; r < r1; r += 8) {
            const double f0 = f.F0[r * f.q + k];
            double dv[KC];
#pragma unroll
            for (int i = 0; i < KC; ++i) dv[i] = (i < K) ? fma(sg[i], f.F[i][r * f.q + k], -f0) : 0.0;
            int p = 0;
#pragma unroll
            for (int i = 0; i < KC; ++i)
#pragma unroll
                for (int j = i; j < KC; ++j) acc[p] = fma(dv[i], dv[j], acc[p]), ++p;
        }
    }
    int p = 0;
#pragma unroll
    for (int i = 0; i < KC; ++i)
#pragma unroll
        for (int j = i; j < KC; ++j, ++p) {
            if (i >= K || j >= K) continue;
            red[threadIdx.y][threadIdx.x] = acc[p];
            __syncthreads();
            if (threadIdx.y == 0 && k < f.q) {
                double s = 0.0;
                for (int y = 0; y < 8; ++y) s += red[y][threadIdx.x];
                atomicAdd(&cd[((long long)i * K + j) * f.q + k], s);
            }
            __syncthreads();
        }
}

// Transposed split operand out[k][seg][j] (Qp rows of 2 Dp) of the d x q
// matrix X, j its row, or of X S_0 (S0 given)
struct SplitT {
    long long d, q;
    const double* X;
    const double* S0;      // optional column factors
    float* out;
    long long Dp, Qp;
};
__global__ void __launch_bounds__(256) k_fr_split_t(SplitT a) {
    pdl_enter();
    __shared__ double t[32][33];
    const long long r0 = (long long)blockIdx.x * 32, k0 = (long long)blockIdx.y * 32;
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long r = r0 + y, k = k0 + threadIdx.x;
        double v = 0.0;
        if (r < a.d && k < a.q) {
            v = a.X[r * a.q + k];
            if (a.S0) v *= a.S0[k];
        }
        t[y][threadIdx.x] = v;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long k = k0 + y, r = r0 + threadIdx.x;
        if (k < a.Qp && r < a.Dp) put_split(a.out + k * 2 * a.Dp, a.Dp, r, t[threadIdx.x][y]);
    }
}

// Row-major split operand out[r][seg][c] (rows_p rows of 2 Lp), element value by mode:
//   0  F_0[r, c]                          (d x q)
//   1  F_0[r, c] + X[r, c]                (d x q)
//   3  Y^T[r, c] of the aggregate          (q x q)
//   4  [E_U S_0 | U_0 S_0]                (m x 2 Qp: c < Qp from X = E_U, else U_0)
//   5  [V_0 + E_V | E_V]                  (n x 2 Qp: X = E_V)
//   6  R = (z + (1 - sqrt cs) I) / sqrt cs (q x q, M = z)
struct SplitR {
    Frames f;
    const double* X;
    const double* M;
    const double* S0;
    const double* sym;     // mode 3: K arrays q x q (Sym_i), then K arrays (Kw_i)
    const double* kw;
    const double* coef;
    const FrameHeader* hdr;
    int side;
    long long k_keep;
    int mode;
    float* out;
    long long rows, rows_p, Lp;
};
__global__ void __launch_bounds__(256) k_fr_split_r(SplitR a) {
    pdl_enter();
    const long long q = a.f.q;
    for (long long r = blockIdx.x; r < a.rows_p; r += gridDim.x)
    for (long long c = threadIdx.x; c < a.Lp; c += blockDim.x) {
        double v = 0.0;
        if (r < a.rows) {
            switch (a.mode) {
                case 0: if (c < q) v = a.f.F0[r * q + c]; break;
                case 1: if (c < q) v = a.f.F0[r * q + c] + a.X[r * q + c]; break;
                case 3:
                    if (c < q) {
                        // Y^T[j, k] = Y[k, j] = Sc[j, k] D_j - Kwc[j, k] (D_j - D_k) / 2
                        const double Dj = r < a.k_keep ? 1.0 : 0.0, Dk = c < a.k_keep ? 1.0 : 0.0;
                        double sc = 0.0, kc = 0.0;
                        for (int i = 0; i < a.f.K; ++i) {
                            sc = fma(a.coef[i], a.sym[((long long)i * q + r) * q + c], sc);
                            kc = fma(a.coef[i], a.kw[((long long)i * q + r) * q + c], kc);
                        }
                        v = sc * Dj - 0.5 * kc * (Dj - Dk);
                    }
                    break;
                case 4: {
                    const long long Qp = a.Lp / 2;
                    if (c < Qp) { if (c < q) v = a.X[r * q + c] * a.S0[c]; }
                    else if (c - Qp < q) v = a.f.F0[r * q + (c - Qp)] * a.S0[c - Qp];
                    break;
                }
                case 5: {
                    const long long Qp = a.Lp / 2;
                    if (c < Qp) { if (c < q) v = a.f.F0[r * q + c] + a.X[r * q + c]; }
                    else if (c - Qp < q) v = a.X[r * q + (c - Qp)];
                    break;
                }
                case 6:
                    if (c < q) {
                        const double sc = sqrt(a.hdr->cs[a.side]);
                        v = (a.M[r * q + c] + (r == c ? 1.0 - sc : 0.0)) / sc;
                    }
                    break;
            }
        }
        put_split(a.out + r * 2 * a.Lp, a.Lp, c, v);
    }
}

// ---------------------------------------------------------------------------
// Exact-slice operands (iso_gemm.cuh) of binary64 columns.  Source z of a
// call: 0 the first operand's columns (F_0, or F_0 + X), 1 + i the columns of
// dF_i = s_i F_i - F_0.
// ---------------------------------------------------------------------------
struct OzSrc {
    Frames f;
    const double* dots;
    const double* X;                 // optional: operand 0 is F_0 + X
    unsigned long long* mx;          // [1 + K][q] largest |bits| of each column (zeroed by the caller)
    int32_t* ex;                     // [1 + K][Qp] column exponents
    long long Qp;
    int32_t* peaked;                 // [1 + K][1 + q]: how many columns are left to binary64, and which
    const double* cd;                // [K][K][q] column dots of the dF (their squared norms on the diagonal)
};
// entry e of source z (sg: the column's sign s_ik, for z > 0)
__device__ __forceinline__ double oz_signed(const OzSrc& a, int z, long long e, double sg) {
    if (z == 0) return a.X ? a.f.F0[e] + a.X[e] : a.f.F0[e];
    return fma(sg, a.f.F[z - 1][e], -a.f.F0[e]);
}
__device__ __forceinline__ double oz_value(const OzSrc& a, int z, long long e, long long k) {
    return oz_signed(a, z, e, z ? sign_of(a.dots, a.f.q, z - 1, k) : 0.0);
}

// every column's largest magnitude, all sources in one pass (reads each
// array once: bound by HBM), and the first operand's sums of squares in
// binary32, one partial per row chunk (part[chunk][column]; summed in order by
// k_oz_columns, so that the same input always gives the same sum)
template <int SC>
__global__ void __launch_bounds__(256) k_oz_colmax(OzSrc a, int sources, int row_chunks, float* part) {
    pdl_enter();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.y == 0 && (int)threadIdx.x < sources)
        a.peaked[threadIdx.x * (1 + a.f.q)] = 0;
    const long long k = (long long)blockIdx.x * 32 + threadIdx.x;
    const long long per = (a.f.d + row_chunks - 1) / row_chunks;
    const long long r0 = (long long)blockIdx.y * per, r1 = k < a.f.q ? min(a.f.d, r0 + per) : r0;
    unsigned long long m[SC];
    float ss = 0.0f;
    double sg[SC];
#pragma unroll
    for (int z = 0; z < SC; ++z) m[z] = 0;
#pragma unroll
    for (int i = 0; i + 1 < SC; ++i) sg[i] = i + 1 < sources && k < a.f.q ? sign_of(a.dots, a.f.q, i, k) : 0.0;
    auto up = [](unsigned long long& x, double v) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
        x = b > x ? b : x;
        return (uint32_t)(b >> 32);
    };
#pragma unroll 4
    for (long long r = r0 + threadIdx.y; r < r1; r += 8) {
        const long long e = r * a.f.q + k;
        const double f0 = a.f.F0[e];
        const uint32_t h = up(m[0], a.X ? f0 + a.X[e] : f0);
        // the square of the value cut to binary32 by integer arithmetic (20
        // mantissa bits; below 2^-63 zero, which only makes the sum smaller)
        const float c = __uint_as_float(h < 0x3C000000u ? 0u : (h - 0x38000000u) << 3);
        ss = __fmaf_rn(c, c, ss);
#pragma unroll
        for (int i = 0; i + 1 < SC; ++i)
            if (i + 1 < sources) up(m[i + 1], fma(sg[i], a.f.F[i][e], -f0));
    }
    // the block's rows first: one atomic per column and block
    __shared__ unsigned long long red[8][33];
    __shared__ float reds[8][33];
#pragma unroll
    for (int z = 0; z < SC; ++z) {
        if (z >= sources) break;
        red[threadIdx.y][threadIdx.x] = m[z];
        if (z == 0) reds[threadIdx.y][threadIdx.x] = ss;
        __syncthreads();
        if (threadIdx.y == 0 && k < a.f.q) {
            unsigned long long v = m[z];
            for (int y = 1; y < 8; ++y) v = red[y][threadIdx.x] > v ? red[y][threadIdx.x] : v;
            atomicMax(&a.mx[(long long)z * a.f.q + k], v);
            if (z == 0) {
                for (int y = 1; y < 8; ++y) ss += reds[y][threadIdx.x];
                part[(long long)blockIdx.y * a.f.q + k] = ss;
            }
        }
        __syncthreads();
    }
}

// |x| < 2^e for a column whose largest magnitude has these bits; columns
// below 2^-900 share the exponent -900, OZ_NONFINITE marks NaN / infinity
__device__ __forceinline__ int oz_exponent(unsigned long long bits) {
    const int be = (int)(bits >> 52);
    if (be >= 0x7FF) return OZ_NONFINITE;
    return max(be - 1022, -900);
}

// Which columns the slices cannot hold well enough: an entry of the product is
// off by about sqrt(d) 2^-56.3 2^(e_a + e_b) (the slice pairs left out), a
// binary64 sum by about 2^-55 |a| |b|, so the slices are the nearer ones while
// 2^e <= 1.6 d^(-1/4) |x| for both columns.  Dense columns are (of random ones,
// at the least favourable scale, all but 7 % at d = 512, 0.7 % at 1024 and none
// at 3584); a column with an entry that holds much of its norm is not, and its
// entries come from k_oz_f64.  RMS error
// over |a| |b| of the slices and of the binary64 sum, d = 3584: dense 9e-18 and
// 4e-17; a peak of 0.2 of the norm in each column, on different rows, 4.9e-17
// and 4.1e-17 (ratio 1.94); of 0.5, 6.6e-16 and 3.2e-17.  Columns outside
// 2^-55 .. 2^50, where the binary32 sum of the first operand's squares does not
// reach, are left to binary64 as well; zero columns are exact, and non-finite ones NaN either way.
__global__ void __launch_bounds__(256) k_oz_columns(OzSrc a, int sources, int row_chunks, const float* part) {
    pdl_enter();
    const long long q = a.f.q, k = (long long)blockIdx.x * 256 + threadIdx.x;
    const int z = blockIdx.y;
    if (k >= q) return;
    const unsigned long long bits = a.mx[(long long)z * q + k];
    const int e = oz_exponent(bits);
    if (bits == 0 || e >= OZ_NONFINITE) return;
    float s = 0.0f;
    if (z) s = (float)a.cd[((long long)(z - 1) * (sources - 1) + z - 1) * q + k];
    else for (int c = 0; c < row_chunks; ++c) s += part[(long long)c * q + k];
    const float lim = 1.6f * 1.6f * rsqrtf((float)a.f.d);            // of (2^e / |x|)^2
    if (e < -55 || e > 50 || !(exp2f((float)(2 * e)) <= lim * s)) {
        int32_t* const list = a.peaked + z * (1 + q);
        list[1 + atomicAdd(&list[0], 1)] = (int32_t)k;
    }
}

// The product's entries of those columns, summed in binary64 on the CUDA cores
// in row order: peaked columns of the first operand against every column of
// the second, and every column of the first against peaked ones of the second
// (an entry of both is written twice, the same sum).  A block takes a group of
// 8 listed columns, one per warp, against 32 columns of the other operand, one
// entry per thread: the binary64 rate (two sums a clock and SM) is what bounds
// it, so a few listed columns are better spread over many blocks than tiled
// (one column of a 1216 x 576 frame: 670 us in 64 x 64 tiles).  32 rows a
// step, the next ones' loads in flight.  Without such columns, the usual
// case, the blocks return at once.
constexpr int OZF_LIST = 8, OZF_COLS = 32, OZF_ROWS = 32;
__global__ void __launch_bounds__(256) k_oz_f64(OzSrc a, int K, double* C) {
    pdl_enter();
    __shared__ double sl[OZF_ROWS][OZF_LIST], so[OZF_ROWS][OZF_COLS];
    const long long q = a.f.q, d = a.f.d;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long nt = (q + OZF_COLS - 1) / OZF_COLS;
    auto groups = [&](int z) { return (long long)(a.peaked[z * (1 + q)] + OZF_LIST - 1) / OZF_LIST; };
    const long long ga = groups(0) * nt;              // work items of the first operand's columns, per pair
    long long first = 0;                              // first work item of this pair
    for (int i = 0; i < (K ? K : 1); ++i) {
        const int zb = K ? 1 + i : 0;
        const long long items = ga + (K ? groups(zb) * nt : 0);
        // this block's items, counted over all pairs
        long long w = ((long long)blockIdx.x - first % gridDim.x + gridDim.x) % gridDim.x;
        for (; w < items; w += gridDim.x) {
            const bool rows = w < ga;                 // the listed column is the product's row
            const int zl = rows ? 0 : zb, zo = rows ? zb : 0;
            const long long v = rows ? w : w - ga;
            const int32_t* const list = a.peaked + zl * (1 + q);
            auto listed = [&](int x) { const long long at = v / nt * OZF_LIST + x; return at < list[0] ? (long long)list[1 + at] : -1LL; };
            const long long kl = listed(threadIdx.x & (OZF_LIST - 1));    // the column this thread loads from
            const long long kw = listed(warp), ko = v % nt * OZF_COLS + lane;
            const double gl = zl && kl >= 0 ? sign_of(a.dots, q, zl - 1, kl) : 0.0;
            const double go = zo && ko < q ? sign_of(a.dots, q, zo - 1, ko) : 0.0;
            double nl, no[OZF_ROWS / 8];
            auto load = [&](long long r0) {
                const long long rl = r0 + threadIdx.x / OZF_LIST;
                nl = rl < d && kl >= 0 ? oz_signed(a, zl, rl * q + kl, gl) : 0.0;
#pragma unroll
                for (int y = 0; y < OZF_ROWS / 8; ++y) {
                    const long long ro = r0 + 8 * y + warp;
                    no[y] = ro < d && ko < q ? oz_signed(a, zo, ro * q + ko, go) : 0.0;
                }
            };
            double acc = 0.0;
            load(0);
            for (long long r0 = 0; r0 < d; r0 += OZF_ROWS) {
                __syncthreads();
                sl[threadIdx.x / OZF_LIST][threadIdx.x & (OZF_LIST - 1)] = nl;
#pragma unroll
                for (int y = 0; y < OZF_ROWS / 8; ++y) so[8 * y + warp][lane] = no[y];
                __syncthreads();
                load(r0 + OZF_ROWS);
                if (kw >= 0) {
#pragma unroll
                    for (int r = 0; r < OZF_ROWS; ++r) acc = fma(sl[r][warp], so[r][lane], acc);
                }
            }
            if (kw >= 0 && ko < q) {
                const long long k = rows ? kw : ko, l = rows ? ko : kw;
                if (K) {
                    C[((long long)i * q + k) * q + l] = acc;
                } else {
                    acc -= k == l ? 1.0 : 0.0;
                    C[k * q + l] = acc;
                    C[l * q + k] = acc;
                }
            }
        }
        first += items;
    }
}

// The slabs of source z0 + blockIdx.z (slot blockIdx.z of `out`): thread =
// (column, 8-row half) of one 16-row chunk.  x 2^(55 - e) as a 64-bit integer,
// its signed base-256 digits from the bottom, one 16-byte store per slice
// (consecutive columns consecutive).
__global__ void __launch_bounds__(256) k_oz_split(OzSrc a, int z0, unsigned char* out, unsigned long long slot_bytes) {
    pdl_enter();
    const int z = z0 + blockIdx.z;
    const int kl = threadIdx.x & 127, half = threadIdx.x >> 7;
    const long long k = (long long)blockIdx.y * OZ_BM + kl;
    const long long chunk = blockIdx.x, r0 = chunk * OZ_BK + 8 * half;
    const long long q = a.f.q, d = a.f.d;
    int e = 0;
    if (k < q) e = oz_exponent(a.mx[(long long)z * q + k]);
    if (chunk == 0 && half == 0) a.ex[(long long)z * a.Qp + k] = e;
    const bool live = k < q && e < OZ_NONFINITE;
    const double scale = __longlong_as_double((long long)(1023 + 55 - (live ? e : 0)) << 52);
    long long v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
        v[j] = (live && r0 + j < d) ? __double2ll_rn(oz_value(a, z, (r0 + j) * q + k, k) * scale) : 0;
    unsigned char* dst = out + blockIdx.z * slot_bytes +
                         ((unsigned long long)blockIdx.y * gridDim.x + chunk) * OZ_SLAB_BYTES +
                         (kl >> 3) * 256 + half * 128 + (kl & 7) * 16;
#pragma unroll
    for (int t = OZ_SLICES - 1; t >= 0; --t) {
        float g[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int dg = t ? (int)(signed char)v[j] : (int)v[j];
            v[j] = (v[j] - dg) >> 8;
            g[j] = (float)dg;
        }
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(g[2 * j], g[2 * j + 1]);
            w[j] = *reinterpret_cast<const uint32_t*>(&h);
        }
        *reinterpret_cast<uint4*>(dst + t * OZ_SLICE_BYTES) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// C (qq entries per z) = the sum of the splits' partial sums, in split order
__global__ void __launch_bounds__(256) k_oz_reduce(const double* part, int splits, int nz, long long q, double* C,
                                                   int minus_identity) {
    pdl_enter();
    const long long total = (long long)nz * q * q;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        double s = part[e];
        for (int p = 1; p < splits; ++p) s += part[(long long)p * total + e];
        if (minus_identity) {
            const long long x = e % (q * q);
            if (x / q == x % q) s -= 1.0;
        }
        C[e] = s;
    }
}

// Split operands of an m x n bf16 / fp32 matrix G (row stride n): row-major
// (rows Mp of 2 Np, element G[r, c]) or transposed (rows Np of 2 Mp, element
// G[r, c] at row c, position r)
__device__ __forceinline__ double load_typed(const void* p, int dtype, long long e) {
    if (dtype == ISO_BF16) return widen(__uint_as_float((uint32_t)static_cast<const unsigned short*>(p)[e] << 16));
    return widen(static_cast<const float*>(p)[e]);
}
__global__ void __launch_bounds__(256) k_op_split_g(const void* G, int dtype, long long m, long long n, long long Mp,
                                                    long long Np, float* out) {
    pdl_enter();
    for (long long r = blockIdx.x; r < Mp; r += gridDim.x)
    for (long long c = threadIdx.x; c < Np; c += blockDim.x) {
        const double v = (r < m && c < n) ? load_typed(G, dtype, r * n + c) : 0.0;
        put_split(out + r * 2 * Np, Np, c, v);
    }
}
__global__ void __launch_bounds__(256) k_op_split_gt(const void* G, int dtype, long long m, long long n, long long Mp,
                                                     long long Np, float* out) {
    pdl_enter();
    __shared__ double t[32][33];
    const long long r0 = (long long)blockIdx.x * 32, c0 = (long long)blockIdx.y * 32;
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long r = r0 + y, c = c0 + threadIdx.x;
        t[y][threadIdx.x] = (r < m && c < n) ? load_typed(G, dtype, r * n + c) : 0.0;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long c = c0 + y, r = r0 + threadIdx.x;
        if (c < Np && r < Mp) put_split(out + c * 2 * Mp, Mp, r, t[threadIdx.x][y]);
    }
}

// F += E (binary64, d x q)
__global__ void __launch_bounds__(256) k_op_add(double* F, const double* E, long long total) {
    pdl_enter();
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x)
        F[e] += E[e];
}

// Sym_i = sym(A_i), Kw_i = A_i - Sym_i (binary64; A is K arrays q x q)
__global__ void __launch_bounds__(256) k_fr_symskew(const double* A, long long Qp, long long q, double* sym, double* kw) {
    pdl_enter();
    __shared__ double ta[32][33], tb[32][33];
    const int i = blockIdx.z;
    const double* Ai = A + (long long)i * q * q;
    const long long r0 = (long long)blockIdx.y * 32, c0 = (long long)blockIdx.x * 32;
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long ra = r0 + y, ca = c0 + threadIdx.x, rb = c0 + y, cb = r0 + threadIdx.x;
        ta[y][threadIdx.x] = (ra < q && ca < q) ? Ai[ra * q + ca] : 0.0;   // A[r0 + y, c0 + x]
        tb[y][threadIdx.x] = (rb < q && cb < q) ? Ai[rb * q + cb] : 0.0;   // A[c0 + y, r0 + x]
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long r = r0 + y, c = c0 + threadIdx.x;
        if (r < q && c < q) {
            const double a = ta[y][threadIdx.x], b = tb[threadIdx.x][y];   // A[r, c], A[c, r]
            sym[((long long)i * q + r) * q + c] = 0.5 * (a + b);
            kw[((long long)i * q + r) * q + c] = 0.5 * (a - b);
        }
    }
}

// Gamma_ij (i <= j), summed into gram[i][j]; block y takes rows y, y + gridDim.y, ... of the q x q entries
struct GramArgs {
    const double* A[2];         // per side: K arrays q x q
    const double* sym[2];
    const double* kw[2];
    const double* cd[2];        // per side: K x K x q
    const double* S0;
    double* gram;
    long long q, Qp, k_keep;
    int K;
};
__global__ void __launch_bounds__(256) k_fr_gram(GramArgs g) {
    pdl_enter();
    __shared__ double red[32];
    // pair (i, j), i <= j, from blockIdx.x
    int i = 0, j = 0, p = blockIdx.x;
    for (i = 0; i < g.K; ++i) {
        if (p < g.K - i) { j = i + p; break; }
        p -= g.K - i;
    }
    const long long q = g.q, qq = q * q;
    double acc = 0.0;
    for (long long r = blockIdx.y; r < q; r += gridDim.y) {
        const double sr = g.S0[r], Dr = r < g.k_keep ? 1.0 : 0.0;
        for (long long c = threadIdx.x; c < q; c += blockDim.x) {
            const long long e = r * q + c;
            const double sc = g.S0[c], Dc = c < g.k_keep ? 1.0 : 0.0;
            // column terms (row l = r, column k = c), both sides
            double colt = 0.0;
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const double ai = g.A[s][(long long)i * qq + e];
                const double aj = g.A[s][(long long)j * qq + e];
                const double si = g.sym[s][(long long)i * qq + e], sj = g.sym[s][(long long)j * qq + e];
                colt += ai * sj + si * aj - si * sj;
            }
            acc -= sc * sc * Dc * colt;
            // cross terms (k = r, l = c)
            const double kui = g.kw[0][(long long)i * qq + e], kuj = g.kw[0][(long long)j * qq + e];
            const double kvi = g.kw[1][(long long)i * qq + e], kvj = g.kw[1][(long long)j * qq + e];
            acc -= sr * sc * Dr * Dc * (kui * kvj + kuj * kvi);
        }
    }
    if (blockIdx.y == 0)
        for (long long k = threadIdx.x; k < min(q, g.k_keep); k += blockDim.x)
            acc += g.S0[k] * g.S0[k] *
                   (g.cd[0][((long long)i * g.K + j) * q + k] + g.cd[1][((long long)i * g.K + j) * q + k]);
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) atomicAdd(&g.gram[i * g.K + j], acc);
}

// c* from Gamma (upper triangle), then the caller's stats
__global__ void k_fr_solve(double* gram, double* coef, int K, double ridge, double c_min, double c_max,
                           double* st_gram, double* st_coef) {
    pdl_enter();
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double G[MAXK * MAXK], c[MAXK];
    for (int a = 0; a < K; ++a)
        for (int b = a; b < K; ++b) {
            G[a * K + b] = gram[a * K + b];
            G[b * K + a] = gram[a * K + b];
        }
    for (int a = 0; a < K * K; ++a) gram[a] = G[a];
    retention_solve(G, K, ridge, c_min, c_max, c);
    for (int a = 0; a < K; ++a) coef[a] = c[a];
    if (st_gram) for (int a = 0; a < K * K; ++a) st_gram[a] = G[a];
    if (st_coef) for (int a = 0; a < K; ++a) st_coef[a] = c[a];
}

// xi* = D dF_c - E (E = F_0 Y from the GEMM, ld Qp)
__global__ void __launch_bounds__(256) k_fr_xi(Frames f, const double* dots, const double* coef, const float* E,
                                               long long Qp, long long k_keep, double* xi) {
    pdl_enter();
    for (long long r = blockIdx.x; r < f.d; r += gridDim.x)
    for (long long k = threadIdx.x; k < f.q; k += blockDim.x) {
        const long long e = r * f.q + k;
        double v = 0.0;
        if (k < k_keep) {
            const double f0 = f.F0[e];
            for (int i = 0; i < f.K; ++i) v = fma(coef[i], fma(sign_of(dots, f.q, i, k), f.F[i][e], -f0), v);
        }
        xi[e] = v - widen(E[r * Qp + k]);
    }
}

// ||N||_F^2 of N = xi^T xi (binary32, ld Qp; or binary64, ld q), one warp per row, summed into the header
__global__ void __launch_bounds__(256) k_fr_norm(const float* N, const double* N64, long long Qp, long long q,
                                                 FrameHeader* h, int side) {
    pdl_enter();
    __shared__ double red[32];
    const int lane = threadIdx.x & 31;
    double acc = 0.0;
    for (long long r = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); r < q; r += (long long)gridDim.x * 8)
        for (long long c = lane; c < q; c += 32) {
            const double v = N64 ? N64[r * q + c] : (double)N[r * Qp + c];
            acc += v * v;
        }
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) atomicAdd(&h->nu2[side], acc);
}

// The Newton-Schulz iterates y, z and the step m are symmetric in exact
// arithmetic (functions of N); the products treat them so (B = M^T = M).  Each
// kernel below symmetrises what it writes, one 32 x 32 tile and its mirror
// per block (blocks below the diagonal return), so that rounding cannot
// build an asymmetric component from one iteration to the next, and writes
// the tile's split operands as well.  Reading both tiles before writing
// either makes the update safe in place.
struct NsArgs {
    const float* N;     // init: N = xi^T xi (binary32, ld Qp), unless N64 is given
    const double* N64;  // init: N in binary64 (ld q)
    const float* T1;    // m: z y (NULL: 0);  update: y m
    const float* T2;    // update: m z (NULL: 0)
    double* y;
    double* z;
    double* m;
    float* y4;          // the split operands of y, z and m (Qp rows of 2 Qp, zero past q)
    float* z4;
    float* m4;
    FrameHeader* h;
    long long q, Qp;
    int side, it;
};

__device__ __forceinline__ bool ns_tile(long long& r0, long long& c0) {
    if (blockIdx.x < blockIdx.y) return false;
    r0 = (long long)blockIdx.y * 32;
    c0 = (long long)blockIdx.x * 32;
    return true;
}

// one entry of a symmetric iterate and of its split operand (zero past q)
__device__ __forceinline__ void ns_put(const NsArgs& a, double* M, float* M4, long long r, long long c, double v) {
    if (r < a.q && c < a.q) M[r * a.q + c] = v;
    uint32_t hw;
    float* const row = M4 + r * 2 * a.Qp;
    row[c] = ns_tf32(v, hw);
    row[a.Qp + c] = ns_tf32(v - __hiloint2double((int)hw, 0), hw);
}

// Y_0 = (I + N) / cs = I + y, Z_0 = I (z = 0); cs = 1 while ||N||_F < 0.9,
// else 1 + ||N||_F / 2, so that the eigenvalues of Y_0 lie in (0, 2)
__global__ void __launch_bounds__(256) k_fr_ns_init(NsArgs a) {
    pdl_enter();
    __shared__ double ta[32][33], tb[32][33];
    long long r0, c0;
    if (!ns_tile(r0, c0)) return;
    const double nu = sqrt(a.h->nu2[a.side]);
    const double cs = nu < 0.9 ? 1.0 : 1.0 + 0.5 * nu;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) {
        a.h->cs[a.side] = cs;
        a.h->conv[a.side] = 0;
    }
    auto f = [&](long long r, long long c) -> double {
        if (r >= a.q || c >= a.q) return 0.0;
        const double id = r == c ? 1.0 : 0.0;
        const double nv = a.N64 ? a.N64[r * a.q + c] : (double)a.N[r * a.Qp + c];
        return (id + nv) / cs - id;
    };
    for (int y = threadIdx.y; y < 32; y += 8) {
        ta[y][threadIdx.x] = f(r0 + y, c0 + threadIdx.x);
        tb[y][threadIdx.x] = f(c0 + y, r0 + threadIdx.x);
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long r = r0 + y, c = c0 + threadIdx.x, r2 = c0 + y, c2 = r0 + threadIdx.x;
        ns_put(a, a.y, a.y4, r, c, halve(ta[y][threadIdx.x] + tb[threadIdx.x][y]));
        ns_put(a, a.y, a.y4, r2, c2, halve(tb[y][threadIdx.x] + ta[threadIdx.x][y]));
        if (r < a.q && c < a.q) a.z[r * a.q + c] = 0.0;
        if (r2 < a.q && c2 < a.q) a.z[r2 * a.q + c2] = 0.0;
    }
}

// w = y + z + z y (the residual Z Y - I), m = -w / 2; the largest |w| of the
// iteration goes to the header
__global__ void __launch_bounds__(256) k_fr_ns_m(NsArgs a) {
    pdl_enter();
    __shared__ double ta[32][33], tb[32][33];
    if (*reinterpret_cast<volatile int32_t*>(&a.h->conv[a.side])) return;
    long long r0, c0;
    if (!ns_tile(r0, c0)) return;
    auto w = [&](long long r, long long c) -> double {
        if (r >= a.q || c >= a.q) return 0.0;
        const long long e = r * a.q + c;
        const double v = a.y[e] + a.z[e];
        return a.T1 ? v + ns_widen(a.T1[r * a.Qp + c]) : v;
    };
    for (int y = threadIdx.y; y < 32; y += 8) {
        ta[y][threadIdx.x] = w(r0 + y, c0 + threadIdx.x);
        tb[y][threadIdx.x] = w(c0 + y, r0 + threadIdx.x);
    }
    __syncthreads();
    unsigned long long most = 0;                   // largest |w| as binary64 bits
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long r = r0 + y, c = c0 + threadIdx.x;
        const double v = halve(ta[y][threadIdx.x] + tb[threadIdx.x][y]);
        ns_put(a, a.m, a.m4, r, c, -halve(v));
        const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
        most = b > most ? b : most;
        ns_put(a, a.m, a.m4, c0 + y, r0 + threadIdx.x, -halve(halve(tb[y][threadIdx.x] + ta[threadIdx.x][y])));
    }
    float wm = (float)__longlong_as_double((long long)most);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xFFFFFFFFu, wm, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&a.h->wmax[a.side][a.it], __float_as_uint(wm));
}

// y += m + y m, z += m + m z, in place.  The iteration stops (this update and
// every later one skipped) once the residual is at the tolerance, or has
// stopped its quadratic fall below 1e-2 (the rounding floor of the products),
// or has grown.
__global__ void __launch_bounds__(256) k_fr_ns_update(NsArgs a) {
    pdl_enter();
    __shared__ double ya[32][33], yb[32][33], za[32][33], zb[32][33];
    if (*reinterpret_cast<volatile int32_t*>(&a.h->conv[a.side])) return;
    const double wc = (double)__uint_as_float(a.h->wmax[a.side][a.it]);
    const double wp = a.it > 0 ? (double)__uint_as_float(a.h->wmax[a.side][a.it - 1]) : 1e300;
    const bool stop = !(wc > FR_NS_TOL) || wc >= wp || (wc < 1e-2 && wc > 0.25 * wp);
    if (stop) {
        if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) a.h->conv[a.side] = 1;
        return;
    }
    long long r0, c0;
    if (!ns_tile(r0, c0)) return;
    auto fy = [&](long long r, long long c) -> double {
        if (r >= a.q || c >= a.q) return 0.0;
        const long long e = r * a.q + c;
        return a.y[e] + a.m[e] + ns_widen(a.T1[r * a.Qp + c]);
    };
    auto fz = [&](long long r, long long c) -> double {
        if (r >= a.q || c >= a.q) return 0.0;
        const long long e = r * a.q + c;
        const double v = a.z[e] + a.m[e];
        return a.T2 ? v + ns_widen(a.T2[r * a.Qp + c]) : v;
    };
    for (int y = threadIdx.y; y < 32; y += 8) {
        ya[y][threadIdx.x] = fy(r0 + y, c0 + threadIdx.x);
        yb[y][threadIdx.x] = fy(c0 + y, r0 + threadIdx.x);
        za[y][threadIdx.x] = fz(r0 + y, c0 + threadIdx.x);
        zb[y][threadIdx.x] = fz(c0 + y, r0 + threadIdx.x);
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long r = r0 + y, c = c0 + threadIdx.x, r2 = c0 + y, c2 = r0 + threadIdx.x;
        ns_put(a, a.y, a.y4, r, c, halve(ya[y][threadIdx.x] + yb[threadIdx.x][y]));
        ns_put(a, a.z, a.z4, r, c, halve(za[y][threadIdx.x] + zb[threadIdx.x][y]));
        ns_put(a, a.y, a.y4, r2, c2, halve(yb[y][threadIdx.x] + ya[threadIdx.x][y]));
        ns_put(a, a.z, a.z4, r2, c2, halve(zb[y][threadIdx.x] + za[threadIdx.x][y]));
    }
}

// E_F = xi* + (F_0 + xi*) R (P from the GEMM, ld Qp), in place over xi*
__global__ void __launch_bounds__(256) k_fr_motion(double* xi, const float* P, long long Qp, long long d, long long q) {
    pdl_enter();
    for (long long r = blockIdx.x; r < d; r += gridDim.x)
        for (long long c = threadIdx.x; c < q; c += blockDim.x) xi[r * q + c] += widen(P[r * Qp + c]);
}

__global__ void k_fr_status(const FrameHeader* h, int32_t* out) {
    pdl_enter();
    if (threadIdx.x == 0 && blockIdx.x == 0) *out = h->status;
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------
size_t al256(size_t v) { return (v + 255) & ~(size_t)255; }

struct FrameLayout {
    long long m, n, q, Mp, Np, Qp, K;
    size_t hdr, gram, coef, dots, mx[2], zero_end, ex, vcopy;
    size_t tail;      // from here on: unused until A_i is formed (its operands' slabs)
                      // (sym[side] holds the side's list of peaked columns until then)
    size_t cd[2], ft4[2], aq[2], sym[2], kw[2], fr4[2], y4[2], e[2], xi[2], nq[2];
    size_t ns_y, ns_z, ns_m, ns_y4, ns_z4, ns_m4, ns_t1, ns_t2, ns_t3;
    size_t a6, b6, total;
};

FrameLayout frame_layout(long long m, long long n, int K) {
    FrameLayout L;
    L.m = m; L.n = n; L.K = K;
    L.q = std::min(m, n);
    L.Mp = pad_up(m); L.Np = pad_up(n); L.Qp = pad_up(L.q);
    const long long q = L.q, Qp = L.Qp;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t at = o; o = al256(o + bytes); return at; };
    L.hdr = take(sizeof(FrameHeader));
    L.gram = take(sizeof(double) * K * K);
    L.coef = take(sizeof(double) * K);
    L.dots = take(sizeof(double) * K * q);
    for (int s = 0; s < 2; ++s) L.cd[s] = take(sizeof(double) * K * K * q);
    for (int s = 0; s < 2; ++s) L.mx[s] = take(sizeof(unsigned long long) * (K + 1) * q);
    L.zero_end = o;
    L.ex = take(sizeof(int32_t) * (K + 1) * Qp);
    L.vcopy = take(sizeof(double) * (K + 1) * n * q);
    for (int s = 0; s < 2; ++s) {
        L.aq[s] = take(sizeof(double) * K * q * q);        // A_i = F_0^T dF_i (binary64)
        L.sym[s] = take(sizeof(double) * K * q * q);
        L.kw[s] = take(sizeof(double) * K * q * q);
    }
    L.tail = o;
    for (int s = 0; s < 2; ++s) {
        const long long Dp = s == 0 ? L.Mp : L.Np, d = s == 0 ? m : n;
        L.ft4[s] = take(sizeof(float) * Qp * 2 * Dp);      // xi*^T split
        L.fr4[s] = take(sizeof(float) * Dp * 2 * Qp);      // F_0 split, later (F_0 + xi*) split
        L.y4[s] = take(sizeof(float) * Qp * 2 * Qp);       // Y^T split, later R split
        L.e[s] = take(sizeof(float) * Dp * Qp);            // F_0 Y, later (F_0 + xi*) R
        L.xi[s] = take(sizeof(double) * d * q);            // xi*, later E_F
        L.nq[s] = take(sizeof(float) * Qp * Qp);
    }
    L.ns_y = take(sizeof(double) * q * q);
    L.ns_z = take(sizeof(double) * q * q);
    L.ns_m = take(sizeof(double) * q * q);
    L.ns_y4 = take(sizeof(float) * Qp * 2 * Qp);
    L.ns_z4 = take(sizeof(float) * Qp * 2 * Qp);
    L.ns_m4 = take(sizeof(float) * Qp * 2 * Qp);
    L.ns_t1 = take(sizeof(float) * Qp * Qp);
    L.ns_t2 = take(sizeof(float) * Qp * Qp);
    L.ns_t3 = take(sizeof(float) * Qp * Qp);
    L.a6 = take(sizeof(float) * L.Mp * 2 * 2 * Qp);
    L.b6 = take(sizeof(float) * L.Np * 2 * 2 * Qp);
    L.total = o;
    return L;
}

int grid_of(long long work, int sms) {
    const long long b = (work + 255) / 256;
    return (int)std::max(1LL, std::min(b, (long long)sms * 8));
}

// Large dynamic shared memory must be opted into once per kernel and device.
template <auto Kernel>
int smem_optin(int bytes) {
    static std::atomic<unsigned long long> done{0};       // a bit per device
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess) return ISO_ERR_CUDA;
    const unsigned long long bit = d < 64 ? 1ull << d : 0;
    if (done.load(std::memory_order_relaxed) & bit) return ISO_OK;
    if (cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return ISO_ERR_CUDA;
    done.fetch_or(bit, std::memory_order_relaxed);
    return ISO_OK;
}

// C (a_rows x b_rows) = A B^T over the three-product split: A and B are
// two-segment operand arrays of segment length L (rows a_rows / b_rows,
// multiples of 128); with A2, a second product C2 = A2 B2^T of the same shape
// in the same launch.  The tile shape with the smaller number of waves times
// what a stage costs in it (clocks per 32 contraction columns: 1900 for 128 x
// 256, bound by shared memory; 1150 for 128 x 128, bound by L2), or the given one.
int frame_gemm(cudaStream_t s, int sms, const float* A, long long a_rows, const float* B, long long b_rows, long long L,
               GemmArgs g, const float* A2 = nullptr, const float* B2 = nullptr, int width = 0) {
    CUtensorMap ta, tb, ta2, tb2;
    ISO_TRY(gemm_tensor_map(&ta, A, a_rows, 2 * L, 2 * L));
    ISO_TRY(gemm_tensor_map(&tb, B, b_rows, 2 * L, 2 * L));
    ISO_TRY(gemm_tensor_map(&ta2, A2 ? A2 : A, a_rows, 2 * L, 2 * L));
    ISO_TRY(gemm_tensor_map(&tb2, A2 ? B2 : B, b_rows, 2 * L, 2 * L));
    g.k_tiles = (int)(L / GEMM_BK);
    g.seg = (int)L;
    g.c_cols = (int)b_rows;
    ISO_TRY(smem_optin<k_gemm_x3<128>>(X3_SMEM));
    ISO_TRY(smem_optin<k_gemm_x3<256>>(X3_SMEM));
    const unsigned nz = A2 ? 2 : 1;
    const long long my = a_rows / GEMM_BM, t128 = my * (b_rows / 128) * nz, t256 = my * ((b_rows + 255) / 256) * nz;
    const bool wide = width ? width == 256 : (t256 + sms - 1) / sms * 1900 <= (t128 + sms - 1) / sms * 1150;
    const int slot = prof_begin(0, s);
    if (wide)
        pdl_launch(k_gemm_x3<256>, dim3((unsigned)((b_rows + 255) / 256), (unsigned)my, nz), GEMM_THREADS, X3_SMEM, s, ta, tb, ta2,
                                                                                                            tb2, g);
    else
        pdl_launch(k_gemm_x3<128>, dim3((unsigned)(b_rows / 128), (unsigned)my, nz), GEMM_THREADS, X3_SMEM, s, ta, tb, ta2, tb2, g);
    prof_end(slot, s);
    return cudaGetLastError() == cudaSuccess ? ISO_OK : ISO_ERR_CUDA;
}

struct OptLayout {
    long long m, n, q, Mp, Np, Qp, Dmax;
    size_t hdr, mx[2], zero_end, ex, gw4, gwt4, su4, sv4, dF[2], n64, xb4, r4, p, a6, b6;
    size_t ns_y, ns_z, ns_m, ns_y4, ns_z4, ns_m4, ns_t1, ns_t2, ns_t3, total;
};

OptLayout opt_layout(long long m, long long n) {
    OptLayout L;
    L.m = m; L.n = n; L.q = std::min(m, n);
    L.Mp = pad_up(m); L.Np = pad_up(n); L.Qp = pad_up(L.q);
    L.Dmax = std::max(L.Mp, L.Np);
    const long long q = L.q, Qp = L.Qp;
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t at = o; o = al256(o + bytes); return at; };
    L.hdr = take(sizeof(FrameHeader));
    for (int s = 0; s < 2; ++s) L.mx[s] = take(sizeof(unsigned long long) * q);
    L.zero_end = o;
    L.ex = take(sizeof(int32_t) * Qp);
    // the four gradient operands, dead after the factor gradients: then the slabs of X_bar
    L.gw4 = take(sizeof(float) * L.Mp * 2 * L.Np);      // G_W, rows m, contraction n
    L.gwt4 = take(sizeof(float) * L.Np * 2 * L.Mp);     // G_W^T, rows n, contraction m
    L.su4 = take(sizeof(float) * Qp * 2 * L.Mp);        // (U S_0)^T
    L.sv4 = take(sizeof(float) * Qp * 2 * L.Np);        // (V S_0)^T
    L.dF[0] = take(sizeof(double) * m * q);             // U_bar - U, later E_U
    L.dF[1] = take(sizeof(double) * n * q);             // V_bar - V, later E_V
    L.n64 = take(sizeof(double) * q * q);               // (F + dF)^T (F + dF) - I
    L.xb4 = take(sizeof(float) * L.Dmax * 2 * Qp);      // F + dF
    L.r4 = take(sizeof(float) * Qp * 2 * Qp);
    L.p = take(sizeof(float) * L.Dmax * Qp);
    L.a6 = take(sizeof(float) * L.Mp * 2 * 2 * Qp);
    L.b6 = take(sizeof(float) * L.Np * 2 * 2 * Qp);
    L.ns_y = take(sizeof(double) * q * q);
    L.ns_z = take(sizeof(double) * q * q);
    L.ns_m = take(sizeof(double) * q * q);
    L.ns_y4 = take(sizeof(float) * Qp * 2 * Qp);
    L.ns_z4 = take(sizeof(float) * Qp * 2 * Qp);
    L.ns_m4 = take(sizeof(float) * Qp * 2 * Qp);
    L.ns_t1 = take(sizeof(float) * Qp * Qp);
    L.ns_t2 = take(sizeof(float) * Qp * Qp);
    L.ns_t3 = take(sizeof(float) * Qp * Qp);
    L.total = o;
    return L;
}

// launch one CUDA-core kernel of the frame merge / optimizer step on stream s
#define FR_LAUNCH(...) do { const int _slot = prof_begin(1, s); __VA_ARGS__; prof_end(_slot, s); \
                                if (cudaGetLastError() != cudaSuccess) return ISO_ERR_CUDA; } while (0)

// C_i = F_0^T dF_i for i < K (K >= 1), or C = (F_0 + X)^T (F_0 + X) - I (K = 0),
// in binary64 through exact slices on the tensor cores (peaked columns summed
// in binary64); `scratch` holds the operands' slabs and, where the contraction
// is split, the partial sums.
// Experts are batched as the scratch allows.  The contraction is split over
// blocks until the last wave is full enough: `splits` minimises the number of
// waves per split, with 1 % per split for the partial sums' traffic.
int exact_product(cudaStream_t s, int sms, const OzSrc& src, int K, double* C, unsigned char* scratch,
                  size_t scratch_bytes, int32_t* status) {
    const long long q = src.f.q, d = src.f.d, Qp = src.Qp;
    const long long nt = Qp / OZ_BM, chunks = (d + OZ_BK - 1) / OZ_BK;
    const unsigned long long slot = (unsigned long long)nt * chunks * OZ_SLAB_BYTES;
    const int rc = (int)std::max(1LL, std::min(256LL, (d + 255) / 256));
    const dim3 mg((unsigned)((q + 31) / 32), rc), mb(32, 8);
    float* const part = reinterpret_cast<float*>(scratch);      // read before the slabs are written
    if (scratch_bytes / sizeof(float) < (size_t)rc * q) return ISO_ERR_WORKSPACE;
    if (K == 0) FR_LAUNCH((pdl_launch(k_oz_colmax<1>, mg, mb, 0, s, src, K + 1, rc, part)));
    else if (K <= 2) FR_LAUNCH((pdl_launch(k_oz_colmax<3>, mg, mb, 0, s, src, K + 1, rc, part)));
    else if (K <= 4) FR_LAUNCH((pdl_launch(k_oz_colmax<5>, mg, mb, 0, s, src, K + 1, rc, part)));
    else FR_LAUNCH((pdl_launch(k_oz_colmax<MAXK + 1>, mg, mb, 0, s, src, K + 1, rc, part)));
    FR_LAUNCH((pdl_launch(k_oz_columns, dim3((unsigned)((q + 255) / 256), (unsigned)(K + 1)), 256, 0, s, src, K + 1, rc, part)));
    ISO_TRY(smem_optin<k_oz_gemm>(OZ_SMEM));
    if (scratch_bytes < slot * (K ? 2 : 1)) return ISO_ERR_WORKSPACE;
    const int most = (int)std::min<unsigned long long>(std::max(K, 1), scratch_bytes / slot - (K ? 1 : 0));
    auto split = [&](int z0, int nz, unsigned char* out) -> int {
        FR_LAUNCH((pdl_launch(k_oz_split, dim3((unsigned)chunks, (unsigned)nt, (unsigned)nz), 256, 0, s, src, z0, out, slot)));
        return ISO_OK;
    };
    ISO_TRY(split(0, 1, scratch));
    for (int b0 = 0; b0 < std::max(K, 1); b0 += most) {
        const int nz = std::min(most, std::max(K, 1) - b0);
        unsigned char* const Bs = K ? scratch + slot : scratch;
        if (K) ISO_TRY(split(1 + b0, nz, Bs));
        const long long tiles = (K ? nt * nt : nt * (nt + 1) / 2) * nz;
        const unsigned long long used = slot * (K ? 1 + nz : 1);
        const long long fit = (long long)((scratch_bytes - used) / (8ull * (unsigned long long)(q * q) * nz));
        const long long least = (chunks * OZ_BK + OZ_MAX_ROWS - 1) / OZ_MAX_ROWS;
        long long best = least;
        double cost = 1e300;
        for (long long S = least; S <= std::max(least, 32LL); ++S) {
            if (S > least && (S > fit || chunks / S < 2 * OZ_STEPS_LOW)) break;
            const double c = (double)((tiles * S + sms - 1) / sms) / (double)S * (1.0 + 0.01 * (double)S);
            if (c < cost) { cost = c; best = S; }
        }
        const long long per = (chunks + best - 1) / best;
        const int splits = (int)((chunks + per - 1) / per);
        if (splits > 1 && splits > fit) return ISO_ERR_WORKSPACE;
        OzArgs g{};
        g.A = scratch;
        g.B = Bs;
        g.b_stride = slot;
        g.ea = src.ex;
        g.eb = src.ex + (K ? (1 + b0) * Qp : 0);
        g.eb_stride = Qp;
        g.C = C + (long long)b0 * q * q;
        g.c_stride = q * q;
        g.part = splits > 1 ? reinterpret_cast<double*>(scratch + used) : nullptr;
        g.q = q;
        g.tiles = (int)nt;
        g.chunks = (int)chunks;
        g.per_split = (int)per;
        g.symmetric = K ? 0 : 1;
        g.minus_identity = K || splits > 1 ? 0 : 1;
        g.status = status;
        const int pslot = prof_begin(0, s);
        pdl_launch(k_oz_gemm, dim3((unsigned)(tiles / nz), (unsigned)splits, (unsigned)nz), OZ_THREADS, OZ_SMEM, s, g);
        prof_end(pslot, s);
        if (cudaGetLastError() != cudaSuccess) return ISO_ERR_CUDA;
        if (splits > 1)
            FR_LAUNCH((pdl_launch(k_oz_reduce, grid_of((long long)nz * q * q, sms), 256, 0, s, g.part, splits, nz, q, g.C, K ? 0 : 1)));
    }
    FR_LAUNCH((pdl_launch(k_oz_f64, 4 * sms, 256, 0, s, src, K, C)));
    return ISO_OK;
}

// Scratch of the inverse square root
struct NsBufs {
    double *y, *z, *m;
    float *y4, *z4, *m4, *t1, *t2, *t3;
};

// R = (I + N)^(-1/2) - I for N = X^T X (binary32, ld Qp) with X^T F_0 skew,
// by the difference-form Newton-Schulz iteration (k_fr_ns_*), written as
// the split operand R4 (Qp rows of 2 Qp; R is symmetric, so it serves as B
// of (F_0 + X) R).  Header slot `side` holds its scaling and state.
int ns_root(cudaStream_t s, int sms, FrameHeader* hdr, int side, const float* Nq, const double* N64, long long q,
            long long Qp, const NsBufs& b, int ns_iters, float* R4) {
    FR_LAUNCH((pdl_launch(k_fr_norm, grid_of(q * 32, sms), 256, 0, s, Nq, N64, Qp, q, hdr, side)));
    NsArgs na{};
    na.N = Nq; na.N64 = N64; na.y = b.y; na.z = b.z; na.m = b.m; na.y4 = b.y4; na.z4 = b.z4; na.m4 = b.m4; na.h = hdr;
    na.q = q; na.Qp = Qp; na.side = side;
    const dim3 tiles((unsigned)(Qp / 32), (unsigned)(Qp / 32)), tb(32, 8);
    FR_LAUNCH((pdl_launch(k_fr_ns_init, tiles, tb, 0, s, na)));
    for (int it = 0; it < ns_iters; ++it) {
        GemmArgs g{};
        g.mode = GEMM_STORE_F32; g.ldc = Qp; g.M = (int)Qp; g.N = (int)Qp; g.status = &hdr->status;
        g.skip = &hdr->conv[side];
        g.C = b.t1;
        if (it) ISO_TRY(frame_gemm(s, sms, b.z4, Qp, b.y4, Qp, Qp, g));     // z y (z = 0 at first)
        na.it = it;
        na.T1 = it ? b.t1 : nullptr;
        FR_LAUNCH((pdl_launch(k_fr_ns_m, tiles, tb, 0, s, na)));
        // y m and, past the first step (z = 0), m z in one launch
        g.C = b.t2;
        g.C2 = b.t3;
        ISO_TRY(frame_gemm(s, sms, b.y4, Qp, b.m4, Qp, Qp, g, it ? b.m4 : nullptr, b.z4));
        na.T1 = b.t2;
        na.T2 = it ? b.t3 : nullptr;
        FR_LAUNCH((pdl_launch(k_fr_ns_update, tiles, tb, 0, s, na)));
    }
    SplitR sr{};
    sr.f.q = q; sr.hdr = hdr; sr.side = side; sr.mode = 6; sr.M = b.z; sr.out = R4;
    sr.rows = q; sr.rows_p = Qp; sr.Lp = Qp;
    FR_LAUNCH((pdl_launch(k_fr_split_r, grid_of(Qp * Qp, sms), 256, 0, s, sr)));
    return ISO_OK;
}

}  // namespace
}  // namespace iso

using namespace iso;

extern "C" {

int32_t iso_frame_workspace_size(int64_t m, int64_t n, int32_t K, size_t* bytes) {
    if (!bytes || m < 1 || n < 1 || K < 1) return ISO_ERR_ARG;
    if (K > ISO_MAX_EXPERTS) return ISO_ERR_UNSUPPORTED;
    if (m >= (1LL << 24) || n >= (1LL << 24) || std::min(m, n) > 32768) return ISO_ERR_UNSUPPORTED;
    *bytes = frame_layout(m, n, K).total;
    return ISO_OK;
}

int32_t iso_frame_merge(const double* U0, const double* S0, const double* Vt0, const double* const* U,
                        const double* const* Vt, int32_t K, int64_t m, int64_t n, const iso_tensor* W0,
                        const iso_tensor* out, const iso_frame_cfg* cfg, void* workspace, size_t ws_bytes,
                        const iso_merge_stats* stats, void* stream) {
    size_t need = 0;
    ISO_TRY(iso_frame_workspace_size(m, n, K, &need));
    if (!U0 || !S0 || !Vt0 || !U || !Vt || !W0 || !out || !cfg) return ISO_ERR_ARG;
    for (int i = 0; i < K; ++i)
        if (!U[i] || !Vt[i]) return ISO_ERR_ARG;
    auto al8 = [](const void* p) { return ((uintptr_t)p & 7u) == 0; };
    if (!al8(U0) || !al8(S0) || !al8(Vt0)) return ISO_ERR_ALIGN;
    for (int i = 0; i < K; ++i)
        if (!al8(U[i]) || !al8(Vt[i])) return ISO_ERR_ALIGN;
    if (!(cfg->rho_keep > 0.0 && cfg->rho_keep <= 1.0)) return ISO_ERR_ARG;
    if (!(cfg->ridge >= 0.0) || !std::isfinite(cfg->ridge)) return ISO_ERR_ARG;
    if (!std::isfinite(cfg->c_min) || !std::isfinite(cfg->c_max) || cfg->c_min > cfg->c_max) return ISO_ERR_ARG;
    if (cfg->ns_iters < 0 || cfg->ns_iters > FR_MAX_NS || cfg->reserved != 0) return ISO_ERR_ARG;
    if (W0->rows != m || W0->cols != n || out->rows != m || out->cols != n) return ISO_ERR_SHAPE;
    if ((W0->dtype != ISO_BF16 && W0->dtype != ISO_F32) || out->dtype != W0->dtype) return ISO_ERR_DTYPE;
    if (!W0->data || !out->data) return ISO_ERR_ARG;
    if (((uintptr_t)W0->data & 15u) || ((uintptr_t)out->data & 15u)) return ISO_ERR_ALIGN;
    if (!workspace || ((uintptr_t)workspace & 255u)) return ISO_ERR_WORKSPACE;
    if (ws_bytes < need) return ISO_ERR_WORKSPACE;
    // out may coincide with W0 (each entry is read and written by one thread);
    // it may share no other byte with an input
    {
        const size_t es = W0->dtype == ISO_BF16 ? 2 : 4;
        const uintptr_t o0 = (uintptr_t)out->data, o1 = o0 + (uintptr_t)(m * n) * es;
        const uintptr_t w0 = (uintptr_t)W0->data;
        if (o0 != w0 && o0 < w0 + (uintptr_t)(m * n) * es && w0 < o1) return ISO_ERR_ARG;
    }
    const FrameLayout L = frame_layout(m, n, K);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* ws = static_cast<char*>(workspace);
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return ISO_ERR_CUDA;
    const long long q = L.q, Qp = L.Qp;
    long long k_keep = (long long)std::floor(cfg->rho_keep * (double)q + 0.5);
    k_keep = std::max(0LL, std::min(q, k_keep));
    const int ns_iters = cfg->ns_iters ? cfg->ns_iters : FR_DEFAULT_NS;
    FrameHeader* hdr = reinterpret_cast<FrameHeader*>(ws + L.hdr);
    double* gram = reinterpret_cast<double*>(ws + L.gram);
    double* coef = reinterpret_cast<double*>(ws + L.coef);
    double* dots = reinterpret_cast<double*>(ws + L.dots);
    auto F = [&](size_t off) { return reinterpret_cast<float*>(ws + off); };
    auto D = [&](size_t off) { return reinterpret_cast<double*>(ws + off); };

    // header, Gamma, c*, the sign dots and the column dots start at zero
    if (cudaMemsetAsync(ws, 0, L.zero_end, s) != cudaSuccess) return ISO_ERR_CUDA;

    // the V side as n x q row-major frames
    Frames fr[2];
    fr[0].F0 = U0; fr[0].K = K; fr[0].d = m; fr[0].q = q;
    fr[1].F0 = D(L.vcopy); fr[1].K = K; fr[1].d = n; fr[1].q = q;
    for (int i = 0; i < MAXK; ++i) {
        fr[0].F[i] = i < K ? U[i] : nullptr;
        fr[1].F[i] = i < K ? D(L.vcopy) + (size_t)(i + 1) * n * q : nullptr;
    }
    {
        const dim3 blk(32, 8), grd((unsigned)((n + 31) / 32), (unsigned)((q + 31) / 32));
        FR_LAUNCH((pdl_launch(k_fr_transpose, grd, blk, 0, s, Vt0, D(L.vcopy), q, n)));
        for (int i = 0; i < K; ++i)
            FR_LAUNCH((pdl_launch(k_fr_transpose, grd, blk, 0, s, Vt[i], D(L.vcopy) + (size_t)(i + 1) * n * q, q, n)));
    }
    // signs (from the U frames), then the column dot products of each side
    {
        const int rc = (int)std::max(1LL, std::min(64LL, ((long long)m + 511) / 512));
        FR_LAUNCH((pdl_launch(k_fr_signdots, dim3((unsigned)((q + 31) / 32), K, rc), dim3(32, 8), 0, s, fr[0], dots, rc)));
        for (int sd = 0; sd < 2; ++sd) {
            const int r2 = (int)std::max(1LL, std::min(256LL, (fr[sd].d + 255) / 256));
            const dim3 cg((unsigned)((q + 31) / 32), r2), cb(32, 8);
            if (K == 1) FR_LAUNCH((pdl_launch(k_fr_coldots<1>, cg, cb, 0, s, fr[sd], dots, D(L.cd[sd]), r2)));
            else if (K == 2) FR_LAUNCH((pdl_launch(k_fr_coldots<2>, cg, cb, 0, s, fr[sd], dots, D(L.cd[sd]), r2)));
            else if (K == 3) FR_LAUNCH((pdl_launch(k_fr_coldots<3>, cg, cb, 0, s, fr[sd], dots, D(L.cd[sd]), r2)));
            else if (K == 4) FR_LAUNCH((pdl_launch(k_fr_coldots<4>, cg, cb, 0, s, fr[sd], dots, D(L.cd[sd]), r2)));
            else FR_LAUNCH((pdl_launch(k_fr_coldots<8>, cg, cb, 0, s, fr[sd], dots, D(L.cd[sd]), r2)));
        }
    }
    // A_i = F_0^T dF_i (binary64), then Sym_i and Kw_i
    for (int sd = 0; sd < 2; ++sd) {
        OzSrc oz{fr[sd], dots, nullptr, reinterpret_cast<unsigned long long*>(ws + L.mx[sd]),
                 reinterpret_cast<int32_t*>(ws + L.ex), Qp, reinterpret_cast<int32_t*>(ws + L.sym[sd]), D(L.cd[sd])};
        ISO_TRY(exact_product(s, sms, oz, K, D(L.aq[sd]), reinterpret_cast<unsigned char*>(ws + L.tail),
                              L.total - L.tail, &hdr->status));
        FR_LAUNCH((pdl_launch(k_fr_symskew, dim3((unsigned)(Qp / 32), (unsigned)(Qp / 32), K), dim3(32, 8), 0, s, 
            D(L.aq[sd]), Qp, q, D(L.sym[sd]), D(L.kw[sd]))));
    }
    // Gamma and c*
    {
        GramArgs ga{};
        for (int sd = 0; sd < 2; ++sd) {
            ga.A[sd] = D(L.aq[sd]); ga.sym[sd] = D(L.sym[sd]); ga.kw[sd] = D(L.kw[sd]); ga.cd[sd] = D(L.cd[sd]);
        }
        ga.S0 = S0; ga.gram = gram; ga.q = q; ga.Qp = Qp; ga.k_keep = k_keep; ga.K = K;
        const int pairs = K * (K + 1) / 2;
        const int slices = (int)std::max(1LL, std::min((long long)sms * 4, q));
        FR_LAUNCH((pdl_launch(k_fr_gram, dim3(pairs, slices), 256, 0, s, ga)));
        FR_LAUNCH((pdl_launch(k_fr_solve, 1, 32, 0, s, gram, coef, K, cfg->ridge, cfg->c_min, cfg->c_max,
                                                stats ? stats->gram : nullptr, stats ? stats->coef : nullptr)));
    }
    // per side: aggregate tangent, polar factor, motion E_F
    for (int sd = 0; sd < 2; ++sd) {
        const long long Dp = sd == 0 ? L.Mp : L.Np, d = fr[sd].d;
        SplitR sr{};
        sr.f = fr[sd]; sr.S0 = S0; sr.sym = D(L.sym[sd]); sr.kw = D(L.kw[sd]); sr.coef = coef; sr.hdr = hdr;
        sr.side = sd; sr.k_keep = k_keep;
        // Y^T, F_0, then E = F_0 Y
        sr.mode = 3; sr.out = F(L.y4[sd]); sr.rows = q; sr.rows_p = Qp; sr.Lp = Qp;
        FR_LAUNCH((pdl_launch(k_fr_split_r, grid_of(Qp * Qp, sms), 256, 0, s, sr)));
        sr.mode = 0; sr.out = F(L.fr4[sd]); sr.rows = d; sr.rows_p = Dp; sr.Lp = Qp;
        FR_LAUNCH((pdl_launch(k_fr_split_r, grid_of(Dp * Qp, sms), 256, 0, s, sr)));
        {
            GemmArgs g{};
            g.mode = GEMM_STORE_F32; g.C = F(L.e[sd]); g.ldc = Qp; g.M = (int)Dp; g.N = (int)Qp; g.status = &hdr->status;
            ISO_TRY(frame_gemm(s, sms, F(L.fr4[sd]), Dp, F(L.y4[sd]), Qp, Qp, g));
        }
        FR_LAUNCH((pdl_launch(k_fr_xi, grid_of(d * q, sms), 256, 0, s, fr[sd], dots, coef, F(L.e[sd]), Qp, k_keep, D(L.xi[sd]))));
        // N = xi*^T xi*
        {
            SplitT st{};
            st.d = fr[sd].d; st.q = q; st.X = D(L.xi[sd]); st.out = F(L.ft4[sd]); st.Dp = Dp; st.Qp = Qp;
            FR_LAUNCH((pdl_launch(k_fr_split_t, dim3((unsigned)(Dp / 32), (unsigned)(Qp / 32)), dim3(32, 8), 0, s, st)));
            GemmArgs g{};
            g.mode = GEMM_STORE_F32; g.C = F(L.nq[sd]); g.ldc = Qp; g.M = (int)Qp; g.N = (int)Qp; g.status = &hdr->status;
            ISO_TRY(frame_gemm(s, sms, F(L.ft4[sd]), Qp, F(L.ft4[sd]), Qp, Dp, g));
        }
        // (I + N)^(-1/2) = I + R by the difference-form Newton-Schulz iteration,
        // then F_0 + xi*, and E_F = xi* + (F_0 + xi*) R
        {
            NsBufs nb{D(L.ns_y), D(L.ns_z), D(L.ns_m), F(L.ns_y4), F(L.ns_z4), F(L.ns_m4), F(L.ns_t1),
                      F(L.ns_t2), F(L.ns_t3)};
            ISO_TRY(ns_root(s, sms, hdr, sd, F(L.nq[sd]), nullptr, q, Qp, nb, ns_iters, F(L.y4[sd])));
        }
        sr.mode = 1; sr.X = D(L.xi[sd]); sr.out = F(L.fr4[sd]); sr.rows = d; sr.rows_p = Dp; sr.Lp = Qp;
        FR_LAUNCH((pdl_launch(k_fr_split_r, grid_of(Dp * Qp, sms), 256, 0, s, sr)));
        {
            GemmArgs g{};
            g.mode = GEMM_STORE_F32; g.C = F(L.e[sd]); g.ldc = Qp; g.M = (int)Dp; g.N = (int)Qp; g.status = &hdr->status;
            ISO_TRY(frame_gemm(s, sms, F(L.fr4[sd]), Dp, F(L.y4[sd]), Qp, Qp, g));
        }
        FR_LAUNCH((pdl_launch(k_fr_motion, grid_of(d * q, sms), 256, 0, s, D(L.xi[sd]), F(L.e[sd]), Qp, d, q)));
        // the reconstruction's operand of this side
        sr.X = D(L.xi[sd]);
        sr.mode = sd == 0 ? 4 : 5;
        sr.out = F(sd == 0 ? L.a6 : L.b6);
        sr.rows = d; sr.rows_p = Dp; sr.Lp = 2 * Qp;
        FR_LAUNCH((pdl_launch(k_fr_split_r, grid_of(Dp * 2 * Qp, sms), 256, 0, s, sr)));
    }
    // W* = W_0 + [E_U S_0 | U_0 S_0] [V* | E_V]^T
    {
        GemmArgs g{};
        g.mode = GEMM_ADD_BASE; g.M = (int)m; g.N = (int)n; g.out = out->data; g.w0 = W0->data; g.ldo = n;
        g.out_dtype = W0->dtype; g.status = &hdr->status;
        ISO_TRY(frame_gemm(s, sms, F(L.a6), L.Mp, F(L.b6), L.Np, 2 * Qp, g));
    }
    if (stats && stats->status) FR_LAUNCH((pdl_launch(k_fr_status, 1, 32, 0, s, hdr, stats->status)));
    return ISO_OK;
}

int32_t iso_opt_workspace_size(int64_t m, int64_t n, size_t* bytes) {
    if (!bytes || m < 1 || n < 1) return ISO_ERR_ARG;
    if (m >= (1LL << 24) || n >= (1LL << 24) || std::min(m, n) > 32768) return ISO_ERR_UNSUPPORTED;
    *bytes = opt_layout(m, n).total;
    return ISO_OK;
}

int32_t iso_opt_step(double* U, double* V, const double* S0, const iso_tensor* G_W, float* mU, float* vU,
                     float* mV, float* vV, const iso_tensor* W, const iso_tensor* W_out, int64_t m, int64_t n,
                     const iso_adamw_cfg* cfg, void* workspace, size_t ws_bytes, const iso_merge_stats* stats,
                     void* stream) {
    size_t need = 0;
    ISO_TRY(iso_opt_workspace_size(m, n, &need));
    if (!U || !V || !S0 || !G_W || !mU || !vU || !mV || !vV || !W || !W_out || !cfg) return ISO_ERR_ARG;
    auto al8 = [](const void* p) { return ((uintptr_t)p & 7u) == 0; };
    auto al4 = [](const void* p) { return ((uintptr_t)p & 3u) == 0; };
    if (!al8(U) || !al8(V) || !al8(S0) || !al4(mU) || !al4(vU) || !al4(mV) || !al4(vV)) return ISO_ERR_ALIGN;
    if (!(cfg->lr >= 0.0) || !std::isfinite(cfg->lr)) return ISO_ERR_ARG;
    if (!(cfg->beta1 >= 0.0 && cfg->beta1 < 1.0) || !(cfg->beta2 >= 0.0 && cfg->beta2 < 1.0)) return ISO_ERR_ARG;
    if (!(cfg->eps > 0.0) || !std::isfinite(cfg->eps)) return ISO_ERR_ARG;
    if (!(cfg->weight_decay >= 0.0) || !std::isfinite(cfg->weight_decay)) return ISO_ERR_ARG;
    if (cfg->step < 1 || cfg->ns_iters < 0 || cfg->ns_iters > FR_MAX_NS || cfg->reserved != 0) return ISO_ERR_ARG;
    for (const iso_tensor* t : {G_W, W, W_out}) {
        if (t->rows != m || t->cols != n) return ISO_ERR_SHAPE;
        if (t->dtype != ISO_BF16 && t->dtype != ISO_F32) return ISO_ERR_DTYPE;
        if (!t->data) return ISO_ERR_ARG;
        if ((uintptr_t)t->data & 15u) return ISO_ERR_ALIGN;
    }
    if (W_out->dtype != W->dtype) return ISO_ERR_DTYPE;
    {
        const size_t es = W->dtype == ISO_BF16 ? 2 : 4;
        const uintptr_t o0 = (uintptr_t)W_out->data, o1 = o0 + (uintptr_t)(m * n) * es, w0 = (uintptr_t)W->data;
        if (o0 != w0 && o0 < w0 + (uintptr_t)(m * n) * es && w0 < o1) return ISO_ERR_ARG;
    }
    if (!workspace || ((uintptr_t)workspace & 255u)) return ISO_ERR_WORKSPACE;
    if (ws_bytes < need) return ISO_ERR_WORKSPACE;
    const OptLayout L = opt_layout(m, n);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* ws = static_cast<char*>(workspace);
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return ISO_ERR_CUDA;
    const long long q = L.q, Qp = L.Qp;
    const int ns_iters = cfg->ns_iters ? cfg->ns_iters : FR_DEFAULT_NS;
    FrameHeader* hdr = reinterpret_cast<FrameHeader*>(ws + L.hdr);
    auto F = [&](size_t off) { return reinterpret_cast<float*>(ws + off); };
    auto D = [&](size_t off) { return reinterpret_cast<double*>(ws + off); };
    if (cudaMemsetAsync(ws + L.hdr, 0, L.zero_end - L.hdr, s) != cudaSuccess) return ISO_ERR_CUDA;

    Frames fr[2];
    fr[0] = Frames{}; fr[0].F0 = U; fr[0].d = m; fr[0].q = q;
    fr[1] = Frames{}; fr[1].F0 = V; fr[1].d = n; fr[1].q = q;
    // operands of the factor gradients G_U = G_W (V S_0), G_V = G_W^T (U S_0)
    FR_LAUNCH((pdl_launch(k_op_split_g, grid_of(L.Mp * L.Np, sms), 256, 0, s, G_W->data, G_W->dtype, m, n, L.Mp, L.Np,
                                                                      F(L.gw4))));
    FR_LAUNCH((pdl_launch(k_op_split_gt, dim3((unsigned)(L.Mp / 32), (unsigned)(L.Np / 32)), dim3(32, 8), 0, s, 
        G_W->data, G_W->dtype, m, n, L.Mp, L.Np, F(L.gwt4))));
    for (int sd = 0; sd < 2; ++sd) {
        SplitT st{};
        st.d = fr[sd].d; st.q = q; st.X = sd == 0 ? U : V; st.S0 = S0; st.Dp = sd == 0 ? L.Mp : L.Np; st.Qp = Qp;
        st.out = F(sd == 0 ? L.su4 : L.sv4);
        FR_LAUNCH((pdl_launch(k_fr_split_t, dim3((unsigned)(st.Dp / 32), (unsigned)(Qp / 32)), dim3(32, 8), 0, s, st)));
    }
    // the factor gradients on the tensor cores with AdamW in the epilogue:
    // dF = F_bar - F, the moments updated in place
    const double bc1 = 1.0 - std::pow(cfg->beta1, (double)cfg->step);
    const double bc2 = 1.0 - std::pow(cfg->beta2, (double)cfg->step);
    for (int sd = 0; sd < 2; ++sd) {
        GemmArgs g{};
        g.mode = GEMM_ADAMW; g.M = (int)(sd == 0 ? m : n); g.N = (int)q; g.ldo = q; g.status = &hdr->status;
        g.adam = AdamwArgs{sd == 0 ? U : V, sd == 0 ? mU : mV, sd == 0 ? vU : vV, D(L.dF[sd]),
                           cfg->beta1, cfg->beta2, cfg->eps, cfg->lr * cfg->weight_decay, cfg->lr / bc1, 1.0 / bc2};
        if (sd == 0) ISO_TRY(frame_gemm(s, sms, F(L.gw4), L.Mp, F(L.sv4), Qp, L.Np, g));
        else ISO_TRY(frame_gemm(s, sms, F(L.gwt4), L.Np, F(L.su4), Qp, L.Mp, g));
    }
    // the polar retraction of each side: N = (F + dF)^T (F + dF) - I in
    // binary64, R = (I + N)^(-1/2) - I, E_F = dF + (F + dF) R
    for (int sd = 0; sd < 2; ++sd) {
        const long long Dp = sd == 0 ? L.Mp : L.Np, d = fr[sd].d;
        OzSrc oz{fr[sd], nullptr, D(L.dF[sd]), reinterpret_cast<unsigned long long*>(ws + L.mx[sd]),
                 reinterpret_cast<int32_t*>(ws + L.ex), Qp, reinterpret_cast<int32_t*>(ws + L.ns_y), nullptr};
        ISO_TRY(exact_product(s, sms, oz, 0, D(L.n64), reinterpret_cast<unsigned char*>(ws + L.gw4),
                              L.dF[0] - L.gw4, &hdr->status));
        NsBufs nb{D(L.ns_y), D(L.ns_z), D(L.ns_m), F(L.ns_y4), F(L.ns_z4), F(L.ns_m4), F(L.ns_t1),
                  F(L.ns_t2), F(L.ns_t3)};
        ISO_TRY(ns_root(s, sms, hdr, sd, nullptr, D(L.n64), q, Qp, nb, ns_iters, F(L.r4)));
        SplitR sr{};
        sr.f = fr[sd]; sr.X = D(L.dF[sd]); sr.mode = 1; sr.out = F(L.xb4); sr.rows = d; sr.rows_p = Dp; sr.Lp = Qp;
        FR_LAUNCH((pdl_launch(k_fr_split_r, grid_of(Dp * Qp, sms), 256, 0, s, sr)));
        {
            GemmArgs g{};
            g.mode = GEMM_STORE_F32; g.C = F(L.p); g.ldc = Qp; g.M = (int)Dp; g.N = (int)Qp; g.status = &hdr->status;
            ISO_TRY(frame_gemm(s, sms, F(L.xb4), Dp, F(L.r4), Qp, Qp, g));
        }
        FR_LAUNCH((pdl_launch(k_fr_motion, grid_of(d * q, sms), 256, 0, s, D(L.dF[sd]), F(L.p), Qp, d, q)));
        // the reconstruction's operand of this side ([E_U S_0 | U S_0] or [V + E_V | E_V])
        sr.S0 = S0; sr.X = D(L.dF[sd]); sr.mode = sd == 0 ? 4 : 5; sr.out = F(sd == 0 ? L.a6 : L.b6);
        sr.rows = d; sr.rows_p = Dp; sr.Lp = 2 * Qp;
        FR_LAUNCH((pdl_launch(k_fr_split_r, grid_of(Dp * 2 * Qp, sms), 256, 0, s, sr)));
    }
    // F+ = F + E_F, then W+ = W + [E_U S_0 | U S_0] [V+ | E_V]^T
    FR_LAUNCH((pdl_launch(k_op_add, grid_of(m * q, sms), 256, 0, s, U, D(L.dF[0]), m * q)));
    FR_LAUNCH((pdl_launch(k_op_add, grid_of(n * q, sms), 256, 0, s, V, D(L.dF[1]), n * q)));
    {
        GemmArgs g{};
        g.mode = GEMM_ADD_BASE; g.M = (int)m; g.N = (int)n; g.out = W_out->data; g.w0 = W->data; g.ldo = n;
        g.out_dtype = W->dtype; g.status = &hdr->status;
        ISO_TRY(frame_gemm(s, sms, F(L.a6), L.Mp, F(L.b6), L.Np, 2 * Qp, g));
    }
    if (stats && stats->status) FR_LAUNCH((pdl_launch(k_fr_status, 1, 32, 0, s, hdr, stats->status)));
    return ISO_OK;
}

// The split product on its own, for tests and timing
int32_t iso_gemm_x3(const float* A, const float* B, const float* A2, const float* B2, float* C, float* C2,
                    const iso_tensor* W0, const iso_tensor* out, int64_t M, int64_t N, int64_t Kc, int32_t width,
                    void* stream) {
    if (!A || !B || !A2 != !B2 || !A2 != !C2 || !W0 != !out || !C == !out || (out && A2)) return ISO_ERR_ARG;
    if (M <= 0 || N <= 0 || Kc <= 0 || (width != 0 && width != 128 && width != 256)) return ISO_ERR_ARG;
    if (M % GEMM_BM || N % GEMM_BN || Kc % GEMM_BK) return ISO_ERR_SHAPE;
    if (M >= (1LL << 23) || N >= (1LL << 23) || Kc >= (1LL << 28)) return ISO_ERR_UNSUPPORTED;
    for (const float* p : {A, B, A2, B2, static_cast<const float*>(C), static_cast<const float*>(C2)})
        if ((uintptr_t)p & 15u) return ISO_ERR_ALIGN;
    GemmArgs g{};
    g.mode = GEMM_STORE_F32; g.C = C; g.C2 = C2; g.ldc = N; g.M = (int)M; g.N = (int)N;
    if (out) {
        if (W0->rows != out->rows || W0->cols != out->cols || out->rows < 1 || out->cols < 1 || out->rows > M || out->cols > N)
            return ISO_ERR_SHAPE;
        if ((W0->dtype != ISO_BF16 && W0->dtype != ISO_F32) || out->dtype != W0->dtype) return ISO_ERR_DTYPE;
        if (!W0->data || !out->data) return ISO_ERR_ARG;
        if (((uintptr_t)W0->data & 15u) || ((uintptr_t)out->data & 15u)) return ISO_ERR_ALIGN;
        g.mode = GEMM_ADD_BASE; g.M = (int)out->rows; g.N = (int)out->cols; g.out = out->data; g.w0 = W0->data;
        g.ldo = out->cols; g.out_dtype = out->dtype;
    }
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return ISO_ERR_CUDA;
    return frame_gemm(static_cast<cudaStream_t>(stream), sms, A, M, B, N, Kc, g, A2, B2, width);
}

// A plain tcgen05 product on its own: C (M x N,
// ldc) = A[:, a_k0 : a_k0 + Kc] B[:, b_k0 : b_k0 + Kc]^T with A (M x lda) and
// B (N x ldb) row-major binary32 read as tf32.
int32_t iso_gemm_tf32(const float* A, int64_t lda, const float* B, int64_t ldb, float* C, int64_t ldc, int64_t M,
                      int64_t N, int64_t Kc, int64_t a_k0, int64_t b_k0, void* stream) {
    if (!A || !B || !C) return ISO_ERR_ARG;
    if (M <= 0 || N <= 0 || Kc <= 0 || a_k0 < 0 || b_k0 < 0) return ISO_ERR_ARG;
    if (M % GEMM_BM || N % GEMM_BN || Kc % GEMM_BK || a_k0 % GEMM_BK || b_k0 % GEMM_BK) return ISO_ERR_SHAPE;
    if (a_k0 + Kc > lda || b_k0 + Kc > ldb || ldc < N || lda % 4 || ldb % 4 || ldc % 4) return ISO_ERR_SHAPE;
    if (M >= (1LL << 31) || N >= (1LL << 31) || lda >= (1LL << 31) || ldb >= (1LL << 31)) return ISO_ERR_UNSUPPORTED;
    if (((uintptr_t)A & 15u) || ((uintptr_t)B & 15u) || ((uintptr_t)C & 15u)) return ISO_ERR_ALIGN;
    CUtensorMap ta, tb;
    ISO_TRY(gemm_tensor_map(&ta, A, M, lda, lda));
    ISO_TRY(gemm_tensor_map(&tb, B, N, ldb, ldb));
    ISO_TRY(smem_optin<k_gemm_tf32>(GEMM_SMEM));
    GemmArgs g{};
    g.mode = GEMM_STORE_F32; g.C = C; g.ldc = ldc; g.M = (int)M; g.N = (int)N;
    g.k_tiles = (int)(Kc / GEMM_BK); g.a_k0 = (int)a_k0; g.b_k0 = (int)b_k0;
    const int slot = prof_begin(0, static_cast<cudaStream_t>(stream));
    k_gemm_tf32<<<dim3((unsigned)(N / GEMM_BN), (unsigned)(M / GEMM_BM)), GEMM_THREADS, GEMM_SMEM,
                  static_cast<cudaStream_t>(stream)>>>(ta, tb, g);
    prof_end(slot, static_cast<cudaStream_t>(stream));
    return cudaGetLastError() == cudaSuccess ? ISO_OK : ISO_ERR_CUDA;
}

}  // extern "C"
