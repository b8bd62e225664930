// iso_gemm.cuh -- the dense contractions of the frame-space merge and the
// optimizer step on the fifth-generation tensor cores: C = A B^T for row-major
// fp32 operands read as tf32, with tcgen05.mma accumulating in tensor memory.
//
// k_gemm_tf32: one product (iso_gemm_tf32 alone; the merge and the step run the
// kernels after it).  One CTA of 128 threads computes one 128 x 128
// tile of C:
//   warp 0, lane 0  loads the operand tiles (TMA, 128 rows x 32 fp32 = 128 B
//                   per row, 128-byte swizzle) into a GEMM_STAGES-deep ring,
//                   one mbarrier per stage counting the copied bytes;
//   warp 1, lane 0  issues four tcgen05.mma (K = 8 each) per stage into a
//                   128-lane x 128-column fp32 accumulator in tensor memory and
//                   frees the stage with tcgen05.commit;
//   all four warps  read the accumulator back with tcgen05.ld (warp w owns
//                   lanes 32 w .. 32 w + 31, one output row per thread) and
//                   store it (the epilogue).
// k_gemm_x3: the three products hi hi + hi lo + lo hi of split operands (x =
// hi + lo, stored as two segments [hi | lo] of each row), the same roles.  A
// stage holds the hi and lo tiles of both operands, so each is loaded once for
// the products it enters, and the two small products have an accumulator of
// their own: their sum is added once, in the epilogue.  Tiles of 128 x 256
// (two stages of 96 KB) or 128 x 128 (three of 64 KB).  What bounds it is the
// path from L2 to the SMs: three products over three separate segments with
// 128 x 128 tiles asked for 128 bytes per clock and SM and ran at 0.46 of the
// tf32 rate; this form asks for 62.  All products of the frame merge of a 3584
// x 18944 matrix: 59.2 -> 31.9 ms.
// Every wait on a barrier is bounded; a wait that gives up records
// ISO_ERR_TIMEOUT, and the kernel still waits (bounded) for its own copies and
// products before it frees its tensor memory and returns.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace iso {

constexpr int GEMM_BM = 128;               // rows of A (and of C) per CTA
constexpr int GEMM_BN = 128;               // rows of B (columns of C) per CTA
constexpr int GEMM_BK = 32;                // contraction elements (fp32) per stage: 128 bytes
constexpr int GEMM_STAGES = 6;
constexpr int GEMM_TILE_BYTES = GEMM_BM * GEMM_BK * 4;                 // 16 KB per operand tile
constexpr int GEMM_SMEM = 1024 + GEMM_STAGES * 2 * GEMM_TILE_BYTES + 256;
constexpr int GEMM_THREADS = 128;

enum GemmEpilogue : int32_t {
    GEMM_STORE_F32 = 0,   // C[row * ldc + col] = acc (the tile is inside C's padded extents)
    GEMM_ADD_BASE = 1,    // out[row * ldo + col] = W0[row * ldo + col] + acc for row < M, col < N
    GEMM_ADAMW = 2        // acc is the gradient of the binary64 variable X (row < M, col < N, row
                          // stride ldo): AdamW moments updated in place, the step X_bar - X stored
};

// AdamW on a binary64 variable in the product's epilogue (decoupled weight
// decay, bias-corrected moments kept in binary32, arithmetic in binary64)
struct AdamwArgs {
    const double* X;      // the variable (read)
    float* m;             // first moment (in place)
    float* v;             // second moment (in place)
    double* dX;           // out: X_bar - X = -lr wd X - lr / bc1 * m / (sqrt(v / bc2) + eps)
    double beta1, beta2, eps;
    double lr_wd, lr_bc1, ibc2;   // lr wd, lr / bc1, 1 / bc2
};

constexpr int X3_SMEM = 1024 + 192 * 1024 + 256;   // both tile shapes
struct GemmArgs {
    int32_t M, N;         // output extents (GEMM_ADD_BASE stores only inside them)
    int32_t k_tiles;      // contraction length / GEMM_BK
    int32_t a_k0, b_k0;   // k_gemm_tf32: first contraction column read from A's and B's arrays
    int32_t seg;          // k_gemm_x3: columns of one segment (the lo segment starts there)
    int32_t c_cols;       // k_gemm_x3: padded columns of C (a 256-wide tile may reach past them)
    int32_t mode;         // GemmEpilogue
    float* C;
    float* C2;            // k_gemm_x3: the output of the second product (grid z = 1)
    long long ldc;
    void* out;            // GEMM_ADD_BASE: output and base (same dtype, iso_dtype out_dtype)
    const void* w0;
    long long ldo;
    int32_t out_dtype;
    int32_t pad;
    const int32_t* skip;  // k_gemm_x3, optional: the whole grid returns at once while *skip != 0
    int32_t* status;      // header status word for ISO_ERR_TIMEOUT
    AdamwArgs adam;       // GEMM_ADAMW
};

__global__ void k_gemm_tf32(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
                            GemmArgs g);
template <int BN>
__global__ void k_gemm_x3(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
                          const __grid_constant__ CUtensorMap ta2, const __grid_constant__ CUtensorMap tb2, GemmArgs g);

// ---------------------------------------------------------------------------
// Binary64 contractions on the tensor cores: C = A^T B for binary64 columns,
// from integer slices whose products and sums are exact in binary32 (the
// error-free splitting of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 59, 2012).
//
// A column x with |x_r| < 2^e is written x_r = 2^(e - 7) sum_t d_t 2^(-8 t),
// t = 0 .. 6, with integer digits |d_t| <= 128 (x rounded to 55 fractional
// bits below 2^e), stored as bf16, which holds them exactly.  Then
//   C_kl = 2^(e_k + e_l - 14) sum_g 2^(-8 g) I_g,  I_g = sum_{s + t = g} <a_s, b_t>
// over g = 0 .. 6 (28 of the 49 slice pairs).  Over d rows the pairs left out
// come to about sqrt(d) 2^-56.3 2^(e_k + e_l), at most 6.1 d 2^-56 2^(e_k +
// e_l), and the rounding of the columns to 2^-56.8 (2^e_k |b| + 2^e_l |a|): for
// dense columns less than the rounding of a binary64 sum, for columns whose
// largest entry holds much of their norm more.  Those are told apart by
// k_oz_columns, which has the figures, and summed in binary64 by k_oz_f64.
// The bounds are on the columns' norms: where two dense columns hardly overlap,
// their product is off by that much of |a| |b|, not of sum |a_r b_r|.
// Each I_g accumulates in tensor
// memory as binary32 over at most OZ_STEPS_* steps, which keeps every partial
// sum at or below 2^24 whatever the digits (an exact integer), and is then
// added to 64-bit integers in registers.
//
// Operand layout: slab (kt, c) holds columns 128 kt .. + 127, rows 16 c ..
// + 15 of all seven slices, slice after slice, each 4 KB in the core-matrix
// order the products read from shared memory (8 columns x 8 rows of 128
// bytes; row halves 128 bytes apart, column groups 256 bytes apart), so one
// bulk copy brings a slab and no tensor map or swizzle is needed.
//
// Measured on one 3584 x 18944 matrix (q = 3584): A_i of three experts, both
// sides, 1441 ms as binary64 on the CUDA cores (64 x 64 tiles, 1.2 TFLOP/s,
// the chip's binary64 rate) against 34 ms here (28 bf16 products for each: 1.4
// PFLOP/s).  The optimizer step of a 1536 x 8960
// matrix was bound by F^T F: 22.6 -> 1.0 ms.
constexpr int OZ_SLICES = 7;
constexpr int OZ_BM = 128;                              // columns of A (and of B) per tile
constexpr int OZ_BK = 16;                               // contraction rows per step
constexpr int OZ_SLICE_BYTES = OZ_BM * OZ_BK * 2;       // 4 KB
constexpr int OZ_SLAB_BYTES = OZ_SLICES * OZ_SLICE_BYTES;
constexpr int OZ_STAGES = 3;
constexpr int OZ_EPI_WARPS = 8;
constexpr int OZ_THREADS = 64 + 32 * OZ_EPI_WARPS;
constexpr int OZ_SMEM = 128 + OZ_STAGES * 2 * OZ_SLAB_BYTES + 256;
// Two sweeps over the contraction (a group takes 128 of the 512 tensor-memory
// columns): groups 0 .. 3 read slices 0 .. 3, groups 4 .. 6 all seven, which
// leaves the sweep with most of the work a fourth accumulator to drain into
// registers behind the products.  Steps per drain: (group + 1) pairs x 16 rows
// x 2^14 <= 2^24.
constexpr int OZ_HIGH = 4;                              // groups of the first sweep
constexpr int OZ_STEPS_HIGH = 16;                       // 4 pairs x 256 rows <= 1024
constexpr int OZ_STEPS_LOW = 9;                         // 7 pairs x 144 rows <= 1024
// 64-bit totals: |I_g| 2^(8 (3 - g)) summed over g = 0 .. 3 stays below 2^63
constexpr long long OZ_MAX_ROWS = 1LL << 20;
constexpr int32_t OZ_NONFINITE = 1 << 20;               // exponent of a column holding a NaN or an infinity

struct OzArgs {
    const unsigned char* A;   // slabs [kt][chunk]
    const unsigned char* B;   // expert z at B + z * b_stride
    unsigned long long b_stride;
    const int32_t* ea;        // column exponents of A; of B at eb + z * eb_stride
    const int32_t* eb;
    long long eb_stride;
    double* C;                // q x q, row stride q; expert z at C + z * c_stride
    long long c_stride;
    double* part;             // split contraction: [split][z][q][q] partial sums (NULL: C is written)
    long long q;
    int32_t tiles;            // tiles a side
    int32_t chunks;           // 16-row chunks of the contraction
    int32_t per_split;        // chunks per split (gridDim.y splits)
    int32_t symmetric;        // A == B: tiles on and above the diagonal, written to both halves
    int32_t minus_identity;   // subtract I (with one split only; k_oz_reduce otherwise)
    int32_t* status;
};
__global__ void k_oz_gemm(OzArgs g);

// Host side: a 2-D tensor map over a row-major fp32 array of `rows` x `cols`
// (cols a multiple of 4, rows and the row stride as given) with a 32 x 128
// box and the 128-byte swizzle the kernel's shared-memory descriptors expect.
int gemm_tensor_map(CUtensorMap* map, const float* base, long long rows, long long cols, long long ld);

// Launch accounting and per-kind device timing shared with the rest of the
// library (iso_api.cu): kind 0 = the tensor-core products, 1 = the other
// frame-merge and optimizer kernels, 2 = the range selection kernels
// (iso_range.cu).  prof_begin returns a slot (or -1 when profiling is
// off); prof_end records the end event and counts the launch.
int prof_begin(int frame_kind, cudaStream_t s);
void prof_end(int slot, cudaStream_t s);

#define ISO_TRY(x) do { int _r = (x); if (_r != ISO_OK) return _r; } while (0)

}  // namespace iso
