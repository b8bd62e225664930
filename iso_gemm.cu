// iso_gemm.cu -- tcgen05 / TMEM / TMA GEMM for the frame-space merge (see
// iso_gemm.cuh for the structure).
#include "iso_gemm.cuh"
#include "iso_internal.cuh"

#include <mutex>
#include <type_traits>

namespace iso {

namespace {

// Shared-memory matrix descriptor of one K-major operand tile in the
// 128-byte swizzle: rows of 128 bytes, 8-row (1024-byte) swizzle atoms
// stacked along M/N (stride 1024 bytes), one atom along K.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);          // start address
    d |= (uint64_t)1u << 16;                            // leading byte offset (unused here)
    d |= (uint64_t)((1024u >> 4) & 0x3FFFu) << 32;      // stride byte offset: one 8-row atom
    d |= (uint64_t)1u << 46;                            // descriptor version of sm_100
    d |= (uint64_t)2u << 61;                            // layout: 128-byte swizzle
    return d;
}

// Instruction descriptor of tcgen05.mma kind::tf32: fp32 accumulator, tf32
// A and B, both K-major, M = 128, N = 128.
constexpr uint32_t UMMA_IDESC = (1u << 4)               // D format: f32
                              | (2u << 7)               // A format: tf32
                              | (2u << 10)              // B format: tf32
                              | ((uint32_t)(GEMM_BN >> 3) << 17)
                              | ((uint32_t)(GEMM_BM >> 4) << 24);

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar) : "memory");
}

__device__ __forceinline__ void umma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
                 :: "r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(UMMA_IDESC), "r"(accumulate) : "memory");
}

// The products of one warp run in warp-uniform control flow with one elected
// lane issuing them: descriptors and accumulator addresses then live in
// uniform registers.  A single-lane branch around the whole loop moved each of
// them there per product, and a 64-clock product took 100 (k_gemm_x3<128>) to
// 140 clocks (k_oz_gemm).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// KIND 0: tf32, 1: bf16; descriptors as their low words (the high word is
// the same for both operands)
template <int KIND>
__device__ __forceinline__ void umma_lo(uint32_t tmem_d, uint32_t alo, uint32_t blo, uint32_t hi, uint32_t idesc,
                                        uint32_t accumulate) {
    if (KIND == 0)
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %5, 0;\n\t"
                     "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
                     "tcgen05.mma.cta_group::1.kind::tf32 [%0], da, db, %4, p;\n\t}"
                     :: "r"(tmem_d), "r"(alo), "r"(blo), "r"(hi), "r"(idesc), "r"(accumulate) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %5, 0;\n\t"
                     "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}"
                     :: "r"(tmem_d), "r"(alo), "r"(blo), "r"(hi), "r"(idesc), "r"(accumulate) : "memory");
}

// arrive on `bar` once every tcgen05.mma this thread issued before has completed
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :: "r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 consecutive fp32 columns of this thread's accumulator row
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                   "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
                   "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
                   "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
                   "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}

// bounded wait on one barrier phase; false once the limit is reached or
// another thread of the CTA gave up already
__device__ __forceinline__ bool wait_phase(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    for (int spin = 0; spin < MBAR_SPIN_LIMIT; ++spin) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((spin & 1023) == 1023 && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
// The same for a whole warp, with one answer for all of its lanes: what
// follows (tensor-memory loads, products, shuffles) takes every lane.
__device__ __forceinline__ bool wait_phase_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    return __all_sync(0xFFFFFFFFu, wait_phase(bar, parity, abort_flag));
}

// c / (sqrt(x) + eps) in binary64.  The division and square root instructions'
// sequences made up most of the epilogue's binary64 work; here a binary32
// reciprocal square root and reciprocal are refined (Newton-Raphson; the last
// step of each forms the residual and adds the correction with one rounding,
// as in Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", 1990).  The approximation entering the last step is
// good to 2^-43, so root and quotient are off by at most half an ulp + 2^-30
// ulp: the rounded values but for near-ties.  That holds while x and the
// divisor are in binary32's comfortable range and c is far from binary64's
// ends; everything else takes the library's.
__device__ __forceinline__ double over_root(double c, double x, double eps) {
    const float xf = (float)x;
    const uint32_t hc = (uint32_t)__double2hiint(c) & 0x7FFFFFFFu;
    const bool plain = xf > 1e-30f && xf < 1e30f && (uint32_t)__double2hiint(eps) < 0x46300000u     // eps < 2^100
                       && (hc - 0x07B00000u < 0x78300000u - 0x07B00000u                             // 2^-900 <= |c| < 2^900
                           || (hc | (uint32_t)__double2loint(c)) == 0);
    if (!plain) return c / (sqrt(x) + eps);
    const double r0 = (double)rsqrtf(xf);
    const double r1 = fma(0.5 * r0, fma(-x * r0, r0, 1.0), r0);       // 1 / sqrt(x) to about 2^-43
    const double s0 = x * r1;
    const double d = fma(fma(-s0, s0, x), 0.5 * r1, s0) + eps;
    const double i0 = (double)__frcp_rn((float)d);
    const double i1 = fma(fma(-d, i0, 1.0), i0, i0);                  // 1 / d to about 2^-46
    const double q = c * i1;
    return fma(fma(-d, q, c), i1, q);
}

// one entry of the AdamW epilogue (a call, so that the unrolled columns stay
// in registers without 32 copies of the binary64 code)
__device__ __noinline__ void adamw_entry(const AdamwArgs& a, long long e, float grad) {
    const double gr = (double)grad;
    const double mm = a.beta1 * (double)a.m[e] + (1.0 - a.beta1) * gr;
    const double vv = a.beta2 * (double)a.v[e] + (1.0 - a.beta2) * gr * gr;
    a.m[e] = (float)mm;
    a.v[e] = (float)vv;
    a.dX[e] = -a.lr_wd * a.X[e] - over_root(a.lr_bc1 * mm, vv * a.ibc2, a.eps);
}

// one row's 32 accumulated columns from col0 on, by epilogue mode
__device__ __forceinline__ void gemm_store32(const GemmArgs& g, float* C, long long row, int col0, const float (&v)[32]) {
    if (g.mode == GEMM_STORE_F32) {
        float4* dst = reinterpret_cast<float4*>(C + row * g.ldc + col0);
#pragma unroll
        for (int j = 0; j < 8; ++j) dst[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    } else if (g.mode == GEMM_ADAMW) {
        if (row < g.M) {
            const AdamwArgs& a = g.adam;
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (col0 + j < g.N) adamw_entry(a, row * g.ldo + col0 + j, v[j]);
        }
    } else if (row < g.M) {
        if (g.out_dtype == ISO_BF16) {
            const unsigned short* w = static_cast<const unsigned short*>(g.w0) + row * g.ldo;
            __nv_bfloat16* o = static_cast<__nv_bfloat16*>(g.out) + row * g.ldo;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const int col = col0 + j;
                if (col < g.N) o[col] = __float2bfloat16_rn(__fadd_rn(__uint_as_float((uint32_t)w[col] << 16), v[j]));
            }
        } else {
            const float* w = static_cast<const float*>(g.w0) + row * g.ldo;
            float* o = static_cast<float*>(g.out) + row * g.ldo;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const int col = col0 + j;
                if (col < g.N) o[col] = __fadd_rn(w[col], v[j]);
            }
        }
    }
}

}  // namespace

__global__ void __launch_bounds__(GEMM_THREADS, 1)
k_gemm_tf32(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, GemmArgs g) {
    extern __shared__ unsigned char gemm_smem_raw[];
    unsigned char* const smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(gemm_smem_raw) + 1023) & ~(uintptr_t)1023);
    unsigned char* const sa = smem;                                        // [stage] A tiles
    unsigned char* const sb = smem + GEMM_STAGES * GEMM_TILE_BYTES;        // [stage] B tiles
    uint64_t* const bars = reinterpret_cast<uint64_t*>(smem + 2 * GEMM_STAGES * GEMM_TILE_BYTES);
    // bars[0, S): full (bytes landed), bars[S, 2S): empty (products done), bars[2S]: accumulator ready
    uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * GEMM_STAGES + 1);
    volatile int* const abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * GEMM_BM, n0 = blockIdx.x * GEMM_BN;
    const uint32_t sa_s = smem_u32(sa), sb_s = smem_u32(sb), bar_s = smem_u32(bars);
    auto full_bar = [&](int s) { return bar_s + 8u * s; };
    auto empty_bar = [&](int s) { return bar_s + 8u * (GEMM_STAGES + s); };
    const uint32_t accum_bar = bar_s + 8u * (2 * GEMM_STAGES);

    if (threadIdx.x == 0) {
        for (int s = 0; s < GEMM_STAGES; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        mbar_init(accum_bar, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(tmem_slot)), "r"(GEMM_BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tmem_slot);
    const int KT = g.k_tiles;

    if (warp == 0 && lane == 0) {
        // producer: stage s is refilled once the products that read it are done
        int issued = 0;
        for (int kt = 0; kt < KT; ++kt) {
            const int s = kt % GEMM_STAGES;
            const uint32_t ph = (uint32_t)(kt / GEMM_STAGES) & 1u;
            if (!wait_phase(empty_bar(s), ph ^ 1u, abort_flag)) break;
            mbar_arrive_tx(full_bar(s), 2 * GEMM_TILE_BYTES);
            tma_load_2d(sa_s + s * GEMM_TILE_BYTES, &ta, g.a_k0 + kt * GEMM_BK, m0, full_bar(s));
            tma_load_2d(sb_s + s * GEMM_TILE_BYTES, &tb, g.b_k0 + kt * GEMM_BK, n0, full_bar(s));
            ++issued;
        }
        // every copy this thread issued has landed before the CTA may exit
        for (int kt = (issued > GEMM_STAGES ? issued - GEMM_STAGES : 0); kt < issued; ++kt) {
            const int s = kt % GEMM_STAGES;
            mbar_wait(full_bar(s), (uint32_t)(kt / GEMM_STAGES) & 1u);
        }
    } else if (warp == 1 && lane == 0) {
        // products: four K = 8 steps per 128-byte stage, the descriptor's start
        // address advanced by 32 bytes per step inside the swizzle atom
        for (int kt = 0; kt < KT; ++kt) {
            const int s = kt % GEMM_STAGES;
            const uint32_t ph = (uint32_t)(kt / GEMM_STAGES) & 1u;
            if (!wait_phase(full_bar(s), ph, abort_flag)) break;
            tc_fence_after();
            const uint32_t a0 = sa_s + s * GEMM_TILE_BYTES, b0 = sb_s + s * GEMM_TILE_BYTES;
#pragma unroll
            for (int kk = 0; kk < GEMM_BK / 8; ++kk)
                umma_tf32(tmem, sw128_desc(a0 + 32u * kk), sw128_desc(b0 + 32u * kk),
                          (kt > 0 || kk > 0) ? 1u : 0u);
            umma_commit(empty_bar(s));
        }
        // the accumulator barrier also tracks products issued before a give-up
        umma_commit(accum_bar);
    }
    __syncwarp();

    // epilogue: one accumulator row per thread, 32 columns per tensor-memory load
    const bool ok = __all_sync(0xFFFFFFFFu, wait_phase(accum_bar, 0u, abort_flag) && !*abort_flag);
    tc_fence_after();
    if (!ok) {
        if (lane == 0 && g.status) atomicCAS(g.status, 0, (int32_t)ISO_ERR_TIMEOUT);
        // tensor memory is freed only when no product writes to it any more
        // (the abort flag cuts the wait above short)
        mbar_wait(accum_bar, 0u);
        __syncwarp();
    } else {
        const int r = warp * 32 + lane;
        const long long row = (long long)m0 + r;
#pragma unroll 1
        for (int c = 0; c < GEMM_BN / 32; ++c) {
            float v[32];
            tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(c * 32), v);
            const int col0 = n0 + c * 32;
            float4* dst = reinterpret_cast<float4*>(g.C + row * g.ldc + col0);
#pragma unroll
            for (int j = 0; j < 8; ++j) dst[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(GEMM_BN) : "memory");
    }
}

// The epilogue of the split product, and its three products per stage.
template <int BN>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
k_gemm_x3(const __grid_constant__ CUtensorMap ta1, const __grid_constant__ CUtensorMap tb1,
          const __grid_constant__ CUtensorMap ta2, const __grid_constant__ CUtensorMap tb2, GemmArgs g) {
    pdl_enter();
    if (g.skip && *reinterpret_cast<const volatile int32_t*>(g.skip)) return;
    constexpr int STAGES = BN == 256 ? 2 : 3;
    constexpr int A_BYTES = GEMM_TILE_BYTES, B_BYTES = GEMM_TILE_BYTES * (BN / 128);
    constexpr int STAGE_BYTES = 2 * (A_BYTES + B_BYTES);                  // A hi, A lo, B hi, B lo
    constexpr uint32_t IDESC = (UMMA_IDESC & ~(0x3Fu << 17)) | ((uint32_t)(BN >> 3) << 17);
    static_assert(1024 + STAGES * STAGE_BYTES + 256 <= X3_SMEM, "shared memory");
    extern __shared__ unsigned char gemm_smem_raw[];
    unsigned char* const smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(gemm_smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* const bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    // bars[0, S): full, bars[S, 2S): empty, bars[2S]: accumulators ready
    uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 1);
    volatile int* const abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * GEMM_BM, n0 = blockIdx.x * BN;
    const CUtensorMap* const ta = blockIdx.z ? &ta2 : &ta1;
    const CUtensorMap* const tb = blockIdx.z ? &tb2 : &tb1;
    float* const C = blockIdx.z ? g.C2 : g.C;
    const uint32_t smem_s = smem_u32(smem), bar_s = smem_u32(bars);
    auto full_bar = [&](int s) { return bar_s + 8u * s; };
    auto empty_bar = [&](int s) { return bar_s + 8u * (STAGES + s); };
    const uint32_t accum_bar = bar_s + 8u * (2 * STAGES);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        mbar_init(accum_bar, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(tmem_slot)), "r"(2 * BN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *reinterpret_cast<volatile uint32_t*>(tmem_slot), 0);
    const int KT = g.k_tiles;

    if (warp == 0 && lane == 0) {
        int issued = 0;
        for (int kt = 0; kt < KT; ++kt) {
            const int s = kt % STAGES;
            if (!wait_phase(empty_bar(s), ((uint32_t)(kt / STAGES) & 1u) ^ 1u, abort_flag)) break;
            // rows past the operand's end are filled with zeros and count as copied
            mbar_arrive_tx(full_bar(s), STAGE_BYTES);
            const uint32_t a0 = smem_s + (uint32_t)(s * STAGE_BYTES), b0 = a0 + 2 * A_BYTES;
            const int x = kt * GEMM_BK;
            tma_load_2d(a0, ta, x, m0, full_bar(s));
            tma_load_2d(a0 + A_BYTES, ta, g.seg + x, m0, full_bar(s));
#pragma unroll
            for (int h = 0; h < BN / 128; ++h) {
                tma_load_2d(b0 + h * GEMM_TILE_BYTES, tb, x, n0 + 128 * h, full_bar(s));
                tma_load_2d(b0 + B_BYTES + h * GEMM_TILE_BYTES, tb, g.seg + x, n0 + 128 * h, full_bar(s));
            }
            ++issued;
        }
        // every copy this thread issued has landed before the CTA may exit
        for (int kt = (issued > STAGES ? issued - STAGES : 0); kt < issued; ++kt)
            mbar_wait(full_bar(kt % STAGES), (uint32_t)(kt / STAGES) & 1u);
    } else if (warp == 1) {
        const bool lead = elect_one();
        const uint32_t hi = (uint32_t)(sw128_desc(smem_s) >> 32), lo0 = (uint32_t)sw128_desc(smem_s);
        for (int kt = 0; kt < KT; ++kt) {
            const int s = kt % STAGES;
            if (!wait_phase_warp(full_bar(s), (uint32_t)(kt / STAGES) & 1u, abort_flag)) break;
            tc_fence_after();
            const uint32_t a0 = lo0 + (uint32_t)(s * (STAGE_BYTES >> 4)), b0 = a0 + (2 * A_BYTES >> 4);
#pragma unroll
            for (int kk = 0; kk < GEMM_BK / 8; ++kk) {
                const uint32_t ah = a0 + 2 * kk, al = ah + (A_BYTES >> 4), bh = b0 + 2 * kk, bl = bh + (B_BYTES >> 4);
                const uint32_t acc = (kt > 0 || kk > 0) ? 1u : 0u;
                if (lead) {
                    umma_lo<0>(tmem, ah, bh, hi, IDESC, acc);
                    umma_lo<0>(tmem + BN, ah, bl, hi, IDESC, acc);
                    umma_lo<0>(tmem + BN, al, bh, hi, IDESC, 1u);
                }
            }
            if (lead) umma_commit(empty_bar(s));
        }
        // the accumulator barrier also tracks products issued before a give-up
        if (lead) umma_commit(accum_bar);
    }
    __syncwarp();

    const bool ok = __all_sync(0xFFFFFFFFu, wait_phase(accum_bar, 0u, abort_flag) && !*abort_flag);
    tc_fence_after();
    if (!ok) {
        if (lane == 0 && g.status) atomicCAS(g.status, 0, (int32_t)ISO_ERR_TIMEOUT);
        // tensor memory is freed only when no product writes to it any more
        // (the abort flag cuts the wait above short)
        mbar_wait(accum_bar, 0u);
        __syncwarp();
    } else {
        const long long row = (long long)m0 + warp * 32 + lane;
        const uint32_t tq = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
            if (n0 + c >= g.c_cols) break;
            float v[32], w[32];
            tmem_ld32(tq + (uint32_t)c, v);
            tmem_ld32(tq + (uint32_t)(BN + c), w);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = __fadd_rn(v[j], w[j]);
            gemm_store32(g, C, row, n0 + c, v);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(2 * BN) : "memory");
    }
}
template __global__ void k_gemm_x3<128>(const __grid_constant__ CUtensorMap, const __grid_constant__ CUtensorMap,
                                        const __grid_constant__ CUtensorMap, const __grid_constant__ CUtensorMap, GemmArgs);
template __global__ void k_gemm_x3<256>(const __grid_constant__ CUtensorMap, const __grid_constant__ CUtensorMap,
                                        const __grid_constant__ CUtensorMap, const __grid_constant__ CUtensorMap, GemmArgs);

// ---------------------------------------------------------------------------
// exact-slice contraction (see iso_gemm.cuh)
// ---------------------------------------------------------------------------
namespace {

// shared-memory descriptor of one slice: K-major, no swizzle; the two 8-row
// halves of the contraction 128 bytes apart, 8-column groups 256 bytes apart
__device__ __forceinline__ uint64_t plain_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)(128u >> 4) << 16;        // leading byte offset: along the contraction
    d |= (uint64_t)(256u >> 4) << 32;        // stride byte offset: along M / N
    d |= (uint64_t)1u << 46;                 // descriptor version of sm_100; layout 0: no swizzle
    return d;
}
constexpr uint32_t OZ_IDESC = (1u << 4)                 // D format: f32
                            | (1u << 7)                 // A format: bf16
                            | (1u << 10)                // B format: bf16
                            | ((uint32_t)(OZ_BM >> 3) << 17)
                            | ((uint32_t)(OZ_BM >> 4) << 24);

// tot += W * (the group's integer sums): this thread's lane, 64 columns
template <int W>
__device__ __forceinline__ void oz_drain(uint32_t taddr, long long (&tot)[64]) {
#pragma unroll
    for (int c = 0; c < 64; c += 8) {
        float v[8];
        tmem_ld8(taddr + c, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) tot[c + j] += (long long)__float2int_rn(v[j]) * (long long)W;
    }
}

}  // namespace

// One CTA per 128 x 128 tile (and contraction split, and expert): warp 0
// copies slabs, warp 1 issues the products, warps 2 .. 9 drain tensor memory.
// Bound by the tensor cores: 28 products of 128 x 128 x 16 per 16 rows, each
// slab read once per sweep for 18 (10) products.
__global__ void __launch_bounds__(OZ_THREADS, 1) k_oz_gemm(OzArgs g) {
    pdl_enter();
    extern __shared__ unsigned char gemm_smem_raw[];
    unsigned char* const smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(gemm_smem_raw) + 127) & ~(uintptr_t)127);
    uint64_t* const bars = reinterpret_cast<uint64_t*>(smem + OZ_STAGES * 2 * OZ_SLAB_BYTES);
    // bars: full[S], empty[S], then per accumulator: ready[4], drained[4]
    uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * OZ_STAGES + 8);
    volatile int* const abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = __shfl_sync(0xFFFFFFFFu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t smem_s = smem_u32(smem), bar_s = smem_u32(bars);
    auto full_bar = [&](int s) { return bar_s + 8u * s; };
    auto empty_bar = [&](int s) { return bar_s + 8u * (OZ_STAGES + s); };
    auto ready_bar = [&](int a) { return bar_s + 8u * (2 * OZ_STAGES + a); };
    auto drained_bar = [&](int a) { return bar_s + 8u * (2 * OZ_STAGES + 4 + a); };

    int ti, tj;
    if (g.symmetric) {
        int rest = blockIdx.x;
        ti = 0;
        while (rest >= g.tiles - ti) { rest -= g.tiles - ti; ++ti; }   // at most `tiles` steps
        tj = ti + rest;
    } else {
        ti = blockIdx.x / g.tiles;
        tj = blockIdx.x % g.tiles;
    }
    const int split = blockIdx.y, z = blockIdx.z;
    const int c0 = split * g.per_split;
    const int nc = min(g.per_split, g.chunks - c0);     // >= 1 (host)
    const unsigned char* const ga = g.A + ((unsigned long long)ti * g.chunks + c0) * OZ_SLAB_BYTES;
    const unsigned char* const gb = g.B + z * g.b_stride + ((unsigned long long)tj * g.chunks + c0) * OZ_SLAB_BYTES;

    if (threadIdx.x == 0) {
        for (int s = 0; s < OZ_STAGES; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int a = 0; a < 4; ++a) {
            mbar_init(ready_bar(a), 1);
            mbar_init(drained_bar(a), OZ_EPI_WARPS);
        }
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, *reinterpret_cast<volatile uint32_t*>(tmem_slot), 0);

    if (warp == 0 && lane == 0) {
        int it = 0;
        for (; it < 2 * nc; ++it) {
            const int s = it % OZ_STAGES;
            if (!wait_phase(empty_bar(s), ((uint32_t)(it / OZ_STAGES) & 1u) ^ 1u, abort_flag)) break;
            const bool high = it < nc;
            const uint32_t bytes = high ? (uint32_t)(OZ_HIGH * OZ_SLICE_BYTES) : (uint32_t)OZ_SLAB_BYTES;
            const unsigned long long off = (unsigned long long)(high ? it : it - nc) * OZ_SLAB_BYTES;
            const uint32_t dst = smem_s + (uint32_t)s * 2u * OZ_SLAB_BYTES;
            mbar_arrive_tx(full_bar(s), 2 * bytes);
            bulk_g2s(dst, ga + off, bytes, full_bar(s));
            bulk_g2s(dst + OZ_SLAB_BYTES, gb + off, bytes, full_bar(s));
        }
        // every copy this thread issued has landed before the CTA may exit
#pragma unroll 1
        for (int k = (it > OZ_STAGES ? it - OZ_STAGES : 0); k < it; ++k)
            mbar_wait(full_bar(k % OZ_STAGES), (uint32_t)(k / OZ_STAGES) & 1u);
    } else if (warp == 1) {
        const bool lead = elect_one();
        const uint32_t hi = (uint32_t)(plain_desc(smem_s) >> 32), lo0 = (uint32_t)plain_desc(smem_s);
        // Every group of a drain interval takes the next of the four
        // accumulators in turn (use u: accumulator u % 4), so in the low sweep,
        // with three groups, one is drained ahead of the products that need it
        bool ok = true;
        int it = 0, use = 0;
        // one sweep: groups G0 .. G0 + NG - 1, a drain every STEPS steps
        auto sweep = [&](auto g0_c, auto ng_c, auto steps_c) {
            constexpr int G0 = decltype(g0_c)::value, NG = decltype(ng_c)::value, STEPS = decltype(steps_c)::value;
            for (int c = 0; c < nc && ok; ++c, ++it) {
                const int s = it % OZ_STAGES;
                if (!wait_phase_warp(full_bar(s), (uint32_t)(it / OZ_STAGES) & 1u, abort_flag)) { ok = false; break; }
                tc_fence_after();
                const bool first = c % STEPS == 0, last = c % STEPS == STEPS - 1 || c == nc - 1;
                const uint32_t a0 = lo0 + (uint32_t)s * (2u * OZ_SLAB_BYTES >> 4), b0 = a0 + (OZ_SLAB_BYTES >> 4);
#pragma unroll
                for (int a = 0; a < NG; ++a) {
                    if (!ok) continue;
                    const int u = use + a;
                    const uint32_t acc = (uint32_t)u & 3u;
                    if (first && u >= 4) {
                        if (!wait_phase_warp(drained_bar(acc), (uint32_t)((u >> 2) - 1) & 1u, abort_flag)) { ok = false; continue; }
                        tc_fence_after();
                    }
                    const int grp = G0 + a;
#pragma unroll
                    for (int t = 0; t <= grp; ++t)
                        if (lead)
                            umma_lo<1>(tmem + acc * OZ_BM, a0 + (uint32_t)t * (OZ_SLICE_BYTES >> 4),
                                       b0 + (uint32_t)(grp - t) * (OZ_SLICE_BYTES >> 4), hi, OZ_IDESC,
                                       (first && t == 0) ? 0u : 1u);
                    if (last && lead) umma_commit(ready_bar(acc));
                }
                if (last) use += NG;
                if (lead) umma_commit(empty_bar(s));
            }
        };
        sweep(std::integral_constant<int, 0>{}, std::integral_constant<int, OZ_HIGH>{}, std::integral_constant<int, OZ_STEPS_HIGH>{});
        if (ok) sweep(std::integral_constant<int, OZ_HIGH>{}, std::integral_constant<int, OZ_SLICES - OZ_HIGH>{},
                      std::integral_constant<int, OZ_STEPS_LOW>{});
        // the products use shared and tensor memory until they complete, also
        // where this warp or a drain gave up: wait for them (the last commit of
        // every stage that was read)
#pragma unroll 1
        for (int k = (it > OZ_STAGES ? it - OZ_STAGES : 0); k < it; ++k)
            mbar_wait(empty_bar(k % OZ_STAGES), (uint32_t)(k / OZ_STAGES) & 1u);
        __syncwarp();
    } else if (warp >= 2) {
        // lane of tensor memory: 32 (warp % 4) + lane; columns 64 h .. + 63
        const int quad = warp & 3, h = (warp - 2) >> 2;
        const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(64 * h);
        const long long row = (long long)ti * OZ_BM + quad * 32 + lane;
        const long long colb = (long long)tj * OZ_BM + 64 * h;
        const long long q = g.q;
        double* const dst = g.part ? g.part + ((long long)split * gridDim.z + z) * q * q : g.C + z * g.c_stride;
        bool ok = true;
        int use = 0;
        auto take = [&](auto w, long long (&tot)[64]) -> bool {
            const int acc = use & 3;
            if (!wait_phase_warp(ready_bar(acc), (uint32_t)(use >> 2) & 1u, abort_flag)) return false;
            tc_fence_after();
            oz_drain<decltype(w)::value>(tq + (uint32_t)acc * OZ_BM, tot);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(drained_bar(acc));
            ++use;
            return true;
        };
        long long tot[64];
#pragma unroll
        for (int j = 0; j < 64; ++j) tot[j] = 0;
        for (int c = 0; c < nc && ok; c += OZ_STEPS_HIGH) {
            ok = take(std::integral_constant<int, 1 << 24>{}, tot) && take(std::integral_constant<int, 1 << 16>{}, tot) &&
                 take(std::integral_constant<int, 1 << 8>{}, tot) && take(std::integral_constant<int, 1>{}, tot);
        }
        // the high groups' total waits in the output array (rounded once to
        // binary64) while the low ones run
#pragma unroll
        for (int j = 0; j < 64; ++j) {
            if (ok && row < q && colb + j < q) dst[row * q + colb + j] = (double)tot[j];
            tot[j] = 0;
        }
        for (int c = 0; c < nc && ok; c += OZ_STEPS_LOW) {
            ok = take(std::integral_constant<int, 1 << 16>{}, tot) && take(std::integral_constant<int, 1 << 8>{}, tot) &&
                 take(std::integral_constant<int, 1>{}, tot);
        }
        if (!ok) {
            if (lane == 0 && g.status) atomicCAS(g.status, 0, (int32_t)ISO_ERR_TIMEOUT);
        } else if (row < q) {
            const int er = g.ea[row];
            const int32_t* eb = g.eb + z * g.eb_stride;
#pragma unroll
            for (int j = 0; j < 64; ++j) {
                const long long col = colb + j;
                if (j % 4 == 0) asm volatile("" ::: "memory");   // keeps the loads of later columns behind (registers)
                if (col >= q) continue;
                const int ec = eb[col];
                double v = fma(dst[row * q + col], 16777216.0, (double)tot[j]);
                v = (er >= OZ_NONFINITE || ec >= OZ_NONFINITE) ? __longlong_as_double(0x7FF8000000000000LL)
                                                                : scalbn(v, er + ec - 62);
                if (g.minus_identity && row == col) v -= 1.0;
                dst[row * q + col] = v;
                if (g.symmetric && ti != tj) dst[col * q + row] = v;
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(512) : "memory");
    }
}

namespace {
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled encode_fn() {
    static std::once_flag once;
    static EncodeTiled fn = nullptr;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    });
    return fn;
}
}  // namespace

int gemm_tensor_map(CUtensorMap* map, const float* base, long long rows, long long cols, long long ld) {
    EncodeTiled fn = encode_fn();
    if (!fn) return ISO_ERR_CUDA;
    if ((reinterpret_cast<uintptr_t>(base) & 15u) || (ld % 4) || (cols % GEMM_BK) || (rows % GEMM_BM))
        return ISO_ERR_ALIGN;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
    const cuuint32_t box[2] = {(cuuint32_t)GEMM_BK, (cuuint32_t)GEMM_BM};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? ISO_OK : ISO_ERR_CUDA;
}

}  // namespace iso
