// iso_merge.cu -- the merge pass of K experts (with bfloat16 experts; the
// binary32 ones are instantiated by iso_merge_f32.cu, which includes this file).
//
//   k_merge   out = theta_0 + update from the K masked task vectors   (App. F)
//               TA    update = lambda * sum_i tau_i
//               TIES  gamma = sign(sum_i m_i tau_i); A = {i : m_i tau_i != 0,
//                     sign(tau_i) = gamma}; update = lambda * mean_{i in A} tau_i
//               ISO   2-D: update = sum_i c_i m_i tau_i           (Sec. 4.2, App. E)
//                     1-D: update = (1/K) sum_i tau_i             (App. E, Algorithm 1)
//               RAM   update = lambda * the mean of the active tau_i (App. F, RAM)
//             An update of exactly zero leaves theta_0 untouched.
//
// The expert count is a compile-time bound KC (1 for RAM's K = 1, then 2, 3,
// 4 or 8; the call's K equals KC up to 4 and is at most 8 beyond), so every
// per-expert array is a register array and all loops over experts unroll.
//
// Arithmetic: binary32, experts taken in the fixed order i = 1..K; the merge
// uses explicit round-to-nearest operations (no contraction) so that every
// output is the one the sequential definition gives.
#include "iso_merge.cuh"

#include <type_traits>

namespace iso {

// a / cnt for cnt = 0 .. KC (0 counts as 1), rounded as the IEEE division: by
// 1, 2, 4 and 8 the product with the reciprocal is exact; by 3, 5, 6 and 7 the
// quotient estimate q = a r is corrected once with its exact remainder
// (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990; equal to the division for every binary32 mantissa).  An
// overflowed sum and quotients near the subnormals take the division itself.
// tab[cnt] = (cnt, 1 / cnt).
template <int KC>
__device__ __forceinline__ float div_count(float a, int cnt, const float2* tab) {
    if (KC <= 2) return cnt == 2 ? __fmul_rn(a, 0.5f) : a;
    const float2 t = tab[cnt];
    const float q = __fmul_rn(a, t.y);
    const uint32_t k = __float_as_uint(q) & 0x7FFFFFFFu, low = 0x03800000u;   // 2^-120
    if (k - low >= KEY_INF - low && k) return __fdiv_rn(a, t.x);
    return __fmaf_rn(__fmaf_rn(-t.x, q, a), t.y, q);
}

// outputs of two neighbouring entries in a tile with per-tile bounds; the
// same operations in the same order as merged_fast, an unselected term left
// out instead of added as +0 (the sums start at +0 and never become -0).
// ALL: an untrimmed TIES tensor, every expert's value taken as it is (no pass
// has looked at it, so a NaN, which no bound admits, is to reach the sum).
template <int OPK, bool ALL, int KC>
__device__ __forceinline__ void merge_pair(const float (&t0)[KC], const float (&t1)[KC], float a0, float a1,
                                           const float (&cf)[KC], const float (&bound)[KC], float lambda, int K,
                                           bool iso1d, const float2* tab, float& bad0, float& bad1, float& o0,
                                           float& o1) {
    float u0, u1;
    if (OPK == OPK_TIES) {
        float x0[KC], x1[KC], s0 = 0.0f, s1 = 0.0f;
#pragma unroll
        for (int q = 0; q < KC; ++q) {
            x0[q] = (ALL ? q < K : fabsf(t0[q]) > bound[q]) ? t0[q] : 0.0f;
            x1[q] = (ALL ? q < K : fabsf(t1[q]) > bound[q]) ? t1[q] : 0.0f;
            add_rn2(s0, s1, s0, s1, x0[q], x1[q]);
        }
        const uint32_t b0 = __float_as_uint(s0) & 0x80000000u, b1 = __float_as_uint(s1) & 0x80000000u;
        float m0 = 0.0f, m1 = 0.0f;
        int c0 = 0, c1 = 0;
#pragma unroll
        for (int q = 0; q < KC; ++q) {
            const float y0 = __uint_as_float(__float_as_uint(x0[q]) ^ b0), y1 = __uint_as_float(__float_as_uint(x1[q]) ^ b1);
            if (y0 > 0.0f) { m0 = __fadd_rn(m0, y0); ++c0; }
            if (y1 > 0.0f) { m1 = __fadd_rn(m1, y1); ++c1; }
        }
        m0 = s0 == 0.0f ? 0.0f : m0;                       // an empty agreeing set
        m1 = s1 == 0.0f ? 0.0f : m1;
        m0 = __uint_as_float(__float_as_uint(div_count<KC>(m0, c0, tab)) ^ b0);
        m1 = __uint_as_float(__float_as_uint(div_count<KC>(m1, c1, tab)) ^ b1);
        mul_rn2(u0, u1, lambda, lambda, m0, m1);
    } else if (OPK == OPK_RAM) {
        float s0 = 0.0f, s1 = 0.0f;
        int c0 = 0, c1 = 0;
#pragma unroll
        for (int q = 0; q < KC; ++q) {
            // 0 * tau is NaN for a non-finite tau and 0 otherwise
            bad0 = __fmaf_rn(t0[q], 0.0f, bad0);
            bad1 = __fmaf_rn(t1[q], 0.0f, bad1);
            if (fabsf(t0[q]) > bound[q]) { s0 = __fadd_rn(s0, t0[q]); ++c0; }
            if (fabsf(t1[q]) > bound[q]) { s1 = __fadd_rn(s1, t1[q]); ++c1; }
        }
        mul_rn2(u0, u1, lambda, lambda, div_count<KC>(s0, c0, tab), div_count<KC>(s1, c1, tab));
    } else if (OPK == OPK_ISO) {
        float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
        for (int q = 0; q < KC; ++q) {
            float p0, p1;
            mul_rn2(p0, p1, cf[q], cf[q], t0[q], t1[q]);
            if (fabsf(t0[q]) > bound[q]) s0 = __fadd_rn(s0, p0);
            if (fabsf(t1[q]) > bound[q]) s1 = __fadd_rn(s1, p1);
        }
        u0 = s0;
        u1 = s1;
    } else {
        float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
        for (int q = 0; q < KC; ++q)
            if (KC < 8 || q < K) add_rn2(s0, s1, s0, s1, t0[q], t1[q]);
        if (iso1d) {
            u0 = __fdiv_rn(s0, (float)K);
            u1 = __fdiv_rn(s1, (float)K);
        } else {
            mul_rn2(u0, u1, lambda, lambda, s0, s1);
        }
    }
    o0 = (u0 == 0.0f) ? a0 : __fadd_rn(a0, u0);
    o1 = (u1 == 0.0f) ? a1 : __fadd_rn(a1, u1);
}

// One warp per tile, a contiguous tile range per warp, the experts and the
// base streamed through the chunk ring.  The operator and the tile's form
// (per-tile bounds, or the exact per-entry test) are decided per chunk, never
// per entry: with uniform branches per entry, per-lane copies and the library
// division the pass was bound by issue (123 instructions per entry for RAM,
// K = 3; 76 for ISO), now by HBM.  1.54G entries, bf16 checkpoints: RAM K = 3
// 8.54 -> 2.91 ms (5.3 TB/s of 10 B per entry), ISO K = 3 4.71 -> 2.51 ms (6.1
// TB/s), TIES K = 2 5.00 -> 2.35 ms; 0.70G entries, eight binary32 task vectors,
// TIES: 5.03 -> 4.66 ms (5.4 TB/s).
template <typename XT, typename BT, bool CK, int KC, int OPF>
__global__ void __launch_bounds__(TPB, 2) k_merge(Plan P) {
    pdl_enter();
    using G = ChunkGeom<XT, BT, KC, true>;
    constexpr int E = G::E;
    extern __shared__ __align__(128) unsigned char s_ring[];
    const int K = KC < 8 ? KC : P.K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ float2 s_tab[KC + 1];
    __shared__ MergeParams<KC> s_mp[WPB];
    if (threadIdx.x <= KC) {
        const int c = threadIdx.x ? threadIdx.x : 1;
        s_tab[threadIdx.x] = make_float2((float)c, 1.0f / (float)c);
    }
    __syncthreads();
    const WarpRange wr = warp_range(P);
    if (wr.beg >= wr.end) return;
    MergeParams<KC>& mp = s_mp[warp];
    int t = -1;
    long long t_end = 0;
    float cf[KC], bound[KC];
    float bad0 = 0.0f, bad1 = 0.0f;     // RAM: turns NaN on a non-finite task vector
    bool exact = false;
    stream_chunks<G, XT, BT, KC, true>(P, K, wr, s_ring, [&](long long g, int c, const unsigned char* stage) {
        if (g >= t_end) {
            if (t < 0) t = tensor_of_tile(P.tens, P.n_tensors, g);
            while (g >= tensor_tile_end(P, t)) ++t;
            t_end = tensor_tile_end(P, t);
            merge_params<KC>(P, t, K, mp);
        }
        const TensorDesc& d = P.tens[t];
        const long long n = d.numel, e0 = (g - d.tile_base) * TILE;
        if (c == 0) {
            int T[KC];
            const long long e1 = (e0 + TILE < n) ? e0 + TILE : n;
            exact = tile_thresholds<KC>(mp, K, (uint32_t)e0, (uint32_t)e1, T);
#pragma unroll
            for (int q = 0; q < KC; ++q) {
                bound[q] = bound_of(T[q]);
                cf[q] = OPF == OPF_ISO ? mp.cf[q] : 0.0f;
            }
        }
        const long long ec = e0 + c * G::CE;
        const bool whole = ec + G::CE <= n;
        const int opk = mp.opk;
        auto steps = [&](auto&& pairs) {
#pragma unroll 1
            for (int s = 0; s < G::SPC; ++s) {
                const long long e = ec + s * G::STEP + lane * E;
                Words<XT, E> x[KC];
                Words<BT, E> b;
                chunk_words<G, XT, BT, KC, true>(stage, whole, s, K, mp.xs, d.base, e, n, lane, x, b);
                if (e >= n) continue;
                float o[E];
                pairs(e, x, b, o);
                store_out<BT, E>(d.out, e, n, o);
            }
        };
        auto fast = [&](auto opk_c, auto all_c) {
            steps([&](long long, const Words<XT, E> (&x)[KC], const Words<BT, E>& b, float (&o)[E]) {
#pragma unroll
                for (int j = 0; j < E; j += 2) {
                    const float a0 = word_f32<BT, E>(b, j), a1 = word_f32<BT, E>(b, j + 1);
                    float t0[KC], t1[KC];
#pragma unroll
                    for (int q = 0; q < KC; ++q) {
                        t0[q] = word_f32<XT, E>(x[q], j);
                        t1[q] = word_f32<XT, E>(x[q], j + 1);
                        if (CK) sub_rn2(t0[q], t1[q], t0[q], t1[q], a0, a1);
                    }
                    merge_pair<decltype(opk_c)::value, decltype(all_c)::value, KC>(
                        t0, t1, a0, a1, cf, bound, P.lambda, K, mp.iso1d, s_tab, bad0, bad1, o[j], o[j + 1]);
                }
            });
        };
        if ((OPF == OPF_TIES || OPF == OPF_ISO) && exact) {
            steps([&](long long e, const Words<XT, E> (&x)[KC], const Words<BT, E>& b, float (&o)[E]) {
                long long r = 0, cc = 0;
                if (mp.sel == SEL_BLOCK) { r = e / d.cols; cc = e - r * d.cols; }
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    const float th0 = word_f32<BT, E>(b, j);
                    float tau[KC];
#pragma unroll
                    for (int q = 0; q < KC; ++q) {
                        tau[q] = (q < K) ? word_f32<XT, E>(x[q], j) : 0.0f;
                        if (CK) tau[q] = __fsub_rn(tau[q], th0);
                    }
                    const uint32_t bits = select_bits<KC>(P, d, mp, K, tau, e + j, r, cc);
                    o[j] = merged_value<KC>(opk, P.lambda, K, th0, tau, cf, bits);
                }
            });
        } else if (OPF == OPF_TIES) {
            if (mp.sel == SEL_ALL) fast(std::integral_constant<int, OPK_TIES>{}, std::true_type{});
            else fast(std::integral_constant<int, OPK_TIES>{}, std::false_type{});
        } else if (OPF == OPF_RAM) {
            fast(std::integral_constant<int, OPK_RAM>{}, std::false_type{});
        } else if (OPF == OPF_SUM || opk == OPK_SUM) {
            fast(std::integral_constant<int, OPK_SUM>{}, std::false_type{});
        } else {
            fast(std::integral_constant<int, OPK_ISO>{}, std::false_type{});
        }
    });
    // RAM reads every entry's magnitude: a NaN or infinity is reported
    if (OPF == OPF_RAM) {
        const float bad = bad0 + bad1;
        if (__any_sync(0xFFFFFFFFu, bad != bad) && lane == 0) set_status(P.hdr, ISO_ERR_NONFINITE);
    }
}

template <typename XT, typename BT, int KC>
int merge_smem_bytes() { return ChunkGeom<XT, BT, KC, true>::SMEM; }

#define ISO_MERGE_INST(XT, BT, CK)                                             \
    template __global__ void k_merge<XT, BT, CK, 1, OPF_RAM>(Plan);           \
    ISO_MERGE_KC(XT, BT, CK, 2)                                                \
    ISO_MERGE_KC(XT, BT, CK, 3)                                                \
    ISO_MERGE_KC(XT, BT, CK, 4)                                                \
    ISO_MERGE_KC(XT, BT, CK, 8)
#define ISO_MERGE_KC(XT, BT, CK, KC)                                           \
    template __global__ void k_merge<XT, BT, CK, KC, OPF_TIES>(Plan);         \
    template __global__ void k_merge<XT, BT, CK, KC, OPF_ISO>(Plan);          \
    template __global__ void k_merge<XT, BT, CK, KC, OPF_RAM>(Plan);          \
    template __global__ void k_merge<XT, BT, CK, KC, OPF_SUM>(Plan);
#define ISO_MERGE_SMEM(XT, BT)                                                 \
    template int merge_smem_bytes<XT, BT, 1>();                               \
    template int merge_smem_bytes<XT, BT, 2>();                               \
    template int merge_smem_bytes<XT, BT, 3>();                               \
    template int merge_smem_bytes<XT, BT, 4>();                               \
    template int merge_smem_bytes<XT, BT, 8>();

#ifndef ISO_MERGE_XT
#define ISO_MERGE_XT __nv_bfloat16
#endif
ISO_MERGE_SMEM(ISO_MERGE_XT, __nv_bfloat16)
ISO_MERGE_SMEM(ISO_MERGE_XT, float)
ISO_MERGE_INST(ISO_MERGE_XT, __nv_bfloat16, false)
ISO_MERGE_INST(ISO_MERGE_XT, float, false)
ISO_MERGE_INST(ISO_MERGE_XT, __nv_bfloat16, true)
ISO_MERGE_INST(ISO_MERGE_XT, float, true)

}  // namespace iso
