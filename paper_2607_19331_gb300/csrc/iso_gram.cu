// iso_gram.cu -- the Gram pass of the ISO retention rule (Sec. 4.2), any K:
// Gamma_ab = <m_a tau_a, m_b tau_b> per trimmed 2-D tensor.
#include "iso_merge.cuh"

#include <type_traits>

namespace iso {

// Gram of the trimmed task vectors, upper triangle, per 2-D trimmed tensor.
// The experts stream through the chunk ring (the base too for checkpoints).
// Tile partials in binary32 (fused multiply-add over one lane's entries of the
// tile, then a warp sum), accumulated per warp as binary32 two-sum pairs and
// added to the tensor's Gamma with one atomic per pair when the warp leaves
// the tensor.  1.54G entries, three bf16 checkpoints: 3.90 -> 1.97 ms (6.3 TB/s),
// see k_merge for what changed.
template <typename XT, typename BT, bool CK, int KC>
__global__ void __launch_bounds__(TPB, 2) k_gramk(Plan P) {
    pdl_enter();
    using G = ChunkGeom<XT, BT, KC, CK>;
    constexpr int E = G::E;
    constexpr int NP = KC * (KC + 1) / 2;
    static_assert(NP <= 64, "two pair sums per lane");
    extern __shared__ __align__(128) unsigned char s_ring[];
    const int K = KC < 8 ? KC : P.K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ MergeParams<KC> s_mp[WPB];
    // lane L accumulates pairs L and 32 + L over the warp's tiles of one
    // tensor as binary32 two-sum pairs (no binary64 arithmetic per tile)
    float gs0 = 0.0f, ge0 = 0.0f, gs1 = 0.0f, ge1 = 0.0f;
    const WarpRange wr = warp_range(P);
    if (wr.beg >= wr.end) return;
    MergeParams<KC>& mp = s_mp[warp];
    int t = -1;
    long long t_end = 0;
    auto flush = [&](int tt) {
        int q = 0;
#pragma unroll
        for (int a = 0; a < KC; ++a) {
#pragma unroll
            for (int b = a; b < KC; ++b, ++q) {
                if (a < K && b < K && (lane == q || lane + 32 == q)) {
                    const double v = (lane == q) ? (double)gs0 + (double)ge0 : (double)gs1 + (double)ge1;
                    if (v != 0.0) atomicAdd(&P.gram[((long long)tt * K + a) * K + b], v);
                }
            }
        }
        gs0 = ge0 = gs1 = ge1 = 0.0f;
    };
    float bound[KC], acc[NP];
    bool exact = false;
    stream_chunks<G, XT, BT, KC, CK>(P, K, wr, s_ring, [&](long long g, int c, const unsigned char* stage) {
        if (g >= t_end) {
            if (t >= 0) flush(t);
            else t = tensor_of_tile(P.tens, P.n_tensors, g);
            while (g >= tensor_tile_end(P, t)) ++t;
            t_end = tensor_tile_end(P, t);
            merge_params<KC>(P, t, K, mp);
        }
        if (!mp.trimmed2d) return;
        const TensorDesc& d = P.tens[t];
        const long long n = d.numel, e0 = (g - d.tile_base) * TILE;
        if (c == 0) {
            int T[KC];
            const long long e1 = (e0 + TILE < n) ? e0 + TILE : n;
            exact = tile_thresholds<KC>(mp, K, (uint32_t)e0, (uint32_t)e1, T);
#pragma unroll
            for (int q = 0; q < KC; ++q) bound[q] = bound_of(T[q]);
#pragma unroll
            for (int q = 0; q < NP; ++q) acc[q] = 0.0f;
        }
        const long long ec = e0 + c * G::CE;
        const bool whole = ec + G::CE <= n;
        auto steps = [&](auto&& kept) {
#pragma unroll 1
            for (int s = 0; s < G::SPC; ++s) {
                const long long e = ec + s * G::STEP + lane * E;
                Words<XT, E> x[KC];
                Words<BT, E> b;
                chunk_words<G, XT, BT, KC, CK>(stage, whole, s, K, mp.xs, d.base, e, n, lane, x, b);
                if (e >= n) continue;
                long long r = 0, cc = 0;
                if (exact && mp.sel == SEL_BLOCK) { r = e / d.cols; cc = e - r * d.cols; }
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    const float th0 = CK ? word_f32<BT, E>(b, j) : 0.0f;
                    float m[KC];
#pragma unroll
                    for (int q = 0; q < KC; ++q) {
                        m[q] = word_f32<XT, E>(x[q], j);
                        if (CK) m[q] = __fsub_rn(m[q], th0);
                    }
                    kept(e + j, n, r, cc, m);
                    int q = 0;
#pragma unroll
                    for (int a2 = 0; a2 < KC; ++a2)
#pragma unroll
                        for (int b2 = a2; b2 < KC; ++b2, ++q) acc[q] = __fmaf_rn(m[a2], m[b2], acc[q]);
                }
            }
        };
        if (exact) {
            steps([&](long long e, long long nn, long long& r, long long& cc, float (&m)[KC]) {
                const uint32_t bits = e < nn ? select_bits<KC>(P, d, mp, K, m, e, r, cc) : 0u;
#pragma unroll
                for (int q = 0; q < KC; ++q) m[q] = ((bits >> q) & 1u) ? m[q] : 0.0f;
            });
        } else {
            // past the tensor's end the words read zero: never above a bound
            // >= 0, and a bound of -1 (everything kept) only leaves zeros
            steps([&](long long, long long, long long&, long long&, float (&m)[KC]) {
#pragma unroll
                for (int q = 0; q < KC; ++q) m[q] = fabsf(m[q]) > bound[q] ? m[q] : 0.0f;
            });
        }
        if (c == G::CPT - 1) {
            // the tile's partial sums: warp sums, then one two-sum per lane
            float w0 = 0.0f, w1 = 0.0f;
            int q = 0;
#pragma unroll
            for (int a2 = 0; a2 < KC; ++a2) {
#pragma unroll
                for (int b2 = a2; b2 < KC; ++b2, ++q) {
                    if (a2 < K && b2 < K) {
                        const float w = warp_sum(acc[q]);
                        if (q < 32) w0 = (lane == q) ? w : w0;
                        else w1 = (lane + 32 == q) ? w : w1;
                    }
                }
            }
            two_sum_add(gs0, ge0, w0);
            if (NP > 32) two_sum_add(gs1, ge1, w1);
        }
    });
    if (t >= 0) flush(t);
}

template <typename XT, typename BT, bool CK, int KC>
int gram_smem_bytes() { return ChunkGeom<XT, BT, KC, CK>::SMEM; }

#define ISO_GRAM_INST(XT, BT, CK)                                              \
    ISO_GRAM_KC(XT, BT, CK, 1)                                                 \
    ISO_GRAM_KC(XT, BT, CK, 2)                                                 \
    ISO_GRAM_KC(XT, BT, CK, 3)                                                 \
    ISO_GRAM_KC(XT, BT, CK, 4)                                                 \
    ISO_GRAM_KC(XT, BT, CK, 8)
#define ISO_GRAM_KC(XT, BT, CK, KC)                                            \
    template __global__ void k_gramk<XT, BT, CK, KC>(Plan);                   \
    template int gram_smem_bytes<XT, BT, CK, KC>();

ISO_GRAM_INST(__nv_bfloat16, __nv_bfloat16, false)
ISO_GRAM_INST(__nv_bfloat16, float, false)
ISO_GRAM_INST(float, __nv_bfloat16, false)
ISO_GRAM_INST(float, float, false)
ISO_GRAM_INST(__nv_bfloat16, __nv_bfloat16, true)
ISO_GRAM_INST(__nv_bfloat16, float, true)
ISO_GRAM_INST(float, __nv_bfloat16, true)
ISO_GRAM_INST(float, float, true)

}  // namespace iso
