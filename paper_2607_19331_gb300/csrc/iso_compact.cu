// iso_compact.cu -- the Gram and merge passes over compact candidates
// (Plan::ccv, off by default), with bfloat16 experts; iso_compact_f32.cu
// includes this file for the binary32 ones.
#include "iso_merge.cuh"

namespace iso {

// ---------------------------------------------------------------------------
// Compact candidates (Plan::ccv).  The count pass has written, per expert and
// tile, the binary32 task-vector values whose key is at least the low edge of
// the unit's band, in position order, and a 32-word mask of their positions.
// When the unit's threshold lies in its band (Unit::v_ok) those values hold
// every entry the selection can keep, so the Gram and merge passes read them
// (about the kept fraction of each expert's bytes) instead of the full task
// vectors; any other expert of the tensor (an untrimmed tensor, a unit whose
// band missed or whose value segment overflowed) is read in full.  An entry
// absent from the values has key < lo <= t: never kept, it enters every sum
// as +0 exactly as an unkept entry does in k_merge / k_gramk, so both give
// the same results.  One warp per tile, lane l taking entries 4 l .. 4 l + 3
// of each 128-entry step: the four bits of word 4 s + l / 8 at 4 (l % 8).
// ---------------------------------------------------------------------------
template <int KC>
struct CompactParams {
    uint32_t vok;                      // bit q: expert q reads its compact values
    unsigned long long voff[KC];       // the unit's value segment in the pool
};

template <int KC>
__device__ __forceinline__ void compact_params(const Plan& P, int t, int K, CompactParams<KC>& cp) {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        const TensorDesc& d = P.tens[t];
        uint32_t ok = 0;
#pragma unroll
        for (int q = 0; q < KC; ++q) {
            cp.voff[q] = 0;
            if (q < K && (d.flags & TF_TRIM)) {
                const Unit& U = P.units[(long long)q * P.n_units + d.unit];
                if (U.v_ok) { ok |= 1u << q; cp.voff[q] = U.v_off; }
            }
        }
        cp.vok = ok;
    }
    __syncwarp();
}

// the tile's mask words, their exclusive popcount prefix and the value
// pointer of each compact expert, in the warp's shared memory (registers
// stay free for the data); the tile's values of each expert (when they fit
// CC_STAGE slots) and the tile's theta_0 are copied into the warp's stage
// with cp.async before the tile is merged, so that the merge reads shared
// memory only: two round trips to memory per tile (mask words, then values)
// instead of one per step.
constexpr int CC_STAGE = 256;
template <int KC, typename BT>
struct CompactTile {
    uint32_t mw[KC][32], pre[KC][32];
    const float* vb[KC];
    uint32_t staged;                   // bit q: expert q's values are in sv[q]
    float sv[KC][CC_STAGE];
    __align__(16) char th0[TILE * sizeof(BT)];
};

__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(dst), "l"(src) : "memory");
}

template <int KC, typename BT>
__device__ __forceinline__ void compact_tile(const Plan& P, const CompactParams<KC>& cp, int K, long long g, int lane,
                                             const void* base, long long e0, long long n, bool want_base,
                                             CompactTile<KC, BT>& ct) {
    __syncwarp();
    uint32_t cnt[KC];
#pragma unroll
    for (int q = 0; q < KC; ++q) {
        cnt[q] = 0;
        if (q < K && ((cp.vok >> q) & 1u)) {
            const long long rec = (long long)q * P.n_tiles + g;
            const uint32_t w = P.vmask[rec * 32 + lane];
            ct.pre[q][lane] = warp_excl_scan((uint32_t)__popc(w), &cnt[q]);
            ct.mw[q][lane] = w;
            if (lane == 0) ct.vb[q] = P.vals + cp.voff[q] + P.tval[rec];
        }
    }
    __syncwarp();
    uint32_t staged = 0;
#pragma unroll
    for (int q = 0; q < KC; ++q) {
        if (q < K && ((cp.vok >> q) & 1u) && cnt[q] <= (uint32_t)CC_STAGE) {
            staged |= 1u << q;
            const float* src = ct.vb[q];
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&ct.sv[q][0]);
            for (uint32_t i = lane; i < cnt[q]; i += 32) cp_async4(dst + 4 * i, src + i);
        }
    }
    if (want_base) {
        // the tile's theta_0, 16 bytes per lane per copy, zero-filled past the tensor's end
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(ct.th0);
        const char* src = static_cast<const char*>(base) + e0 * (long long)sizeof(BT);
        const long long avail = (n - e0) * (long long)sizeof(BT);
#pragma unroll
        for (int k = 0; k < (int)(TILE * sizeof(BT)) / 512; ++k) {
            const long long off = (long long)k * 512 + lane * 16;
            cp_async16(dst + (uint32_t)off, src + (avail > off ? off : 0), clamp_bytes(avail - off, 16));
        }
    }
    cp_async_commit();
    cp_async_wait<0>();
    if (lane == 0) ct.staged = staged;
    __syncwarp();
}

template <typename BT>
__device__ __forceinline__ float staged_base(const char* th0, int p) {
    if (sizeof(BT) == 4) return reinterpret_cast<const float*>(th0)[p];
    return __uint_as_float((uint32_t)reinterpret_cast<const unsigned short*>(th0)[p] << 16);
}

// tau of entries e .. e + 3 (step s of the tile) for every expert: compact
// values, or the full task vector; entries past the tensor's end read 0
template <typename XT, typename BT, bool CK, int KC>
__device__ __forceinline__ void compact_step(const CompactParams<KC>& cp, const CompactTile<KC, BT>& ct,
                                             const void* const* xs, int K, long long e, long long n, int s, int lane,
                                             const float (&th0)[4], float (&tau)[KC][4]) {
    const int w = s * 4 + (lane >> 3), bo = (lane & 7) * 4;
#pragma unroll
    for (int q = 0; q < KC; ++q) {
#pragma unroll
        for (int j = 0; j < 4; ++j) tau[q][j] = 0.0f;
        if (q >= K) continue;
        if ((cp.vok >> q) & 1u) {
            const uint32_t word = ct.mw[q][w];
            const uint32_t at = ct.pre[q][w] + (uint32_t)__popc(word & ((1u << bo) - 1u));
            const uint32_t nib = (word >> bo) & 0xFu;
            const bool st = (ct.staged >> q) & 1u;
            const float* vb = (st ? &ct.sv[q][0] : ct.vb[q]) + at;
            uint32_t r = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if ((nib >> j) & 1u) { tau[q][j] = st ? vb[r] : __ldg(vb + r); ++r; }
            }
        } else {
            Words<XT, 4> x;
            load_words<XT, 4>(xs[q], e, n, x);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                tau[q][j] = word_f32<XT, 4>(x, j);
                if (CK) tau[q][j] = __fsub_rn(tau[q][j], th0[j]);
            }
        }
    }
}

template <typename XT, typename BT, bool CK, int KC, int OPF>
__global__ void __launch_bounds__(TPB, 2) k_merge_c(Plan P) {
    pdl_enter();
    constexpr int E = 4, SPT = TILE / (32 * E);
    const int K = P.K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const WarpRange wr = warp_range(P);
    if (wr.beg >= wr.end) return;
    __shared__ MergeParams<KC> s_mp[WPB];
    __shared__ CompactParams<KC> s_cp[WPB];
    extern __shared__ __align__(16) char s_cstage[];
    CompactTile<KC, BT>& ct = reinterpret_cast<CompactTile<KC, BT>*>(s_cstage)[warp];
    MergeParams<KC>& mp = s_mp[warp];
    CompactParams<KC>& cp = s_cp[warp];
    int t = tensor_of_tile(P.tens, P.n_tensors, wr.beg);
    long long t_end = tensor_tile_end(P, t);
    merge_params<KC>(P, t, K, mp);
    compact_params<KC>(P, t, K, cp);
    const long long nt = wr.count();
#pragma unroll 1
    for (long long jt = 0; jt < nt; ++jt) {
        const long long g = wr.tile(jt);
        if (g >= t_end) {
            while (g >= t_end) t_end = tensor_tile_end(P, ++t);
            merge_params<KC>(P, t, K, mp);
            compact_params<KC>(P, t, K, cp);
        }
        const TensorDesc& d = P.tens[t];
        const long long n = d.numel;
        const long long e0 = (g - d.tile_base) * TILE;
        const long long e1 = (e0 + TILE < n) ? e0 + TILE : n;
        int T[KC];
        float cf[KC];
        const bool exact = tile_thresholds<KC>(mp, K, (uint32_t)e0, (uint32_t)e1, T);
#pragma unroll
        for (int q = 0; q < KC; ++q) cf[q] = (OPF == OPF_TIES) ? 0.0f : mp.cf[q];
        const int opk = (OPF == OPF_TIES) ? (int)OPK_TIES : mp.opk;
        compact_tile<KC, BT>(P, cp, K, g, lane, d.base, e0, n, true, ct);
#pragma unroll 1
        for (int s = 0; s < SPT; ++s) {
            const long long e = e0 + (long long)s * (32 * E) + lane * E;
            float th0[E];
#pragma unroll
            for (int j = 0; j < E; ++j) th0[j] = staged_base<BT>(ct.th0, s * (32 * E) + lane * E + j);
            float tau[KC][E];
            compact_step<XT, BT, CK, KC>(cp, ct, mp.xs, K, e, n, s, lane, th0, tau);
            long long r = 0, c = 0;
            if (exact && mp.sel == SEL_BLOCK) { r = e / d.cols; c = e - r * d.cols; }
            float o[E];
#pragma unroll
            for (int j = 0; j < E; ++j) {
                float tj[KC];
#pragma unroll
                for (int q = 0; q < KC; ++q) tj[q] = tau[q][j];
                if (exact) {
                    const uint32_t bits = (e + j < n) ? select_bits<KC>(P, d, mp, K, tj, e + j, r, c) : 0u;
                    o[j] = merged_value<KC>(opk, P.lambda, K, th0[j], tj, cf, bits);
                } else {
                    o[j] = merged_fast<KC>(opk, P.lambda, K, th0[j], tj, cf, T);
                }
            }
            store_out<BT, E>(d.out, e, n, o);
        }
    }
}

// Gram of the trimmed task vectors from the compact candidates (see above);
// partial sums as in k_gramk: per lane over the tile's entries in order,
// warp sums per tile, binary32 two-sum pairs per tensor, one atomic per pair.
template <typename XT, typename BT, bool CK, int KC>
__global__ void __launch_bounds__(TPB, 2) k_gramk_c(Plan P) {
    pdl_enter();
    constexpr int E = 4, SPT = TILE / (32 * E);
    constexpr int NP = KC * (KC + 1) / 2;
    static_assert(NP <= 64, "two pair sums per lane");
    const int K = P.K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float gs0 = 0.0f, ge0 = 0.0f, gs1 = 0.0f, ge1 = 0.0f;
    const WarpRange wr = warp_range(P);
    if (wr.beg >= wr.end) return;
    __shared__ MergeParams<KC> s_mp[WPB];
    __shared__ CompactParams<KC> s_cp[WPB];
    extern __shared__ __align__(16) char s_cstage[];
    CompactTile<KC, BT>& ct = reinterpret_cast<CompactTile<KC, BT>*>(s_cstage)[warp];
    MergeParams<KC>& mp = s_mp[warp];
    CompactParams<KC>& cp = s_cp[warp];
    int t = tensor_of_tile(P.tens, P.n_tensors, wr.beg);
    long long t_end = tensor_tile_end(P, t);
    merge_params<KC>(P, t, K, mp);
    compact_params<KC>(P, t, K, cp);
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
    const long long nt = wr.count();
#pragma unroll 1
    for (long long jt = 0; jt < nt; ++jt) {
        const long long g = wr.tile(jt);
        if (g >= t_end) {
            flush(t);
            while (g >= t_end) t_end = tensor_tile_end(P, ++t);
            merge_params<KC>(P, t, K, mp);
            compact_params<KC>(P, t, K, cp);
        }
        if (!mp.trimmed2d) continue;
        const TensorDesc& d = P.tens[t];
        const long long n = d.numel;
        const long long e0 = (g - d.tile_base) * TILE;
        const long long e1 = (e0 + TILE < n) ? e0 + TILE : n;
        int T[KC];
        const bool exact = tile_thresholds<KC>(mp, K, (uint32_t)e0, (uint32_t)e1, T);
        const bool want_base = CK && cp.vok != ((1u << K) - 1u);
        compact_tile<KC, BT>(P, cp, K, g, lane, d.base, e0, n, want_base, ct);
        float acc[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) acc[q] = 0.0f;
#pragma unroll 1
        for (int s = 0; s < SPT; ++s) {
            const long long e = e0 + (long long)s * (32 * E) + lane * E;
            float th0[E] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (want_base) {
#pragma unroll
                for (int j = 0; j < E; ++j) th0[j] = staged_base<BT>(ct.th0, s * (32 * E) + lane * E + j);
            }
            float tau[KC][E];
            compact_step<XT, BT, CK, KC>(cp, ct, mp.xs, K, e, n, s, lane, th0, tau);
            long long r = 0, c = 0;
            if (exact && mp.sel == SEL_BLOCK) { r = e / d.cols; c = e - r * d.cols; }
#pragma unroll
            for (int j = 0; j < E; ++j) {
                float tj[KC], m[KC];
#pragma unroll
                for (int q = 0; q < KC; ++q) tj[q] = tau[q][j];
                if (exact) {
                    const uint32_t bits = (e + j < n) ? select_bits<KC>(P, d, mp, K, tj, e + j, r, c) : 0u;
#pragma unroll
                    for (int q = 0; q < KC; ++q) m[q] = ((bits >> q) & 1u) ? tj[q] : 0.0f;
                } else {
#pragma unroll
                    for (int q = 0; q < KC; ++q) m[q] = ((int)key_of(tj[q]) > T[q]) ? tj[q] : 0.0f;
                }
                int q = 0;
#pragma unroll
                for (int a2 = 0; a2 < KC; ++a2)
#pragma unroll
                    for (int b2 = a2; b2 < KC; ++b2, ++q) acc[q] = __fmaf_rn(m[a2], m[b2], acc[q]);
            }
        }
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
    flush(t);
}

template <typename BT, int KC>
int compact_smem_bytes() { return WPB * (int)sizeof(CompactTile<KC, BT>); }

#ifndef ISO_COMPACT_XT   // once over the two translation units
template int compact_smem_bytes<__nv_bfloat16, 2>();
template int compact_smem_bytes<__nv_bfloat16, 4>();
template int compact_smem_bytes<__nv_bfloat16, 8>();
template int compact_smem_bytes<float, 2>();
template int compact_smem_bytes<float, 4>();
template int compact_smem_bytes<float, 8>();
#endif

#define ISO_COMPACT_INST(XT, BT, CK)                                           \
    template __global__ void k_merge_c<XT, BT, CK, 2, OPF_TIES>(Plan);        \
    template __global__ void k_merge_c<XT, BT, CK, 4, OPF_TIES>(Plan);        \
    template __global__ void k_merge_c<XT, BT, CK, 8, OPF_TIES>(Plan);        \
    template __global__ void k_merge_c<XT, BT, CK, 2, OPF_ISO>(Plan);         \
    template __global__ void k_merge_c<XT, BT, CK, 4, OPF_ISO>(Plan);         \
    template __global__ void k_merge_c<XT, BT, CK, 8, OPF_ISO>(Plan);         \
    template __global__ void k_gramk_c<XT, BT, CK, 2>(Plan);                  \
    template __global__ void k_gramk_c<XT, BT, CK, 4>(Plan);                  \
    template __global__ void k_gramk_c<XT, BT, CK, 8>(Plan);

#ifndef ISO_COMPACT_XT
#define ISO_COMPACT_XT __nv_bfloat16
#endif
ISO_COMPACT_INST(ISO_COMPACT_XT, __nv_bfloat16, false)
ISO_COMPACT_INST(ISO_COMPACT_XT, float, false)
ISO_COMPACT_INST(ISO_COMPACT_XT, __nv_bfloat16, true)
ISO_COMPACT_INST(ISO_COMPACT_XT, float, true)

}  // namespace iso
