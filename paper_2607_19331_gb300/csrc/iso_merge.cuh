// iso_merge.cuh -- what the passes over the K experts of a merge share: entry
// access, the per-tensor parameters, the per-tile thresholds, the merged value
// of one entry, and the chunk ring that streams the experts and the base.
#pragma once

#include "iso_kernels.cuh"

namespace iso {

namespace {

// raw words of E consecutive entries of T (E * sizeof(T) is 8, 16 or 32 bytes)
template <typename T, int E>
struct Words {
    static constexpr int N = E * (int)sizeof(T) / 4;
    uint32_t w[N];
};

__device__ __forceinline__ uint2 ld_stream2(const void* p) {
    uint2 r;
    asm("ld.global.nc.L1::no_allocate.L2::256B.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "l"(p));
    return r;
}

// entries [e, e + E) of p (e a multiple of E); entries at or past n read as 0
template <typename T, int E>
__device__ __forceinline__ void load_words(const void* p, long long e, long long n, Words<T, E>& r) {
    constexpr int N = Words<T, E>::N;
    const char* a = static_cast<const char*>(p) + e * (long long)sizeof(T);
    if (e + E <= n) {
        if (N == 2) {
            const uint2 v = ld_stream2(a);
            r.w[0] = v.x; r.w[1] = v.y;
        } else {
#pragma unroll
            for (int q = 0; q < N / 4; ++q) {
                const uint4 v = ld_stream(a + 16 * q);
                r.w[4 * q] = v.x; r.w[4 * q + 1] = v.y; r.w[4 * q + 2] = v.z; r.w[4 * q + 3] = v.w;
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) r.w[q] = 0;
        if (sizeof(T) == 2) {
            const unsigned short* s = static_cast<const unsigned short*>(p);
#pragma unroll
            for (int j = 0; j < E; ++j)
                if (e + j < n) r.w[j >> 1] |= (uint32_t)s[e + j] << (16 * (j & 1));
        } else {
            const uint32_t* s = static_cast<const uint32_t*>(p);
#pragma unroll
            for (int j = 0; j < E; ++j)
                if (e + j < n) r.w[j] = s[e + j];
        }
    }
}

template <typename T, int E>
__device__ __forceinline__ float word_f32(const Words<T, E>& r, int j) {
    if (sizeof(T) == 2)
        return __uint_as_float((j & 1) ? (r.w[j >> 1] & 0xFFFF0000u) : (r.w[j >> 1] << 16));
    return __uint_as_float(r.w[j]);
}

// E outputs of type T at [e, e + E), rounded to nearest even for bf16
template <typename T, int E>
__device__ __forceinline__ void store_out(void* p, long long e, long long n, const float (&v)[E]) {
    constexpr int N = Words<T, E>::N;
    uint32_t w[N];
    if (sizeof(T) == 2) {
#pragma unroll
        for (int q = 0; q < N; ++q) {
            __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
            w[q] = *reinterpret_cast<uint32_t*>(&h);
        }
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) w[q] = __float_as_uint(v[q]);
    }
    char* a = static_cast<char*>(p) + e * (long long)sizeof(T);
    if (e + E <= n) {
        if (N == 2) {
            __stcs(reinterpret_cast<uint2*>(a), make_uint2(w[0], w[1]));
        } else {
#pragma unroll
            for (int q = 0; q < N / 4; ++q)
                __stcs(reinterpret_cast<uint4*>(a) + q, make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]));
        }
    } else if (sizeof(T) == 2) {
        unsigned short* s = reinterpret_cast<unsigned short*>(a);
#pragma unroll
        for (int j = 0; j < E; ++j)
            if (e + j < n) s[j] = (unsigned short)(w[j >> 1] >> (16 * (j & 1)));
    } else {
        uint32_t* s = reinterpret_cast<uint32_t*>(a);
#pragma unroll
        for (int j = 0; j < E; ++j)
            if (e + j < n) s[j] = w[j];
    }
}

// how the entries of one tensor are tested against their units' thresholds
enum SelMode : int {
    SEL_ALL = 0,      // no mask (TA, ISO 1-D)
    SEL_PACKED = 1,   // one unit per tensor and expert: (key, ~pos) > (t, ~cut)
    SEL_BLOCK = 2,    // BLOCK scope: the unit of each entry's block
};

enum OpKind : int { OPK_SUM = 0, OPK_TIES = 1, OPK_ISO = 2, OPK_RAM = 3 };

template <int KC>
struct MergeParams {
    const void* xs[KC];
    unsigned long long thr[KC];   // SEL_PACKED, tensor-local positions
    float cf[KC];                 // ISO 2-D coefficients
    int sel, opk;
    int teps;                     // RAM: key of eps_act (active: key > teps)
    bool iso1d, trimmed2d;
};

// the warp's copy of one tensor's parameters lives in shared memory, which
// keeps the registers for the data in flight; lane q fetches expert q's, lane
// 0 the tensor's
template <int KC>
__device__ __forceinline__ void merge_params(const Plan& P, int t, int K, MergeParams<KC>& mp) {
    __syncwarp();
    const int lane = threadIdx.x & 31;
    const TensorDesc& d = P.tens[t];
    const bool is1d = (d.flags & TF_1D) != 0;
    const bool trim = (d.flags & TF_TRIM) != 0;
    const bool iso1d = (P.op == ISO_OP_ISO) && is1d;
    const int opk = (P.op == ISO_OP_TA || iso1d) ? OPK_SUM
                  : (P.op == ISO_OP_TIES ? OPK_TIES : (P.op == ISO_OP_RAM ? OPK_RAM : OPK_ISO));
    int sel;
    if (opk == OPK_SUM || opk == OPK_RAM || (opk == OPK_TIES && !trim)) sel = SEL_ALL;
    else if (trim && P.scope == ISO_SCOPE_BLOCK) sel = SEL_BLOCK;
    else sel = SEL_PACKED;
    if (lane == 0) {
        mp.iso1d = iso1d;
        mp.trimmed2d = trim && !is1d;
        mp.opk = opk;
        mp.teps = (int)__float_as_uint(P.eps_act);   // eps_act >= +0 and finite: below 2^31
        mp.sel = sel;
    }
    if (lane < KC) {
        const int i = lane;
        mp.xs[i] = (i < K) ? P.xptr[i * P.n_tensors + t] : nullptr;
        mp.cf[i] = (i < K && opk == OPK_ISO) ? (float)P.coef[(long long)t * K + i] : 0.0f;
        uint32_t tk = 0;
        long long cut = CUT_ALL;
        if (i < K && trim && sel != SEL_BLOCK) {
            const Unit& U = P.units[(long long)i * P.n_units + ((P.scope == ISO_SCOPE_GLOBAL) ? 0 : d.unit)];
            tk = U.t;
            cut = U.cut;
        }
        // GLOBAL scope: the unit's cut is a position in the concatenation; entry
        // e of this tensor sits at uoff + e, so the tensor-local cut is cut - uoff
        // clamped to [0, 2^32 - 1] (numel < 2^32 keeps every local position below)
        const long long pos_off = (P.scope == ISO_SCOPE_GLOBAL) ? d.uoff : 0;
        const long long lc = (cut == CUT_ALL) ? cut : cut - pos_off;
        const uint32_t c32 = (lc >= 0xFFFFFFFFLL) ? 0xFFFFFFFFu : (lc <= 0 ? 0u : (uint32_t)lc);
        mp.thr[i] = ((unsigned long long)tk << 32) | (uint32_t)~c32;
    }
    __syncwarp();
}

// selection bits of the K experts at entry e (tensor-local), bit i for expert i
template <int KC>
__device__ __forceinline__ uint32_t select_bits(const Plan& P, const TensorDesc& d, const MergeParams<KC>& mp,
                                                int K, const float (&tau)[KC], long long e, long long& r,
                                                long long& c) {
    uint32_t bits = 0;
    if (mp.sel == SEL_ALL) return (1u << KC) - 1u;
    if (mp.sel == SEL_PACKED) {
        const uint32_t np = ~(uint32_t)e;
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            const unsigned long long kp = ((unsigned long long)key_of(tau[i]) << 32) | np;
            if (i < K && kp > mp.thr[i]) bits |= 1u << i;
        }
    } else {
        const int u = d.unit + (int)(r / P.block_rows) * d.bpr + (int)(c / P.block_cols);
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            if (i < K) {
                const Unit& U = P.units[(long long)i * P.n_units + u];
                SelParam s;
                s.t = U.t;
                s.cut = U.cut;
                if (kept(key_of(tau[i]), e, s)) bits |= 1u << i;
            }
        }
        if (++c == d.cols) { c = 0; ++r; }
    }
    return bits;
}

// the merged output of one entry of a trimmed tensor (TIES or ISO 2-D); every
// argument is in registers.  Untrimmed tensors (SEL_ALL) never come here: every
// tile of theirs takes a per-tile form.
template <int KC>
__device__ __forceinline__ float merged_value(int opk, float lambda, int K, float th0, const float (&tau)[KC],
                                              const float (&cf)[KC], uint32_t bits) {
    float upd;
    if (opk == OPK_TIES) {
        // gamma = sign(sum of the trimmed values); the agreeing set holds the
        // non-zero trimmed values of that sign (none when the sum is 0)
        float tt[KC];
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            tt[i] = (i < K && ((bits >> i) & 1u)) ? tau[i] : 0.0f;
            if (i < K) s = __fadd_rn(s, tt[i]);
        }
        const uint32_t sbit = __float_as_uint(s) & 0x80000000u;
        float a = 0.0f;
        int cnt = 0;
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            const bool agree = (i < K) && (tt[i] != 0.0f) && ((__float_as_uint(tt[i]) & 0x80000000u) == sbit);
            a = agree ? __fadd_rn(a, tt[i]) : a;
            cnt += agree;
        }
        if (s == 0.0f) cnt = 0;
        const float m = cnt ? __fdiv_rn(a, (float)cnt) : 0.0f;
        upd = __fmul_rn(lambda, m);
    } else {
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < KC; ++i)
            if (i < K && ((bits >> i) & 1u)) s = __fadd_rn(s, __fmul_rn(cf[i], tau[i]));
        upd = s;
    }
    return (upd == 0.0f) ? th0 : __fadd_rn(th0, upd);
}

// Per-tile thresholds.  Inside a tile that lies wholly before (after) a unit's
// cut, an entry with key == t is kept (dropped), so the selection is the
// single comparison  (int)key > T  with T = t - 1 (T = t); keys are below 2^31.
// A tile holding the cut, and BLOCK scope, take the exact per-entry test.
template <int KC>
__device__ __forceinline__ bool tile_thresholds(const MergeParams<KC>& mp, int K, uint32_t e0, uint32_t e1,
                                                int (&T)[KC]) {
    bool exact = (mp.sel == SEL_BLOCK);
#pragma unroll
    for (int i = 0; i < KC; ++i) {
        T[i] = (i < K) ? -1 : 0x7FFFFFFF;                      // experts past K: nothing kept
        if (i < K && mp.opk == OPK_RAM) T[i] = mp.teps;        // RAM: active where |tau| > eps_act
        if (i < K && mp.sel == SEL_PACKED) {
            const unsigned long long th = mp.thr[i];
            const uint32_t tk = (uint32_t)(th >> 32), c32 = ~(uint32_t)th;
            if (tk > 0x7FFFFFFEu) T[i] = 0x7FFFFFFF;          // nothing is kept
            else if (e1 <= c32) T[i] = (int)tk - 1;            // ties kept
            else if (e0 >= c32) T[i] = (int)tk;                // ties dropped
            else exact = true;
        }
    }
    return exact;
}

// merged output of one entry inside a tile with per-tile thresholds (the
// compact passes; k_merge has merge_pair): the selection of expert q is
// (int)key > T[q] (never for q >= K), unselected terms enter the sums as +0,
// which leaves every sum and the output as the skipping form gives them
template <int KC>
__device__ __forceinline__ float merged_fast(int opk, float lambda, int K, float th0, const float (&tau)[KC],
                                             const float (&cf)[KC], const int (&T)[KC]) {
    float upd;
    if (opk == OPK_TIES) {
        // gamma = sign of the trimmed sum; the agreeing set: the non-zero
        // trimmed values of that sign.  u = tt with the sign of the sum
        // cleared is |tt| exactly for the agreeing ones, so their sum in
        // order is the magnitude of the signed sum, bit for bit.
        float tt[KC];
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < KC; ++q) {
            tt[q] = ((int)key_of(tau[q]) > T[q]) ? tau[q] : 0.0f;
            s = __fadd_rn(s, tt[q]);
        }
        const uint32_t sb = __float_as_uint(s) & 0x80000000u;
        float a = 0.0f;
        int cnt = 0;
#pragma unroll
        for (int q = 0; q < KC; ++q) {
            const float u = __uint_as_float(__float_as_uint(tt[q]) ^ sb);
            const bool ag = u > 0.0f;
            a = ag ? __fadd_rn(a, u) : a;
            cnt += ag;
        }
        if (s == 0.0f) cnt = 0;
        float m = cnt ? __fdiv_rn(a, (float)cnt) : 0.0f;
        m = __uint_as_float(__float_as_uint(m) ^ sb);
        upd = __fmul_rn(lambda, m);
    } else if (opk == OPK_ISO) {
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < KC; ++q)
            s = __fadd_rn(s, ((int)key_of(tau[q]) > T[q]) ? __fmul_rn(cf[q], tau[q]) : 0.0f);
        upd = s;
    } else {
        float s = 0.0f;
#pragma unroll
        for (int q = 0; q < KC; ++q)
            if (q < K) s = __fadd_rn(s, tau[q]);
        upd = __fdiv_rn(s, (float)K);                  // ISO 1-D
    }
    return (upd == 0.0f) ? th0 : __fadd_rn(th0, upd);
}

// the warp's tiles: beg, beg + step, ... below end -- dealt round-robin over
// the warps (all warps sweep one window of the tensors together, for DRAM
// page locality) or one contiguous range per warp
struct WarpRange {
    long long beg, end, step;
    __device__ __forceinline__ long long count() const { return beg < end ? (end - beg + step - 1) / step : 0; }
    __device__ __forceinline__ long long tile(long long j) const { return beg + j * step; }
};
__device__ __forceinline__ WarpRange warp_range(const Plan& P) {
    const long long W = (long long)gridDim.x * WPB;
    const long long wid = (long long)blockIdx.x * WPB + (threadIdx.x >> 5);
    WarpRange r;
    if (PASS_INTERLEAVE) {
        r.beg = wid;
        r.end = P.n_tiles;
        r.step = W;
    } else {
        const long long per = (P.n_tiles + W - 1) / W;
        r.beg = wid * per;
        r.end = (r.beg + per < P.n_tiles) ? r.beg + per : P.n_tiles;
        r.step = 1;
    }
    return r;
}

__device__ __forceinline__ long long tensor_tile_end(const Plan& P, int t) {
    return P.tens[t].tile_base + (P.tens[t].numel + TILE - 1) / TILE;
}

}  // namespace

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" :: "r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

__device__ __forceinline__ uint32_t clamp_bytes(long long avail, uint32_t cap) {
    return avail <= 0 ? 0u : (avail >= (long long)cap ? cap : (uint32_t)avail);
}

namespace {

// ---------------------------------------------------------------------------
// Chunk ring.  A warp walks its tiles chunk by chunk (CE consecutive entries);
// lane 0 brings a chunk of every expert, and of the base, into the warp's
// ring of DEPTH stages in shared memory with one bulk copy each, DEPTH chunks
// ahead, tracked by one mbarrier per stage.  The data in flight (about 100 KB
// per SM) then needs no registers and no per-lane copy instructions.  A
// tensor's last, partial chunk is not copied (its stage's barrier is arrived
// on without bytes): the warp reads it from global memory.
// ---------------------------------------------------------------------------
template <typename XT, typename BT, int KC, bool NB>
struct ChunkGeom {
    static constexpr int E = 16 / (int)sizeof(XT);                  // entries per lane per step
    static constexpr int STEP = 32 * E;
    static constexpr int BPE = KC * (int)sizeof(XT) + (NB ? (int)sizeof(BT) : 0);   // bytes per entry
    static constexpr int BUDGET = 13824;                            // ring bytes per warp: two blocks per SM
    static constexpr int CE = BPE * 1024 * 3 <= BUDGET ? 1024 : BPE * 512 * 2 <= BUDGET ? 512
                            : BPE * 256 * 2 <= BUDGET ? 256 : 128;
    static constexpr int SPC = CE / STEP;                           // steps per chunk
    static constexpr int CPT = TILE / CE;                           // chunks per tile
    static constexpr int BYTES = CE * BPE;
    static constexpr int D0 = BUDGET / BYTES;
    static constexpr int DEPTH = D0 > 4 ? 4 : D0;
    static constexpr int SMEM = WPB * DEPTH * (BYTES + 8);          // rings, then barriers
    static_assert(DEPTH >= 2 && SPC >= 1 && CE % STEP == 0, "chunk ring");
};

// body(g, c, stage): chunk c of tile g, its data at `stage` (expert q's CE
// entries at q * CE * sizeof(XT), the base's after KC of them) when the chunk
// is whole.  Returns false when a wait gave up (reported in the status word).
template <typename G, typename XT, typename BT, int KC, bool NB, typename Body>
__device__ __forceinline__ bool stream_chunks(const Plan& P, int K, const WarpRange& wr, unsigned char* smem,
                                              Body&& body) {
    constexpr int D = G::DEPTH;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char* const ring = smem + (size_t)warp * D * G::BYTES;
    const uint32_t ring_s = smem_u32(ring);
    const uint32_t bar_s = smem_u32(smem + (size_t)WPB * D * G::BYTES) + 8u * D * warp;
    __shared__ const char* s_xs[WPB][KC + 1];
    if (lane == 0) {
        for (int s = 0; s < D; ++s) mbar_init(bar_s + 8u * s, 1);
        mbar_fence_init();
    }
    __syncwarp();
    const long long NC = wr.count() * G::CPT;
    // lane 0's cursor: the tensor that the next copies come from
    int it = -1;
    long long it_end = 0, it_base = 0, in = 0;
    auto issue = [&](long long i, int s) {
        if (lane != 0) return;
        const long long g = wr.tile(i / G::CPT);
        if (g >= it_end) {
            if (it < 0) it = tensor_of_tile(P.tens, P.n_tensors, g);
            while (g >= tensor_tile_end(P, it)) ++it;
            const TensorDesc& d = P.tens[it];
            it_base = d.tile_base;
            it_end = tensor_tile_end(P, it);
            in = d.numel;
            for (int q = 0; q < K; ++q) s_xs[warp][q] = static_cast<const char*>(P.xptr[q * P.n_tensors + it]);
            s_xs[warp][KC] = static_cast<const char*>(d.base);
        }
        const long long e = (g - it_base) * TILE + (i % G::CPT) * G::CE;
        const uint32_t bar = bar_s + 8u * s, dst = ring_s + (uint32_t)(s * G::BYTES);
        if (e + G::CE <= in) {
            constexpr uint32_t XB = G::CE * sizeof(XT), BB = G::CE * sizeof(BT);
            mbar_arrive_tx(bar, K * XB + (NB ? BB : 0u));
#pragma unroll
            for (int q = 0; q < KC; ++q)
                if (q < K) bulk_g2s(dst + q * XB, s_xs[warp][q] + e * (long long)sizeof(XT), XB, bar);
            if (NB) bulk_g2s(dst + KC * XB, s_xs[warp][KC] + e * (long long)sizeof(BT), BB, bar);
        } else {
            mbar_arrive(bar);
        }
    };
    for (int s = 0; s < D; ++s)
        if (s < NC) issue(s, s);
    uint32_t phases = 0;
    int s = 0;
#pragma unroll 1
    for (long long i = 0; i < NC; ++i) {
        const uint32_t bar = bar_s + 8u * s;
        if (!mbar_wait_warp(bar, (phases >> s) & 1u)) {
            // give up: report, then wait (bounded) for the copies this
            // warp still has in flight before the block may exit
            if (lane == 0) set_status(P.hdr, ISO_ERR_TIMEOUT);
            const int pend = (int)(NC - i < D ? NC - i : D);
            for (int j = 0; j < pend; ++j) {
                const int sj = (s + j) % D;
                mbar_wait(bar_s + 8u * sj, (phases >> sj) & 1u);
            }
            __syncwarp();
            return false;
        }
        phases ^= 1u << s;
        body(wr.tile(i / G::CPT), (int)(i % G::CPT), ring + s * G::BYTES);
        // the stage's reads come before its next copy
        __syncwarp();
        if (i + D < NC) {
            if (lane == 0) fence_proxy_async_smem();
            issue(i + D, s);
        }
        s = (s + 1 == D) ? 0 : s + 1;
    }
    return true;
}

// this lane's words of one step: from the stage, or from global memory for a
// partial chunk (entries past the tensor's end read 0); experts K .. KC - 1
// read 0
template <typename G, typename XT, typename BT, int KC, bool NB>
__device__ __forceinline__ void chunk_words(const unsigned char* stage, bool whole, int s, int K, const void* const* xs,
                                            const void* base, long long e, long long n, int lane,
                                            Words<XT, G::E> (&x)[KC], Words<BT, G::E>& b) {
    constexpr int E = G::E;
    if (whole) {
        const unsigned char* p = stage + (s * G::STEP + lane * E) * (int)sizeof(XT);
#pragma unroll
        for (int q = 0; q < KC; ++q) {
            uint4 v = make_uint4(0, 0, 0, 0);
            if (q < K) v = *reinterpret_cast<const uint4*>(p + q * (G::CE * (int)sizeof(XT)));
            x[q].w[0] = v.x; x[q].w[1] = v.y; x[q].w[2] = v.z; x[q].w[3] = v.w;
        }
        if (NB) {
            const unsigned char* pb = stage + KC * (G::CE * (int)sizeof(XT)) + (s * G::STEP + lane * E) * (int)sizeof(BT);
            constexpr int N = Words<BT, E>::N;
            if (N == 2) {
                const uint2 v = *reinterpret_cast<const uint2*>(pb);
                b.w[0] = v.x; b.w[1] = v.y;
            } else {
#pragma unroll
                for (int q = 0; q < N / 4; ++q) {
                    const uint4 v = *reinterpret_cast<const uint4*>(pb + 16 * q);
                    b.w[4 * q] = v.x; b.w[4 * q + 1] = v.y; b.w[4 * q + 2] = v.z; b.w[4 * q + 3] = v.w;
                }
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < KC; ++q) {
#pragma unroll
            for (int w = 0; w < Words<XT, E>::N; ++w) x[q].w[w] = 0;
            if (q < K && e < n) load_words<XT, E>(xs[q], e, n, x[q]);
        }
        if (NB) {
#pragma unroll
            for (int w = 0; w < Words<BT, E>::N; ++w) b.w[w] = 0;
            if (e < n) load_words<BT, E>(base, e, n, b);
        }
    }
}

// The per-tile threshold as a binary32 bound: for finite tau, (int)key > T
// exactly where |tau| > bound (binary32 magnitudes order like their bits).
__device__ __forceinline__ float bound_of(int T) {
    return T < 0 ? -1.0f : (T == 0x7FFFFFFF ? __uint_as_float(KEY_INF) : __int_as_float(T));
}

}  // namespace

}  // namespace iso
