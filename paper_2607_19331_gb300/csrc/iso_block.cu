// iso_block.cu -- TopKMask with per-block thresholds (BLOCK scope).
//
// Each unit is one block_rows x block_cols tile of a row-major tensor, in
// row-major tile order; entries inside a tile keep the tensor's own index
// order, so "lowest index first" among equal |tau| is the tile's row-major
// order.  One CTA holds a whole unit on chip: a full block as task-vector values
// in registers, 32 consecutive entries a thread, a partial edge block as keys
// in shared memory.  The k-th largest key comes from a radix select (11 bits a
// level) and the ties from an ordered block scan.  Where the call is the K = 1
// TIES update the same kernel writes the unit's outputs; otherwise the result
// (t, cut) feeds the streaming passes of the other scopes.
#include "iso_kernels.cuh"

#include <type_traits>

namespace iso {

__device__ __forceinline__ long long k_of_density_b(double rho, long long n) {
    double kk = floor(__dadd_rn(__dmul_rn(rho, (double)n), 0.5));
    if (kk < 0.0) kk = 0.0;
    if (kk > (double)n) kk = (double)n;
    return (long long)kk;
}

__device__ void block_find_from_top_b(const uint32_t* hist, int nb, long long rank,
                                      long long* sm_scan, int* res_bin, long long* res_above) {
    const int per = (nb + blockDim.x - 1) / blockDim.x;
    const int j0 = threadIdx.x * per;
    if (threadIdx.x == 0) { *res_bin = 0; *res_above = 0; }
    long long local = 0;
    for (int j = j0; j < j0 + per && j < nb; ++j) local += hist[nb - 1 - j];
    long long total;
    const long long excl = block_excl_scan(local, sm_scan, &total);
    if (excl < rank && rank <= excl + local) {
        long long acc = excl;
        for (int j = j0; j < j0 + per && j < nb; ++j) {
            const uint32_t h = hist[nb - 1 - j];
            if (rank <= acc + h) { *res_bin = nb - 1 - j; *res_above = acc; break; }
            acc += h;
        }
    }
    __syncthreads();
}

// Among the nb <= RADIX_BINS counters from the top, the bin that holds rank
// (1 <= rank <= their sum): its index, the count above it and its own count,
// in res.  Two barriers; every thread of the block calls it.
struct BinHit { int bin; uint32_t above, count; };
__device__ __forceinline__ void block_find32(const uint32_t* hist, int nb, uint32_t rank, uint32_t* sm, BinHit* res) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int PER = RADIX_BINS / BLOCK_TPB;
    const int j0 = threadIdx.x * PER;
    uint32_t h[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        h[j] = j0 + j < nb ? hist[nb - 1 - j0 - j] : 0u;
        sum += h[j];
    }
    uint32_t tot;
    uint32_t excl = warp_excl_scan(sum, &tot);
    if (lane == 0) sm[warp] = tot;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < BLOCK_TPB / 32; ++w) excl += w < warp ? sm[w] : 0u;
    if (excl < rank && rank <= excl + sum) {
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (rank > excl && rank <= excl + h[j]) { res->bin = nb - 1 - j0 - j; res->above = excl; res->count = h[j]; }
            excl += h[j];
        }
    }
    __syncthreads();
}

// keys sit at q + q / 32: a thread walking its own contiguous range and a
// warp walking consecutive entries are both free of bank conflicts
__device__ __forceinline__ int kpad(int q) { return q + (q >> 5); }

template <typename XT, typename BT, bool CK>
__global__ void __launch_bounds__(BLOCK_TPB, BLOCK_CTAS_PER_SM) k_block_select(Plan P) {
    pdl_enter();
    extern __shared__ __align__(16) uint32_t s_keys[];      // kpad(BLOCK_MAX_ENTRIES)
    __shared__ uint32_t s_hist[RADIX_BINS];
    __shared__ long long s_scan[33];
    __shared__ uint32_t s_scan32[33];
    __shared__ double s_dred[33];
    __shared__ int s_bin;
    __shared__ long long s_above;
    __shared__ long long s_cutq;
    __shared__ uint32_t s_or;
    __shared__ BinHit s_hit;

    const int idx = blockIdx.x;
    const int i = idx / P.n_units, u = idx % P.n_units;
    // owning tensor: last tensor whose first unit is <= u and that has blocks
    int lo = 0, hi = P.n_tensors - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (P.tens[mid].unit <= u) lo = mid; else hi = mid - 1;
    }
    while (lo > 0 && P.tens[lo].nblocks == 0) --lo;
    const int t = lo;
    const TensorDesc& d = P.tens[t];
    Unit& U = P.units[idx];
    const int b = u - d.unit;
    const int br = b / d.bpr, bc = b % d.bpr;
    const long long r0 = (long long)br * P.block_rows, c0 = (long long)bc * P.block_cols;
    const long long h = min((long long)P.block_rows, d.rows - r0);
    const long long w = min((long long)P.block_cols, d.cols - c0);
    const int n = (int)(h * w);
    auto stats = [&](uint32_t tk, long long k, long long above, long long ties, long long need) {
        if (!P.st_units) return;
        iso_unit_stats s;
        s.thresh_key = tk; s.flags = 0; s.k = k; s.count_above = above;
        s.ties_at_thresh = ties; s.ties_taken = need;
        P.st_units[(long long)i * P.st_units_stride + P.st_unit_base + u] = s;
    };
    const void* x = P.xptr[i * P.n_tensors + t];
    const bool vec = (w % VEC == 0) && (d.cols % VEC == 0) && (c0 % VEC == 0);
    // fused K = 1 update (TIES / masked update): the block's outputs are
    // written here, theta_0 + lambda tau for the kept entries, theta_0 else
    const bool obf = sizeof(BT) == 2;
    auto apply_block = [&](uint32_t tk, long long cut, bool keep_all) {
        if (vec) {
            const int w8 = (int)(w / VEC);
            for (int q8 = threadIdx.x; q8 < n / VEC; q8 += blockDim.x) {
                const int rr = q8 / w8, cc = (q8 - rr * w8) * VEC;
                const long long e = (r0 + rr) * d.cols + c0 + cc;
                float th0[VEC], tau[VEC], o[VEC];
                load8_tail<BT>(d.base, e, d.numel, th0);
                TauSrc<XT, BT, CK>::load8(x, d.base, e, d.numel, tau);
#pragma unroll
                for (int j = 0; j < VEC; ++j) {
                    const uint32_t kk = key_of(tau[j]);
                    const bool kept = keep_all || kk > tk || (kk == tk && e + j < cut);
                    o[j] = kept ? out_of(th0[j], tau[j], P.lambda) : th0[j];
                }
                store8(d.out, e, d.numel, o, obf);
            }
        } else {
            for (int q = threadIdx.x; q < n; q += blockDim.x) {
                const int rr = q / (int)w, cc = q - rr * (int)w;
                const long long e = (r0 + rr) * d.cols + c0 + cc;
                const float th0 = Load8<BT>::one(d.base, e);
                const float tau = TauSrc<XT, BT, CK>::load1(x, d.base, e);
                const uint32_t kk = key_of(tau);
                const bool kept = keep_all || kk > tk || (kk == tk && e < cut);
                const float o = kept ? out_of(th0, tau, P.lambda) : th0;
                if (obf) static_cast<__nv_bfloat16*>(d.out)[e] = __float2bfloat16_rn(o);
                else static_cast<float*>(d.out)[e] = o;
            }
        }
    };
    if (!(d.flags & TF_TRIM)) {
        if (threadIdx.x == 0) {
            U.state = ST_OFF; U.k = -1; U.t = 0; U.cut = CUT_ALL;
            stats(KEY_NONE, -1, 0, 0, 0);
        }
        if (P.fuse_block) apply_block(0u, CUT_ALL, true);
        return;
    }
    // k in binary64 by one thread (binary64 is slow on this GPU), then shared
    __shared__ long long s_k;
    if (threadIdx.x == 0) s_k = k_of_density_b(P.density, n);
    __syncthreads();
    const long long k = s_k;
    if (k == 0) {
        if (threadIdx.x == 0) {
            U.state = ST_NONE; U.k = 0; U.t = KEY_NONE; U.cut = 0;
            stats(KEY_NONE, 0, 0, 0, 0);
        }
        if (P.fuse_block) apply_block(KEY_NONE, 0, false);
        return;
    }
    const bool want_gamma = (P.op == ISO_OP_ISO) && (P.K == 1);

    // Full block of BLOCK_TPB x BFE entries in rows of a multiple of BFE: each
    // thread holds BFE consecutive entries (block order) of the task vector in
    // registers, and the threshold comes from a radix select over those
    // registers, 11 bits per level down to the lowest bit any key has set (two
    // levels for bf16-valued task vectors).  Bound by issue: a descent bit by
    // bit spent two instructions per key and bit (235 us for a 4096 x 14336
    // bf16 task vector at 5 %, outputs included), keys and signs kept apart
    // and rejoined for the outputs 208 us, separate passes for the counts above
    // and at the threshold 188 us, this form 169 us.
    constexpr int BFE = BLOCK_MAX_ENTRIES / BLOCK_TPB;
    if (n == BLOCK_TPB * BFE && w % BFE == 0 && (d.cols % VEC) == 0 && (c0 % VEC) == 0 &&
        blockDim.x == BLOCK_TPB) {
        const int tq = threadIdx.x * BFE;
        const int rr = tq / (int)w, cc = tq - rr * (int)w;
        const long long ea = (r0 + rr) * d.cols + c0 + cc;     // tensor position of the thread's first entry
        // theta_0 is needed only after the select: its lines go to L2 meanwhile
        if (P.fuse_block)
            for (int by = 0; by < BFE * (int)sizeof(BT); by += 64)
                asm volatile("prefetch.global.L2 [%0];" :: "l"(static_cast<const char*>(d.base) + ea * (long long)sizeof(BT) + by));
        float v[BFE];
#pragma unroll
        for (int g = 0; g < BFE / VEC; ++g) {
            float t8[VEC];
            TauSrc<XT, BT, CK>::load8(x, d.base, ea + g * VEC, d.numel, t8);
#pragma unroll
            for (int j = 0; j < VEC; ++j) v[g * VEC + j] = t8[j];
        }
        for (int q = threadIdx.x; q < RADIX_BINS; q += BLOCK_TPB) s_hist[q] = 0;
        if (threadIdx.x == 0) { s_or = 0; s_cutq = CUT_ALL; s_hit = BinHit{0, 0u, 0u}; }
        uint32_t kor = 0;
        float bad0 = 0.0f, bad1 = 0.0f;                // 0 * tau: NaN once a tau is not finite
#pragma unroll
        for (int j = 0; j < BFE; j += 2) {
            kor |= __float_as_uint(v[j]) | __float_as_uint(v[j + 1]);
            fma_rn2(bad0, bad1, v[j], v[j + 1], 0.0f, 0.0f, bad0, bad1);
        }
        if (!(bad0 + bad1 == 0.0f)) set_status(P.hdr, ISO_ERR_NONFINITE);
        kor = __reduce_or_sync(0xFFFFFFFFu, kor & KEY_MAX);
        __syncthreads();
        if ((threadIdx.x & 31) == 0 && kor) atomicOr(&s_or, kor);
        // first level: the top 11 bits of every key
        constexpr int SH1 = 31 - RADIX_BITS;
#pragma unroll
        for (int j = 0; j < BFE; ++j) atomicAdd(&s_hist[(__float_as_uint(v[j]) >> SH1) & (RADIX_BINS - 1)], 1u);
        __syncthreads();
        const int low = s_or ? __ffs(s_or) - 1 : 31;
        uint32_t rank = (uint32_t)k;
        block_find32(s_hist, RADIX_BINS, rank, s_scan32, &s_hit);
        rank -= s_hit.above;
        uint32_t prefix = (uint32_t)s_hit.bin;
        int pshift = SH1;
        while (pshift > low) {
            const int shift = max(pshift > RADIX_BITS ? pshift - RADIX_BITS : 0, low);
            const uint32_t nm = (1u << (pshift - shift)) - 1u;
            for (int q = threadIdx.x; q <= (int)nm; q += BLOCK_TPB) s_hist[q] = 0;
            __syncthreads();
            const uint32_t want = prefix << pshift, mask = KEY_MAX & ~((1u << pshift) - 1u);
#pragma unroll
            for (int j = 0; j < BFE; ++j) {
                const uint32_t b = __float_as_uint(v[j]);
                if ((b & mask) == want) atomicAdd(&s_hist[(b >> shift) & nm], 1u);
            }
            __syncthreads();
            block_find32(s_hist, (int)nm + 1, rank, s_scan32, &s_hit);
            rank -= s_hit.above;
            prefix = (prefix << (pshift - shift)) | (uint32_t)s_hit.bin;
            pshift = shift;
        }
        const uint32_t tk = prefix << pshift;
        const float tf = __uint_as_float(tk);
        // what is left of the rank are the ties to keep, of as many as the last bin holds
        const long long need = (long long)rank, tot_above = k - need;
        const uint32_t tot_ties = s_hit.count;
        if (need < (long long)tot_ties) {
            uint32_t ties = 0, all;
#pragma unroll
            for (int j = 0; j < BFE; ++j) ties += fabsf(v[j]) == tf;
            const uint32_t ties_before = block_excl_scan(ties, s_scan32, &all);
            if ((long long)ties_before < need && need <= (long long)(ties_before + ties)) {
                uint32_t acc = ties_before;
#pragma unroll
                for (int j = 0; j < BFE; ++j)
                    if (fabsf(v[j]) == tf && (long long)(++acc) == need) s_cutq = ea + j + 1;
            }
        }
        double g = 0.0;
        if (want_gamma) {
            // squares of the entries above t as binary32 two-sum pairs, then binary64 over the block
            float sg = 0.0f, eg = 0.0f;
#pragma unroll
            for (int j = 0; j < BFE; ++j)
                if (fabsf(v[j]) > tf) two_sum_add(sg, eg, __fmul_rn(v[j], v[j]));
            g = block_sum((double)sg + (double)eg, s_dred);
        }
        __syncthreads();
        const long long cut = s_cutq;
        if (threadIdx.x == 0) {
            U.n = n; U.k = k; U.t = tk; U.cut = cut;
            U.count_above = tot_above; U.ties = tot_ties; U.need = need;
            U.state = ST_DONE;
            if (want_gamma) {
                const double ft = (double)__uint_as_float(tk);
                U.gamma = g + (double)need * ft * ft;
            }
            stats(tk, k, tot_above, tot_ties, need);
        }
        if (P.fuse_block) {
            // ties are kept at the thread's first kt entries: |tau| above this
            // bound (below t's magnitude, or t's own) is kept
            const long long before = cut - ea;
            const int kt = before <= 0 ? 0 : (before >= BFE ? BFE : (int)before);
            const float tl = tk ? __uint_as_float(tk - 1) : -1.0f;
            auto put = [&](auto same, float bound) {
#pragma unroll
                for (int gq = 0; gq < BFE / VEC; ++gq) {
                    const long long e = ea + gq * VEC;
                    float th0[VEC], o[VEC];
                    load8_tail<BT>(d.base, e, d.numel, th0);
#pragma unroll
                    for (int j = 0; j < VEC; ++j) {
                        const int q = gq * VEC + j;
                        const float bd = decltype(same)::value ? bound : (q < kt ? tl : tf);
                        o[j] = fabsf(v[q]) > bd ? out_of(th0[j], v[q], P.lambda) : th0[j];
                    }
                    store8(d.out, e, d.numel, o, obf);
                }
            };
            if (kt == 0 || kt == BFE) put(std::integral_constant<bool, true>{}, kt ? tl : tf);
            else put(std::integral_constant<bool, false>{}, 0.0f);
        }
        return;
    }
    // keys in block order (row-major inside the block)
    bool bad = false;
    uint32_t kor = 0;                        // OR of the keys: trailing zero bits need no radix level
    if (threadIdx.x == 0) s_or = 0;
    __syncthreads();
    if (vec) {
        const int w8 = (int)(w / VEC);
        for (int q8 = threadIdx.x; q8 < n / VEC; q8 += blockDim.x) {
            const int rr = q8 / w8, cc = (q8 - rr * w8) * VEC;
            const long long e = (r0 + rr) * d.cols + c0 + cc;
            float tau[VEC];
            TauSrc<XT, BT, CK>::load8(x, d.base, e, d.numel, tau);
#pragma unroll
            for (int j = 0; j < VEC; ++j) {
                const uint32_t kk = key_of(tau[j]);
                bad |= kk >= KEY_INF;
                kor |= kk;
                s_keys[kpad(q8 * VEC + j)] = kk;
            }
        }
    } else {
        for (int q = threadIdx.x; q < n; q += blockDim.x) {
            const int rr = q / (int)w, cc = q - rr * (int)w;
            const long long e = (r0 + rr) * d.cols + c0 + cc;
            const uint32_t kk = key_of(TauSrc<XT, BT, CK>::load1(x, d.base, e));
            bad |= kk >= KEY_INF;
            kor |= kk;
            s_keys[kpad(q)] = kk;
        }
    }
    if (bad) set_status(P.hdr, ISO_ERR_NONFINITE);
    kor = __reduce_or_sync(0xFFFFFFFFu, kor);
    if ((threadIdx.x & 31) == 0 && kor) atomicOr(&s_or, kor);
    __syncthreads();
    // k-th largest key: radix levels down to the lowest bit any key has set
    // (bf16-valued task vectors leave the low 16 bits clear)
    const int low = s_or ? __ffs(s_or) - 1 : 31;
    uint32_t prefix = 0;
    long long rank = k;
    int pshift = 31;
    for (;;) {
        int shift = pshift > RADIX_BITS ? pshift - RADIX_BITS : 0;
        if (shift < low) shift = low;
        const int nb = 1 << (pshift - shift);
        for (int q = threadIdx.x; q < nb; q += blockDim.x) s_hist[q] = 0;
        __syncthreads();
        for (int q = threadIdx.x; q < n; q += blockDim.x) {
            const uint32_t v = s_keys[kpad(q)];
            if ((v >> pshift) == prefix) atomicAdd(&s_hist[(v >> shift) & (nb - 1)], 1u);
        }
        __syncthreads();
        block_find_from_top_b(s_hist, nb, rank, s_scan, &s_bin, &s_above);
        rank -= s_above;
        prefix = (prefix << (pshift - shift)) | (uint32_t)s_bin;
        __syncthreads();
        if (shift == low) break;
        pshift = shift;
    }
    const uint32_t tk = prefix << low;
    // counts above / at the threshold, and the squared norm of the kept entries
    const int per = (n + blockDim.x - 1) / blockDim.x;
    const int q0 = threadIdx.x * per;
    uint32_t above = 0, ties = 0;
    double gsum = 0.0;
    for (int q = q0; q < q0 + per && q < n; ++q) {
        const uint32_t v = s_keys[kpad(q)];
        above += v > tk;
        ties += v == tk;
        if (want_gamma && v > tk) {
            const double f = (double)__uint_as_float(v);
            gsum += f * f;
        }
    }
    uint32_t tot_ties;
    const uint32_t ties_before = block_excl_scan(ties, s_scan32, &tot_ties);
    const uint32_t tot_above = block_sum(above, s_scan32);
    const long long need = k - (long long)tot_above;
    if (threadIdx.x == 0) s_cutq = -1;
    __syncthreads();
    if (need < (long long)tot_ties) {
        if ((long long)ties_before < need && need <= (long long)(ties_before + ties)) {
            uint32_t acc = ties_before;
            for (int q = q0; q < q0 + per && q < n; ++q)
                if (s_keys[kpad(q)] == tk && (long long)(++acc) == need) { s_cutq = q; break; }
        }
    }
    __syncthreads();
    double g = 0.0;
    if (want_gamma) g = block_sum(gsum, s_dred);
    long long cut = CUT_ALL;
    if (s_cutq >= 0) {
        const long long rr = s_cutq / w, cc = s_cutq - rr * w;
        cut = (r0 + rr) * d.cols + c0 + cc + 1;
    }
    if (threadIdx.x == 0) {
        U.n = n; U.k = k; U.t = tk; U.cut = cut;
        U.count_above = tot_above; U.ties = tot_ties; U.need = need;
        U.state = ST_DONE;
        if (want_gamma) {
            const double ft = (double)__uint_as_float(tk);
            U.gamma = g + (double)need * ft * ft;
        }
        stats(tk, k, tot_above, tot_ties, need);
    }
    if (P.fuse_block) apply_block(tk, cut, false);
}

// K = 1 ISO: a tensor's Gamma from its units' sums, in a fixed order (one block
// per tensor)
__global__ void __launch_bounds__(TPB) k_block_gamma(Plan P) {
    pdl_enter();
    __shared__ double red[33];
    const TensorDesc& d = P.tens[blockIdx.x];
    double g = 0.0;
    for (int b = threadIdx.x; b < d.nblocks; b += TPB) g += P.units[d.unit + b].gamma;
    g = block_sum(g, red);
    if (threadIdx.x == 0) P.gram[blockIdx.x] = g;
}

#define ISO_BLOCK_INST(XT, BT, CK) template __global__ void k_block_select<XT, BT, CK>(Plan);
ISO_BLOCK_INST(__nv_bfloat16, __nv_bfloat16, false)
ISO_BLOCK_INST(__nv_bfloat16, float, false)
ISO_BLOCK_INST(float, __nv_bfloat16, false)
ISO_BLOCK_INST(float, float, false)
ISO_BLOCK_INST(__nv_bfloat16, __nv_bfloat16, true)
ISO_BLOCK_INST(__nv_bfloat16, float, true)
ISO_BLOCK_INST(float, __nv_bfloat16, true)
ISO_BLOCK_INST(float, float, true)

}  // namespace iso
