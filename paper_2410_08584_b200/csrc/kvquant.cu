// Mixed-precision KV cache (Sec. 4.3, Table 3: the tokens of T at 4 bits, the others at 2)
// and the decode step over it (Algorithm 2, Eq. 4-5, with the rows dequantised on the fly).
//
// The paper takes the quantiser from the work it cites and fixes only the bit allocation.
// The reading built here: no token is evicted; keys and values are quantised per (token,
// KV head) over the head_dim channels with an asymmetric uniform quantiser,
//     scale = (max - min) / (2^b - 1),  code = clip(rint((x - min) * (1 / scale)), 0, 2^b - 1),
// scale and min rounded to the storage type and kept beside the codes; every step that
// decides a code is a single correctly rounded fp32 operation, so the codes are the same
// bits as the CPU checker's.  Softmax attention does not depend on the order of the cached
// rows, so the cache is two blocks: "hi" (the tokens of T, in T's order; decoded tokens are
// appended here) and "lo" (the others, ascending).  Codes are packed little-end first
// (channel c in byte c*b/8 at bit (c*b)%8); a row of a block is Hkv * d*b/8 bytes; the
// parameters of a block are [rows, Hkv, 4] storage-type values (k scale, k min, v scale, v min).
#include <math.h>

#include "kvquant.cuh"

namespace zipvl {
namespace {

using namespace kvq;

// What bounds the encoder: it reads 4 bytes and writes about 1 per (channel of K and V), so HBM has
// to be kept busy at some 25 values per SM and cycle, i.e. with about ten instructions per value at
// most.  One lane per eight channels, a division and a reciprocal per lane and tensor, a
// conversion each way per value and, in front of all, a 12-step binary search per token took 30 us for
// the 2944-token, 32-head layer (60 MB).  Here
//   - eight lanes share a row of 64 or 128 channels of K and V of two (token, head) pairs, so the four
//     divisions and reciprocals of a group are done by four different lanes at once;
//   - the row's maximum and negated minimum travel in one register of packed 16-bit values (the
//     minimum is an element: storing it as the row's zero rounds nothing);
//   - rint is an addition of 1.5 * 2^23 (exact to even for the values up to 15 that occur), and the
//     sums of the code words' terms come out by integer multiply-adds modulo 2^32;
//   - the loads of a CTA's first rows are under way while the token set is searched, 32 ways at a time.
// 30 -> 17 us.
constexpr int kQuantThreads = 128;
constexpr int kQuantIters = 4;      // steps of 32 (token, head) pairs per CTA
constexpr int kQuantPairs = (kQuantThreads / 8) * 2;

// packed pair of storage-type values
template <bool kHalf>
__device__ __forceinline__ uint32_t pk_max(uint32_t a, uint32_t b) {        // NaN if either is
    uint32_t d;
    if (kHalf) asm("max.NaN.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    else asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
template <bool kHalf>
__device__ __forceinline__ uint32_t pk_min(uint32_t a, uint32_t b) {
    uint32_t d;
    if (kHalf) asm("min.NaN.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    else asm("min.NaN.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

template <bool kHalf, int D>
__global__ void __launch_bounds__(kQuantThreads, 5)
quantize_kv_kernel(LayerArgs a, const unsigned short *__restrict__ k, const unsigned short *__restrict__ v,
                   const int32_t *__restrict__ idx, const int32_t *__restrict__ k_dev, int k_max,
                   QuantBlocks qb, int32_t *__restrict__ lens_out, int32_t *status_word) {
    constexpr int P = D / 64;                     // 16-byte pieces per lane (8 lanes to a row)
    constexpr int kPairsPerCta = kQuantPairs * kQuantIters;
    __shared__ int s_row[kPairsPerCta + 2];       // where a token goes: >= 0: hi row; < 0: -(lo row) - 1
    __shared__ int s_entry[kPairsPerCta + 2], s_low;
    grid_launch_dependents();
    grid_dependency_wait(k, v, idx, k_dev);       // T and k are the selection's output
    const int lane = threadIdx.x & 31, lg = lane & 7;
    // (pair numbers fit 32 bits: 2^32 rows of K alone would be half a terabyte)
    const uint32_t n_pairs = (uint32_t)a.L * (uint32_t)a.Hkv, p0 = blockIdx.x * (uint32_t)kPairsPerCta;
    const uint32_t t_first = p0 / (uint32_t)a.Hkv, g_first = p0 - t_first * (uint32_t)a.Hkv;
    const unsigned long long inv_heads = ((1ull << 32) + a.Hkv - 1) / (uint32_t)a.Hkv;    // exact quotients below 2^16
    // combination u: tensor u & 1 (K, V) of pair u >> 1 of this group of lanes
    uint4 w[4][P];
    auto pair_of = [&](int it, int half) { return p0 + (uint32_t)(it * kQuantPairs + (threadIdx.x >> 3) * 2 + half); };
    auto token_of = [&](uint32_t p) { return (uint32_t)(((unsigned long long)(p - p0 + g_first) * inv_heads) >> 32); };   // behind t_first
    auto load = [&](int it) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const uint32_t p = pair_of(it, half);
            if (p < n_pairs) {
                const uint32_t j = token_of(p), h = p - p0 + g_first - j * (uint32_t)a.Hkv;
                const long long off = (long long)(t_first + j) * a.kv_stride + h * D + lg * 8;
#pragma unroll
                for (int i = 0; i < P; ++i) {
                    w[2 * half][i] = __ldg(reinterpret_cast<const uint4 *>(k + off + i * 64));
                    w[2 * half + 1][i] = __ldg(reinterpret_cast<const uint4 *>(v + off + i * 64));
                }
            } else {
#pragma unroll
                for (int i = 0; i < P; ++i) { w[2 * half][i] = make_uint4(0, 0, 0, 0); w[2 * half + 1][i] = make_uint4(0, 0, 0, 0); }
            }
        }
    };
    load(0);
    int n = *k_dev;
    if (n > k_max || n < 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) report(status_word, ZIPVL_DEV_CAPACITY);
        n = n < 0 ? 0 : k_max;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (n > qb.cap_hi || a.L - n > qb.cap_lo) report(status_word, ZIPVL_DEV_CAPACITY);
        lens_out[0] = min(n, qb.cap_hi);
        lens_out[1] = min(a.L - n, qb.cap_lo);
    }
    // A CTA takes consecutive (token, head) pairs, i.e. a short run of tokens.  Where each of those
    // goes -- row i of the 4-bit block if it is T's i-th entry, else row (t - #entries of T below t)
    // of the 2-bit block -- is looked up once: the first warp finds the first entry >= t_first,
    // splitting the range 32 ways per step, and the entries behind it are compared.
    const int count = (int)token_of(min(p0 + kPairsPerCta, n_pairs) - 1) + 1;
    if (threadIdx.x < 32) {
        const int tf = (int)t_first;
        int lo = max(0, tf - (a.L - n)), hi = max(lo, min(n, tf));   // (ascending: idx[i] >= i, and L - n are left out)
        while (lo < hi) {                         // idx[lo - 1] < t_first <= idx[hi]
            const int step = (hi - lo + 31) / 32, at = lo + (lane + 1) * step - 1;
            const bool below = at < hi && idx[at] < tf;
            const int c = __popc(__ballot_sync(0xffffffffu, below));
            lo += c * step;
            hi = min(hi, lo + step - 1);
        }
        if (lane == 0) s_low = lo;
    }
    __syncthreads();
    const int low = s_low;
    for (int i = threadIdx.x; i < count; i += kQuantThreads) s_entry[i] = low + i < n ? idx[low + i] : 0x7fffffff;
    __syncthreads();
    for (int j = threadIdx.x; j < count; j += kQuantThreads) {
        const int t = (int)t_first + j;
        int below = 0;                            // entries below token t
        while (below < count && s_entry[below] < t) ++below;
        s_row[j] = (below < count && s_entry[below] == t) ? low + below : -(t - low - below) - 1;
    }
    __syncthreads();

#pragma unroll 1
    for (int it = 0; it < kQuantIters; ++it) {
        if (p0 + it * kQuantPairs + (threadIdx.x >> 5) * 8 >= n_pairs) break;      // (the warp's first pair)
        int row[2], bits[2];
        long long rh[2];
        bool fits[2];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const uint32_t p = pair_of(it, half);
            const bool live = p < n_pairs;
            const uint32_t j = live ? token_of(p) : 0, h = live ? p - p0 + g_first - j * (uint32_t)a.Hkv : 0;
            const int where = s_row[j];
            bits[half] = where >= 0 ? 4 : 2;
            row[half] = where >= 0 ? where : -where - 1;
            fits[half] = live && row[half] >= 0 && row[half] < (where >= 0 ? qb.cap_hi : qb.cap_lo);
            rh[half] = (long long)row[half] * a.Hkv + h;
        }
        // (max, -min) of each combination
        uint32_t mm[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            uint32_t hi = w[u][0].x, lo = w[u][0].x;
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const uint32_t x[4] = {w[u][i].x, w[u][i].y, w[u][i].z, w[u][i].w};
#pragma unroll
                for (int e = (i == 0); e < 4; ++e) { hi = pk_max<kHalf>(hi, x[e]); lo = pk_min<kHalf>(lo, x[e]); }
            }
            lo ^= 0x80008000u;
            mm[u] = pk_max<kHalf>(__byte_perm(hi, lo, 0x5410), __byte_perm(hi, lo, 0x7632));
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1)
#pragma unroll
            for (int u = 0; u < 4; ++u) mm[u] = pk_max<kHalf>(mm[u], __shfl_xor_sync(0xffffffffu, mm[u], o));
        // scale and reciprocal of combination lg & 3
        const int mine = lg & 3;
        const uint32_t m = mine == 0 ? mm[0] : mine == 1 ? mm[1] : mine == 2 ? mm[2] : mm[3];
        const int my_bits = mine < 2 ? bits[0] : bits[1];
        const float mx = storage_to_float<kHalf>((unsigned short)(m & 0xffffu));
        const unsigned short zero_bits = (unsigned short)((m >> 16) ^ 0x8000u);
        const float zero_mine = storage_to_float<kHalf>(zero_bits);
        unsigned short scale_bits;
        const float scale = storage_round<kHalf>(__fdiv_rn(__fsub_rn(mx, zero_mine), my_bits == 4 ? 15.f : 3.f), &scale_bits);
        const float inv_mine = scale > 0.f ? __frcp_rn(scale) : 0.f;
        // A scale that is no normal number of its type (its rounding error may take a code past the
        // last level), a row with a NaN or an infinity: the quantiser of the append, step by step
        const float smallest = kHalf ? 6.103515625e-5f : 1.17549435e-38f;
        const bool odd = !(scale >= smallest && scale < 3e38f) && !(mx == zero_mine);
        if (__any_sync(0xffffffffu, odd || mx != mx || fabsf(mx) > 3.3e38f || fabsf(zero_mine) > 3.3e38f)) {
#pragma unroll 1
            for (int u = 0; u < 4; ++u) {
                const int bt = u < 2 ? bits[0] : bits[1];
                float x[P][8];
                for (int e = 0; e < P; ++e) unpack8s<kHalf>(u == 0 ? w[0][e] : u == 1 ? w[1][e] : u == 2 ? w[2][e] : w[3][e], x[e]);
                uint32_t packed[P];
                unsigned short sb, zb;
                quantise<kHalf, 8, P>(x, bt, packed, &sb, &zb);
                if (u < 2 ? fits[0] : fits[1]) {
                    unsigned char *base = (u & 1) ? (bt == 4 ? qb.v_hi : qb.v_lo) : (bt == 4 ? qb.k_hi : qb.k_lo);
                    const long long r = u < 2 ? rh[0] : rh[1];
                    for (int e = 0; e < P; ++e) store_codes(base + r * (D * bt / 8), e * 8 + lg, bt, packed[e]);
                    if (lg == 0) reinterpret_cast<uint32_t *>((bt == 4 ? qb.p_hi : qb.p_lo) + r * 4)[u & 1] = (uint32_t)sb | ((uint32_t)zb << 16);
                }
            }
            if (it + 1 < kQuantIters) load(it + 1);
            continue;
        }
        if (lg < 4 && (mine < 2 ? fits[0] : fits[1]))
            reinterpret_cast<uint32_t *>((my_bits == 4 ? qb.p_hi : qb.p_lo) + (mine < 2 ? rh[0] : rh[1]) * 4)[mine & 1] =
                (uint32_t)scale_bits | ((uint32_t)zero_bits << 16);
        uint32_t code[4][P];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float inv = __shfl_sync(0xffffffffu, inv_mine, (lane & ~7) | u);
            const float neg = storage_to_float<kHalf>((unsigned short)(mm[u] >> 16));      // -zero
            const uint32_t mul = bits[u >> 1] == 4 ? 16u : 4u;
#pragma unroll
            for (int i = 0; i < P; ++i) {
                float x[8];
                unpack8s<kHalf>(w[u][i], x);
                uint32_t acc = 0;
#pragma unroll
                for (int e = 7; e >= 0; --e)
                    acc = acc * mul + __float_as_uint(__fadd_rn(__fmul_rn(__fadd_rn(x[e], neg), inv), 12582912.f));
                // (the magic number's bits, 0x4B400000, of eight terms add up to this; 2-bit words keep 16 bits)
                code[u][i] = acc - 0x3F400000u;
            }
        }
        if (it + 1 < kQuantIters) load(it + 1);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int h = u >> 1;
            if (!fits[h]) continue;
            const bool hi4 = bits[h] == 4;
            unsigned char *base = (u & 1) ? (hi4 ? qb.v_hi : qb.v_lo) : (hi4 ? qb.k_hi : qb.k_lo);
#pragma unroll
            for (int i = 0; i < P; ++i) store_codes(base + rh[h] * (hi4 ? D / 2 : D / 4), i * 8 + lg, hi4 ? 4 : 2, code[u][i]);
        }
    }
}

template <bool kHalf, int D>
zipvl_status run_quantize(const LayerArgs &a, const void *k, const void *v, const int32_t *idx,
                          const int32_t *k_dev, int k_max, const QuantBlocks &qb, int32_t *lens_out,
                          int32_t *status_word, cudaStream_t st) {
    const long long pairs = (long long)a.L * a.Hkv;
    const int per_cta = kQuantPairs * kQuantIters;
    const long long grid = (pairs + per_cta - 1) / per_cta;
    const cudaError_t e = launch_dependent(quantize_kv_kernel<kHalf, D>, dim3((unsigned)grid), dim3(kQuantThreads), 0, st,
                                           a, (const unsigned short *)k, (const unsigned short *)v, idx, k_dev, k_max,
                                           qb, lens_out, status_word);
    if (e != cudaSuccess) return fail(ZIPVL_ERR_CUDA, "zipvl_quantize_kv: launch: %s", cudaGetErrorString(e));
    count_launches(1);
    return check_launch("zipvl_quantize_kv");
}

}  // namespace
}  // namespace zipvl

using namespace zipvl;
using namespace zipvl::kvq;

static zipvl_status check_blocks(const char *who, int Hkv, void *k_hi, void *v_hi, void *p_hi, int cap_hi, void *k_lo,
                                 void *v_lo, void *p_lo, int cap_lo, QuantBlocks *qb) {
    if (!k_hi || !v_hi || !p_hi || !k_lo || !v_lo || !p_lo) return fail(ZIPVL_ERR_INVALID_ARG, "%s: NULL cache block", who);
    if (cap_hi < 1 || cap_lo < 1) return fail(ZIPVL_ERR_INVALID_ARG, "%s: capacities %d / %d", who, cap_hi, cap_lo);
    if (((uintptr_t)k_hi | (uintptr_t)v_hi | (uintptr_t)p_hi | (uintptr_t)k_lo | (uintptr_t)v_lo | (uintptr_t)p_lo) & 15u)
        return fail(ZIPVL_ERR_INVALID_ARG, "%s: cache blocks must be 16-byte aligned", who);
    if (Hkv > 1024 / 16) return fail(ZIPVL_ERR_UNSUPPORTED, "%s: more than 64 KV heads", who);
    *qb = QuantBlocks{(unsigned char *)k_hi, (unsigned char *)v_hi, (unsigned char *)k_lo, (unsigned char *)v_lo,
                      (unsigned short *)p_hi, (unsigned short *)p_lo, cap_hi, cap_lo};
    return ZIPVL_OK;
}

extern "C" zipvl_status zipvl_quantize_kv(const zipvl_layer *l, const void *k, const void *v, const int32_t *idx,
                                          const int32_t *k_dev, int32_t k_max, void *k_hi, void *v_hi,
                                          void *params_hi, int32_t cap_hi, void *k_lo, void *v_lo,
                                          void *params_lo, int32_t cap_lo, int32_t *lens_out,
                                          int32_t *status_word, void *stream) {
    const char *who = "zipvl_quantize_kv";
    if (!l) return fail(ZIPVL_ERR_INVALID_ARG, "%s: layer is NULL", who);
    if (l->L < 1 || l->n_kv_heads < 1 || l->n_q_heads < 1 || l->n_q_heads % l->n_kv_heads)
        return fail(ZIPVL_ERR_INVALID_ARG, "%s: L %d heads %d / %d", who, l->L, l->n_q_heads, l->n_kv_heads);
    if ((l->dtype != ZIPVL_BF16 && l->dtype != ZIPVL_F16) || (l->head_dim != 64 && l->head_dim != 128))
        return fail(ZIPVL_ERR_UNSUPPORTED, "%s: dtype %d head_dim %d (16-bit storage, head_dim 64 or 128)", who,
                    l->dtype, l->head_dim);
    const long long ks = l->kv_stride_tok ? l->kv_stride_tok : (long long)l->n_kv_heads * l->head_dim;
    if (ks < (long long)l->n_kv_heads * l->head_dim || ks % 8)
        return fail(ZIPVL_ERR_INVALID_ARG, "%s: token stride %lld", who, ks);
    if (!k || !v || !idx || !k_dev || !lens_out) return fail(ZIPVL_ERR_INVALID_ARG, "%s: NULL pointer", who);
    if (k_max < 1 || k_max > l->L) return fail(ZIPVL_ERR_INVALID_ARG, "%s: k_max = %d not in [1, L]", who, k_max);
    if (((uintptr_t)k | (uintptr_t)v) & 15u) return fail(ZIPVL_ERR_INVALID_ARG, "%s: k, v must be 16-byte aligned", who);
    QuantBlocks qb;
    const zipvl_status s = check_blocks(who, l->n_kv_heads, k_hi, v_hi, params_hi, cap_hi, k_lo, v_lo, params_lo, cap_lo, &qb);
    if (s != ZIPVL_OK) return s;
    LayerArgs a{};
    a.L = l->L; a.Hq = l->n_q_heads; a.Hkv = l->n_kv_heads; a.D = l->head_dim; a.G = a.Hq / a.Hkv;
    a.kv_stride = ks; a.q_stride = (long long)a.Hq * a.D; a.half = (l->dtype == ZIPVL_F16); a.n_seq = 1;
    cudaStream_t st = (cudaStream_t)stream;
    if (a.half) return a.D == 128 ? run_quantize<true, 128>(a, k, v, idx, k_dev, k_max, qb, lens_out, status_word, st)
                                  : run_quantize<true, 64>(a, k, v, idx, k_dev, k_max, qb, lens_out, status_word, st);
    return a.D == 128 ? run_quantize<false, 128>(a, k, v, idx, k_dev, k_max, qb, lens_out, status_word, st)
                      : run_quantize<false, 64>(a, k, v, idx, k_dev, k_max, qb, lens_out, status_word, st);
}

// what the two decode entries check alike
static zipvl_status check_decode_quant(const char *who, const zipvl_decode_desc *d, const void *q, const void *k_new,
                                       const void *v_new, int max_len, const void *out, const void *ws) {
    if (!d) return fail(ZIPVL_ERR_INVALID_ARG, "%s: desc is NULL", who);
    if (d->n_q_heads < 1 || d->n_kv_heads < 1 || d->n_q_heads % d->n_kv_heads)
        return fail(ZIPVL_ERR_INVALID_ARG, "%s: heads %d / %d", who, d->n_q_heads, d->n_kv_heads);
    const int G = d->n_q_heads / d->n_kv_heads;
    if ((d->dtype != ZIPVL_BF16 && d->dtype != ZIPVL_F16) || (d->head_dim != 64 && d->head_dim != 128) ||
        (G != 1 && G != 2 && G != 4))
        return fail(ZIPVL_ERR_UNSUPPORTED, "%s: dtype %d head_dim %d group %d (16-bit storage, head_dim 64 or 128, "
                    "1, 2 or 4 query heads per KV head)", who, d->dtype, d->head_dim, G);
    if (!q || !out || !ws) return fail(ZIPVL_ERR_INVALID_ARG, "%s: NULL pointer", who);
    if ((k_new == NULL) != (v_new == NULL))
        return fail(ZIPVL_ERR_INVALID_ARG, "%s: k_new and v_new must both be given or both NULL", who);
    if (max_len < 1) return fail(ZIPVL_ERR_INVALID_ARG, "%s: max_len = %d", who, max_len);
    if (!(d->softmax_scale >= 0.f) || isinf(d->softmax_scale)) return fail(ZIPVL_ERR_INVALID_ARG, "%s: softmax_scale", who);
    if (((uintptr_t)q | (uintptr_t)out | (uintptr_t)ws | (uintptr_t)k_new | (uintptr_t)v_new) & 15u)
        return fail(ZIPVL_ERR_INVALID_ARG, "%s: tensors must be 16-byte aligned", who);
    return ZIPVL_OK;
}

extern "C" zipvl_status zipvl_decode_quant(const zipvl_decode_desc *d, const void *q, const void *k_new,
                                           const void *v_new, void *k_hi, void *v_hi, void *params_hi,
                                           int32_t cap_hi, void *k_lo, void *v_lo, void *params_lo,
                                           int32_t cap_lo, int32_t *lens, int32_t max_len, void *out, void *ws,
                                           size_t ws_bytes, int32_t *status_word, void *stream) {
    const char *who = "zipvl_decode_quant";
    const zipvl_status sv = check_decode_quant(who, d, q, k_new, v_new, max_len, out, ws);
    if (sv != ZIPVL_OK) return sv;
    if (d->batch != 1) return fail(ZIPVL_ERR_UNSUPPORTED, "%s: batch %d (one request per call)", who, d->batch);
    if (!lens) return fail(ZIPVL_ERR_INVALID_ARG, "%s: NULL pointer", who);
    QuantBlocks qb;
    const zipvl_status s = check_blocks(who, d->n_kv_heads, k_hi, v_hi, params_hi, cap_hi, k_lo, v_lo, params_lo, cap_lo, &qb);
    if (s != ZIPVL_OK) return s;
    const size_t need = (decode_quant_ws_need(1, d->n_q_heads, d->n_kv_heads, d->head_dim, max_len) + 255) & ~(size_t)255;
    if (ws_bytes < need) return fail(ZIPVL_ERR_WORKSPACE, "%s: workspace %zu < %zu", who, ws_bytes, need);
    const float scale = (d->softmax_scale > 0.f ? d->softmax_scale : 1.0f / sqrtf((float)d->head_dim)) * kLog2e;
    return launch_decode_quant(*d, scale, q, k_new, v_new, qb, lens, nullptr, max_len, out, ws, status_word,
                                 (cudaStream_t)stream);
}

extern "C" zipvl_status zipvl_decode_quant_batch(const zipvl_decode_desc *d, const void *q, const void *k_new,
                                                 const void *v_new, const zipvl_quant_cache *caches,
                                                 int32_t max_len, void *out, void *ws, size_t ws_bytes,
                                                 int32_t *status_word, void *stream) {
    const char *who = "zipvl_decode_quant_batch";
    const zipvl_status s = check_decode_quant(who, d, q, k_new, v_new, max_len, out, ws);
    if (s != ZIPVL_OK) return s;
    if (d->batch < 1 || d->batch > 65535) return fail(ZIPVL_ERR_INVALID_ARG, "%s: batch %d not in [1, 65535]", who, d->batch);
    if (d->n_kv_heads > 1024 / 16) return fail(ZIPVL_ERR_UNSUPPORTED, "%s: more than 64 KV heads", who);
    if (!caches || ((uintptr_t)caches & 7u)) return fail(ZIPVL_ERR_INVALID_ARG, "%s: caches is NULL or misaligned", who);
    const size_t need = (decode_quant_ws_need(d->batch, d->n_q_heads, d->n_kv_heads, d->head_dim, max_len) + 255) & ~(size_t)255;
    if (ws_bytes < need) return fail(ZIPVL_ERR_WORKSPACE, "%s: workspace %zu < %zu", who, ws_bytes, need);
    const float scale = (d->softmax_scale > 0.f ? d->softmax_scale : 1.0f / sqrtf((float)d->head_dim)) * kLog2e;
    return launch_decode_quant(*d, scale, q, k_new, v_new, QuantBlocks{}, nullptr, caches, max_len, out, ws, status_word,
                                 (cudaStream_t)stream);
}
