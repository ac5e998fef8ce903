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

constexpr int kQuantThreads = 256;
constexpr int kQuantIters = 8;      // (token, head) pairs per lane group and CTA

template <bool kHalf, int D>
__global__ void __launch_bounds__(kQuantThreads)
quantize_kv_kernel(LayerArgs a, const unsigned short *__restrict__ k, const unsigned short *__restrict__ v,
                   const int32_t *__restrict__ idx, const int32_t *__restrict__ k_dev, int k_max,
                   QuantBlocks qb, int32_t *__restrict__ lens_out, int32_t *status_word) {
    constexpr int kLanes = D / 8;                 // lanes per (token, head)
    constexpr int kGroups = 32 / kLanes;          // groups per warp
    grid_launch_dependents();
    grid_dependency_wait(k, v, idx, k_dev);       // T and k are the selection's output
    int n = *k_dev;
    if (n > k_max || n < 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) report(status_word, ZIPVL_DEV_CAPACITY);
        n = n < 0 ? 0 : k_max;
    }
    if (n > qb.cap_hi || a.L - n > qb.cap_lo) {
        if (blockIdx.x == 0 && threadIdx.x == 0) report(status_word, ZIPVL_DEV_CAPACITY);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        lens_out[0] = min(n, qb.cap_hi);
        lens_out[1] = min(a.L - n, qb.cap_lo);
    }
    // A CTA takes kPairsPerCta consecutive (token, head) pairs, i.e. a short run of tokens.
    // Where each of those tokens goes -- row i of the 4-bit block if it is T's i-th entry, else
    // row (t - #entries of T below t) of the 2-bit block -- is looked up once per token (a
    // binary search in the ascending list) by the first threads and shared.
    constexpr int kPairsPerIter = (kQuantThreads / 32) * kGroups;
    constexpr int kPairsPerCta = kPairsPerIter * kQuantIters;
    __shared__ int s_row[kPairsPerCta + 2];            // >= 0: hi row; < 0: -(lo row) - 1
    const int lane = threadIdx.x & 31, lg = lane % kLanes;
    const long long n_pairs = (long long)a.L * a.Hkv;
    const long long p0 = (long long)blockIdx.x * kPairsPerCta;
    const int t_first = (int)(p0 / a.Hkv);
    const int t_last = (int)(min(p0 + kPairsPerCta, n_pairs) - 1) / a.Hkv;
    for (int t = t_first + (int)threadIdx.x; t <= t_last; t += kQuantThreads) {
        int lo = 0, hi = n;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (idx[mid] < t) lo = mid + 1; else hi = mid;
        }
        s_row[t - t_first] = (lo < n && idx[lo] == t) ? lo : -(t - lo) - 1;
    }
    __syncthreads();
#pragma unroll 2
    for (int it = 0; it < kQuantIters; ++it) {
        const long long p = p0 + (long long)it * kPairsPerIter + (threadIdx.x >> 5) * kGroups + lane / kLanes;
        const bool live = p < n_pairs;
        const int t = live ? (int)(p / a.Hkv) : t_first, g = live ? (int)(p % a.Hkv) : 0;
        const int where = s_row[t - t_first];
        const bool in_T = where >= 0;
        const int bits = in_T ? 4 : 2;
        const int row = in_T ? where : -where - 1;         // its row in the "hi" / "lo" block
        const bool fits = live && row < (in_T ? qb.cap_hi : qb.cap_lo);
        float xk[8], xv[8];
        if (live) {
            const long long off = (long long)t * a.kv_stride + (long long)g * D + lg * 8;
            unpack8s<kHalf>(*reinterpret_cast<const uint4 *>(k + off), xk);
            unpack8s<kHalf>(*reinterpret_cast<const uint4 *>(v + off), xv);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) { xk[e] = 0.f; xv[e] = 0.f; }
        }
        unsigned short ks, kz, vs, vz;
        const uint32_t ck = quantise8<kHalf, kLanes>(xk, bits, &ks, &kz);
        const uint32_t cv = quantise8<kHalf, kLanes>(xv, bits, &vs, &vz);
        if (fits) {
            const long long rh = (long long)row * a.Hkv + g;
            const int row_bytes = D * bits / 8;
            store_codes((in_T ? qb.k_hi : qb.k_lo) + rh * row_bytes, lg, bits, ck);
            store_codes((in_T ? qb.v_hi : qb.v_lo) + rh * row_bytes, lg, bits, cv);
            if (lg == 0) {
                unsigned short *pp = (in_T ? qb.p_hi : qb.p_lo) + rh * 4;
                *reinterpret_cast<uint2 *>(pp) = make_uint2((uint32_t)ks | ((uint32_t)kz << 16),
                                                            (uint32_t)vs | ((uint32_t)vz << 16));
            }
        }
    }
}

template <bool kHalf, int D>
zipvl_status run_quantize(const LayerArgs &a, const void *k, const void *v, const int32_t *idx,
                          const int32_t *k_dev, int k_max, const QuantBlocks &qb, int32_t *lens_out,
                          int32_t *status_word, cudaStream_t st) {
    const long long pairs = (long long)a.L * a.Hkv;
    const int per_cta = (kQuantThreads / 32) * (32 / (D / 8)) * kQuantIters;
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
    const size_t need = (decode_quant_ws_bytes(1, d->n_q_heads, d->n_kv_heads, d->head_dim, max_len) + 255) & ~(size_t)255;
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
    const size_t need = (decode_quant_ws_bytes(d->batch, d->n_q_heads, d->n_kv_heads, d->head_dim, max_len) + 255) & ~(size_t)255;
    if (ws_bytes < need) return fail(ZIPVL_ERR_WORKSPACE, "%s: workspace %zu < %zu", who, ws_bytes, need);
    const float scale = (d->softmax_scale > 0.f ? d->softmax_scale : 1.0f / sqrtf((float)d->head_dim)) * kLog2e;
    return launch_decode_quant(*d, scale, q, k_new, v_new, QuantBlocks{}, nullptr, caches, max_len, out, ws, status_word,
                                 (cudaStream_t)stream);
}
