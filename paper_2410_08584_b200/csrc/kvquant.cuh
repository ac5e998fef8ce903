// What the quantiser (kvquant.cu) and the decode step over the mixed-precision cache
// (kvquant_decode.cu) share: the quantiser's arithmetic, the cache blocks of a request.
#pragma once
#include "common.cuh"

namespace zipvl {
namespace kvq {

template <bool kHalf>
__device__ __forceinline__ float storage_round(float x, unsigned short *bits) {
    if (kHalf) {
        const __half h = __float2half_rn(x);
        *bits = __half_as_ushort(h);
        return __half2float(h);
    }
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    *bits = __bfloat16_as_ushort(h);
    return __bfloat162float(h);
}
template <bool kHalf>
__device__ __forceinline__ float storage_to_float(unsigned short bits) {
    return kHalf ? __half2float(__ushort_as_half(bits)) : __bfloat162float(__ushort_as_bfloat16(bits));
}
template <bool kHalf>
__device__ __forceinline__ void unpack8s(const uint4 r, float (&x)[8]) {
    if (kHalf) unpack8h(r, x);
    else unpack8(r, x);
}

// One (row, head) group of kLanes adjacent lanes, 8 P channels per lane: the quantiser's
// parameters (rounded to the storage type) and this lane's codes packed at `bits` each, eight to a word.
template <bool kHalf, int kLanes, int P>
__device__ __forceinline__ void quantise(const float (&x)[P][8], int bits, uint32_t (&packed)[P],
                                         unsigned short *scale_bits, unsigned short *zero_bits) {
    float mn = x[0][0], mx = x[0][0];
#pragma unroll
    for (int i = 0; i < P; ++i)
#pragma unroll
        for (int e = 0; e < 8; ++e) { mn = fminf(mn, x[i][e]); mx = fmaxf(mx, x[i][e]); }
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    const float levels = (float)((1 << bits) - 1);
    const float scale = storage_round<kHalf>(__fdiv_rn(__fsub_rn(mx, mn), levels), scale_bits);
    const float zero = storage_round<kHalf>(mn, zero_bits);
    const float inv = scale > 0.f ? __frcp_rn(scale) : 0.f;             // one correctly rounded reciprocal per row
#pragma unroll
    for (int i = 0; i < P; ++i) {
        packed[i] = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float c = fminf(fmaxf(rintf(__fmul_rn(__fsub_rn(x[i][e], zero), inv)), 0.f), levels);
            packed[i] |= (scale > 0.f ? (uint32_t)c : 0u) << (bits * e);
        }
    }
}

// Writes one lane's eight codes (32 bits at 4 bits each, 16 at 2) and, from the group's first
// lane, the four parameters of the (row, head).
__device__ __forceinline__ void store_codes(unsigned char *row_base, int lane_in_group, int bits, uint32_t packed) {
    if (bits == 4) reinterpret_cast<uint32_t *>(row_base)[lane_in_group] = packed;
    else reinterpret_cast<unsigned short *>(row_base)[lane_in_group] = (unsigned short)packed;
}

struct QuantBlocks {
    unsigned char *k_hi, *v_hi, *k_lo, *v_lo;
    unsigned short *p_hi, *p_lo;      // [rows, Hkv, 4] storage-type bits
    int cap_hi, cap_lo;
};

// The blocks of request b: the call's own (one request) or entry b of the caller's device table.
// A table entry cannot be checked on the host: one with a NULL or misaligned block or a capacity
// below 1 is reported and its request skipped (no append, an output of zeros).
__device__ __forceinline__ bool request_blocks(const zipvl_quant_cache *caches, int b, QuantBlocks &qb,
                                               int32_t *&lens) {
    if (caches == nullptr) return true;
    const zipvl_quant_cache c = caches[b];
    qb = QuantBlocks{(unsigned char *)c.k_hi, (unsigned char *)c.v_hi, (unsigned char *)c.k_lo, (unsigned char *)c.v_lo,
                     (unsigned short *)c.params_hi, (unsigned short *)c.params_lo, c.cap_hi, c.cap_lo};
    lens = c.lens;
    const unsigned long long all = (unsigned long long)c.k_hi | (unsigned long long)c.v_hi | (unsigned long long)c.k_lo |
                                   (unsigned long long)c.v_lo | (unsigned long long)c.params_hi |
                                   (unsigned long long)c.params_lo;
    return c.k_hi && c.v_hi && c.k_lo && c.v_lo && c.params_hi && c.params_lo && c.lens && !(all & 15ull) &&
           !((unsigned long long)c.lens & 3ull) && c.cap_hi >= 1 && c.cap_lo >= 1;
}

// Decode over the cache of one request (caches == nullptr: blocks and lens) or of a batch (device table).
zipvl_status launch_decode_quant(const zipvl_decode_desc &d, float scale_log2, const void *q, const void *k_new,
                                 const void *v_new, const QuantBlocks &qb, int32_t *lens,
                                 const zipvl_quant_cache *caches, int max_len, void *out, void *ws,
                                 int32_t *status_word, cudaStream_t st);

}  // namespace kvq
}  // namespace zipvl
