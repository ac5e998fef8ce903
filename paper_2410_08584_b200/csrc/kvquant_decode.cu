// Decode step over the mixed-precision cache (Sec. 4.3, Table 3; Algorithm 2, Eq. 4-5): the new
// token's key and value are quantised at 4 bits and appended, and the query attends over all
// rows, dequantised on the fly.
//
// What bounds it: a cached value is 2 or 4 bits, so one SM has to get through about 45 values per
// cycle to keep up with HBM.  With a shift, a conversion and a multiply-add per value and query
// head on the CUDA cores the step took 75 us for six requests of 1.4K-5.9K tokens, 32 heads
// (1.1 TB/s); this kernel and the merge behind it take 36.6 us.  Here the contractions run on the tensor cores
// straight from registers (mma.sync m16n8k16: the operand is unpacked in registers and used once, a tcgen05 operand
// would have to go through shared memory first), and unpacking costs three instructions per four values:
//   - a code c at bit p of a 16-bit half, with the exponent of 2^(10 - p) put above it, is the IEEE half number
//     2^(10 - p) + c; a packed subtraction leaves c - centre, exactly (centre: 8 of 0..15, 2 of 0..3).
//     Left as a subnormal, c * 2^(p - 24), a code needs no subtraction, but the tensor core lines products
//     up by their nominal exponents and cuts off below: such codes lose up to ten bits of the sum (30 us per step instead
//     of 36.6, errors of the fp32 results 10 to 130 times those of a plain fp32 evaluation);
//   - the order of the 16 contraction indices of an MMA is free as long as both operands share it, so a
//     lane takes whole 32-bit words of a row and the halves of a word pair up by themselves;
//   - S = Q K^T: A = codes [16 rows x 16 channels], B = q [16 channels x 8 columns = query heads], q in
//     half precision scaled by a power of two per head (exact for bfloat16 and half values down to
//     2^-28 of the largest; fp32 accumulation);
//   - O = P V: A = codes [16 channels x 16 rows], B = p * v_scale [16 rows x 8 columns], split into
//     two half numbers, w = hi + 2^-11 lo, in columns g and g + 4: 22 bits of a weight down to 2^-22 of
//     the largest, 2^-44 of that below.  The products are exact; p is the one that the denominator adds up;
//   - k^ = (code - centre) * s + (z + centre * s): the second term adds sum(q) times itself to a score and p times itself
//     to every channel of the output.  With the codes centred both sums stay near the results and nothing
//     large has to cancel: the tensor core cuts its sums off instead of rounding them, 2^-23 of the running
//     sum per MMA.  Error of the fp32 results against 64 bits, N(0, 1) keys and values, queries of four sizes,
//     1.4K to 9K rows: 0.2 to 0.9 of that of the plain fp32 evaluation that this kernel replaced.
// A warp owns a chunk of rows of one block of one (request, kv head) (a chunk across both blocks pays the set-up and the first
// loads of either: 1 us of a step of 5); the four warps of a CTA take four
// neighbouring heads of the same rows (their parameters share 32-byte sectors).  32 rows per step: each
// lane evaluates the softmax weight of one row (the query repeated over the columns brings a
// row's score to the lane that needs it), and two more steps are on their way into the warp's own ring.  Nothing is shared between warps: each leaves (m, l, o) for
// decode_merge_kernel.
#include <math.h>

#include <algorithm>

#include "kvquant.cuh"
#include "tc_ptx.cuh"

namespace zipvl {
namespace kvq {
namespace {

constexpr int kWarps = 4, kStages = 3;
constexpr float kLowScale = 2048.f;          // of the low part of a weight, which would be subnormal otherwise
template <int D> struct Ring { static constexpr int kBytes = kStages * (2 * 32 * (D / 2) + 256); };   // per warp, 4-bit rows

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the same with a sum of its own, d = a b + c
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, float c0, float c1, float c2, float c3) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}
// 2^e for e in [-252, 254]: two normal factors
__device__ __forceinline__ float pow2(int e) {
    const int a = e / 2, b = e - a;
    return __int_as_float((a + 127) << 23) * __int_as_float((b + 127) << 23);
}

// The i-th code pair of a 32-bit word of 16-bit halves with BITS-bit codes: codes i and i + 16 / BITS
// of the word (one from each half), less kCentre, as two half numbers.  A code c at bit p of a half's mantissa,
// with the exponent bits of 2^(10 - p) put above it, reads 2^(10 - p) + c; taking 2^(10 - p) + kCentre off is exact.
// Bits 0..9 are the mantissa; the codes above it are moved down first.
template <int BITS>
struct Code {
    static constexpr int kCentre = 1 << (BITS - 1);
    static __device__ __forceinline__ uint32_t pair(uint32_t w, int i) {
        const int p = BITS == 4 ? 4 * (i & 1) : (i < 5 ? 2 * i : 2 * (i - 5));
        const uint32_t moved = (BITS == 4) ? (i >= 2 ? w >> 8 : w) : (i >= 5 ? w >> 10 : w);
        const uint32_t both = 0x00010001u;
        const uint32_t raised = (moved & ((BITS == 4 ? 15u : 3u) * both << p)) | (uint32_t)(25 - p) * (both << 10);
        // 2^(10 - p) + kCentre: its mantissa is kCentre at bit p
        const uint32_t off = ((uint32_t)(25 - p) * (both << 10)) | ((uint32_t)kCentre * both << p);
        uint32_t d;
        asm("sub.f16x2 %0, %1, %2;" : "=r"(d) : "r"(raised), "r"(off));
        return d;
    }
};

// W consecutive 32-bit words (or one 16-bit half, W == 0) of shared memory
template <int W>
__device__ __forceinline__ void load_words(const unsigned char *p, uint32_t (&w)[W < 1 ? 1 : W]) {
    if constexpr (W == 4) {
        const uint4 v = *reinterpret_cast<const uint4 *>(p);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    } else if constexpr (W == 2) {
        const uint2 v = *reinterpret_cast<const uint2 *>(p);
        w[0] = v.x; w[1] = v.y;
    } else if constexpr (W == 1) {
        w[0] = *reinterpret_cast<const uint32_t *>(p);
    } else {
        w[0] = *reinterpret_cast<const unsigned short *>(p);
    }
}

// Running state of a warp.  Query heads: column n of an MMA is head n & (G - 1); a lane evaluates the
// weights of NH heads (first_head, + 1) for NT of the 32 rows of a step.
template <int D, int G>
struct Warp {
    static constexpr int VS = D / 16;        // MMA steps (16 channels each) of a value tile
    static constexpr int NH = G == 1 ? 1 : 2, NT = G == 4 ? 2 : 1;
    float o[VS][4];                          // o[s]: channels base + 2 s (c0, c1) and + 2 s + 1 (c2, c3), columns 2t, 2t + 1
    float m[NH], m_w[NH];                    // integer references of s and of s + exponent(v scale)
    float l[NH], zacc[NH];                   // over this lane's rows only
};
// sum / maximum over the lanes that hold the same heads
template <int G, typename F>
__device__ __forceinline__ float reduce(float x, F f) {
#pragma unroll
    for (int off = G == 4 ? 2 : 1; off < 32; off <<= 1) x = f(x, __shfl_xor_sync(0xffffffffu, x, off));
    return x;
}

// Eq. 4: the new token's key and value of one kv head, quantised at 4 bits and stored as row `row` of the 4-bit
// block: lanes 0 .. D/8 - 1 the key, the next D/8 the value.  Returns this lane's codes and its
// tensor's parameters.
struct NewRow {
    const unsigned short *k, *v;             // [D] of this kv head
    unsigned char *k_hi, *v_hi;              // the block at this kv head's row
    unsigned short *p_hi;
    template <bool kHalf, int D>
    __device__ __forceinline__ uint32_t quantise(int lane, uint32_t &par) const {
        constexpr int kLanes = D / 8;
        const int lg = lane % kLanes, which = lane / kLanes;
        float x[1][8];
        unpack8s<kHalf>(*reinterpret_cast<const uint4 *>(((which & 1) ? v : k) + lg * 8), x[0]);
        unsigned short scale, zero;
        uint32_t codes[1];
        kvq::quantise<kHalf, kLanes, 1>(x, 4, codes, &scale, &zero);
        par = (uint32_t)scale | ((uint32_t)zero << 16);
        if (which < 2) {
            store_codes((which & 1) ? v_hi : k_hi, lg, 4, codes[0]);
            if (lg == 0) reinterpret_cast<uint32_t *>(p_hi)[which] = par;
        }
        return codes[0];
    }
};

// One block of the cache ("hi": BITS = 4, "lo": BITS = 2), rows [r0, r1) of kv head hkv.  fresh: the last of
// them is the appended token, which is not in memory yet.
template <int BITS, bool kHalf, int D, int G>
__device__ __forceinline__ void run_block(Warp<D, G> &st, const unsigned char *kb, const unsigned char *vb,
                                          const unsigned short *pb, int r0, int r1, int Hkv, int hkv,
                                          const unsigned short *__restrict__ q, float scale_log2, unsigned char *ring,
                                          int lane, NewRow *fresh = nullptr) {
    using W = Warp<D, G>;
    constexpr int NH = W::NH, NT = W::NT;
    constexpr int KW = D * BITS / 128;       // 32-bit words of a K row per lane (4 lanes to a row)
    constexpr int VW = D * BITS / 256;       // 32-bit words of a V row per lane (8 lanes to a row); 0: a 16-bit half
    constexpr int VN = VW < 1 ? 1 : VW;
    constexpr int RB = D * BITS / 8;         // bytes of a row
    constexpr int PER = 16 / BITS;           // codes per 16-bit half
    constexpr int KS = D / 16;
    constexpr float kCentre = Code<BITS>::kCentre;
    if (r0 >= r1) return;
    const int g = lane >> 2, t = lane & 3;
    // ---- the warp's ring of kStages steps: 32 rows of K, of V and their parameters each, fetched 16
    // bytes at a time (a row of one head is 16 to 64 contiguous bytes).  V's rows are stored even ones first,
    // so that the reads below (rows 2t of a tile side by side) are free of bank conflicts.
    constexpr int CPR = RB / 16, ROWS = 32 / CPR;            // pieces of a row; rows per copy instruction of the warp
    constexpr int kStage = 2 * 32 * RB + 256;
    const long long row_bytes = (long long)Hkv * RB;
    const int cr = lane / CPR, cc = (lane % CPR) * 16;
    const unsigned char *ksrc = kb + (long long)hkv * RB + (long long)(r0 + cr) * row_bytes + cc;
    const unsigned char *vsrc = vb + (long long)hkv * RB + (long long)(r0 + cr) * row_bytes + cc;
    const unsigned short *psrc = pb + ((long long)(r0 + lane) * Hkv + hkv) * 4;
    const uint32_t ring32 = ptx::smem_u32(ring);
    auto fetch = [&](int step) {
        const int left = (fresh ? r1 - 1 : r1) - r0 - step * 32;   // rows of this step (none: an empty group)
        if (left >= 0) {                                     // (rows past the end become zeros: their weight is zero, but 0 x NaN is not)
            const uint32_t dst = ring32 + (step % kStages) * kStage;
#pragma unroll
            for (int i = 0; i < CPR; ++i) {
                const int r = cr + i * ROWS;
                const uint32_t n = r < left ? 16u : 0u;
                const long long off = (long long)(i * ROWS) * row_bytes;
                ptx::cp_async16(dst + r * RB + cc, n ? ksrc + off : kb, n);
                ptx::cp_async16(dst + 32 * RB + ((r >> 1) + 16 * (r & 1)) * RB + cc, n ? vsrc + off : vb, n);
            }
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst + 64 * RB + lane * 8),
                         "l"(lane < left ? psrc : pb), "r"(lane < left ? 8u : 0u) : "memory");
            ksrc += 32 * row_bytes;
            vsrc += 32 * row_bytes;
            psrc += 32 * Hkv * 4;
        }
        ptx::cp_async_commit();
    };
    // row of this lane's u-th item inside a step: the accumulator rows it holds
    auto item_row = [&](int u) { return G == 4 ? 16 * u + 8 * (t >> 1) + g : 8 * t + g; };
#pragma unroll
    for (int i = 0; i < kStages - 1; ++i) fetch(i);
    // ---- the query as B operand: head g & (G-1)'s channels D/4 * t ..., paired like the codes of K's words
    uint32_t qf[KS][2];
    float k_factor[NH], q_sum[NH];           // dot * k_factor = scale_log2 * <q, code - centre>; scale_log2 * sum(q)
    {
        float mx = 0.f, sum = 0.f;
        float x[D / 4];
#pragma unroll
        for (int c = 0; c < D / 4; c += 8) {
            float y[8];
            unpack8s<kHalf>(*reinterpret_cast<const uint4 *>(q + (g & (G - 1)) * D + t * (D / 4) + c), y);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                x[c + e] = y[e];
                mx = fmaxf(mx, fabsf(y[e]));
                sum += y[e];
            }
        }
#pragma unroll
        for (int off = 1; off < 4; off <<= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            sum += __shfl_xor_sync(0xffffffffu, sum, off);
        }
        const int e = (int)(__float_as_uint(mx) >> 23) - 127;
        const int up = e >= 127 ? 0 : 14 - max(e, -86);      // largest |q| * 2^up in [2^14, 2^15)
        const float f = pow2(up);
#pragma unroll
        for (int j = 0; j < KW; ++j)
#pragma unroll
            for (int s = 0; s < PER / 2; ++s)
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const int i = 2 * s + b, c = j * 2 * PER + i;
                    qf[j * (PER / 2) + s][b] = pack_half2(x[c] * f, x[c + PER] * f);
                }
        const float kf = pow2(-up) * scale_log2, qs = sum * scale_log2;
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const int src = 4 * (h + (G == 4 ? 2 * (t & 1) : 0));
            k_factor[h] = __shfl_sync(0xffffffffu, kf, src);
            q_sum[h] = __shfl_sync(0xffffffffu, qs, src);
        }
    }
    // weights: columns g < 4 take the hi part of head g, columns g + 4 the lo part; others are zero (the sign
    // of a weight, replicated)
    const uint32_t pick = (g & 3) >= G ? 0x9999u : g < 4 ? 0x5410u : 0x7632u;

    uint32_t new_codes = 0, new_par = 0;
    if (fresh) new_codes = fresh->quantise<kHalf, D>(lane, new_par);
    const int n_steps = (r1 - r0 + 31) / 32;
    for (int step = 0; step < n_steps; ++step) {
        ptx::cp_async_wait<kStages - 2>();
        __syncwarp();                        // the step has landed for all lanes, and all are done with the one before
        fetch(step + kStages - 1);
        unsigned char *buf = ring + (step % kStages) * kStage;
        if (fresh && step == n_steps - 1) {  // the appended row, the block's last, from this warp's registers
            const int r = (r1 - 1 - r0) & 31, which = lane / (D / 8);
            if (which < 2) {
                const int at = which ? (32 + (r >> 1) + 16 * (r & 1)) * RB : r * RB;
                *reinterpret_cast<uint32_t *>(buf + at + (lane % (D / 8)) * 4) = new_codes;
                if (lane % (D / 8) == 0) *reinterpret_cast<uint32_t *>(buf + 64 * RB + r * 8 + which * 4) = new_par;
            }
            __syncwarp();
        }
        const int base = r0 + step * 32;
        uint32_t kw[2][2][KW];
#pragma unroll
        for (int u = 0; u < 4; ++u) load_words<KW>(buf + (g + 8 * u) * RB + t * (KW * 4), kw[u >> 1][u & 1]);
        // ---- scores of 2 x 16 rows, two chains of MMAs side by side
        float c[2][4];
#pragma unroll
        for (int j = 0; j < KW; ++j)
#pragma unroll
            for (int s = 0; s < PER / 2; ++s) {
                const int i = j * (PER / 2) + s;
#pragma unroll
                for (int tile = 0; tile < 2; ++tile) {
                    const uint32_t w0 = kw[tile][0][j], w1 = kw[tile][1][j];
                    const uint32_t a[4] = {Code<BITS>::pair(w0, 2 * s), Code<BITS>::pair(w1, 2 * s),
                                           Code<BITS>::pair(w0, 2 * s + 1), Code<BITS>::pair(w1, 2 * s + 1)};
                    if (i == 0) mma16816(c[tile], a, qf[i][0], qf[i][1], 0.f, 0.f, 0.f, 0.f);
                    else mma16816(c[tile], a, qf[i][0], qf[i][1]);
                }
            }
        uint2 pr[NT];
#pragma unroll
        for (int u = 0; u < NT; ++u) pr[u] = *reinterpret_cast<const uint2 *>(buf + 64 * RB + item_row(u) * 8);
        // ---- this lane's weights
        float sc[NT][NH], ev[NT], fv[NT], vc[NT];
        bool grow = false;
#pragma unroll
        for (int u = 0; u < NT; ++u) {
            const float ks = storage_to_float<kHalf>((unsigned short)(pr[u].x & 0xffffu));
            const float kz = fmaf(kCentre, ks, storage_to_float<kHalf>((unsigned short)(pr[u].x >> 16)));
            const float vs = storage_to_float<kHalf>((unsigned short)(pr[u].y & 0xffffu));
            // v scale = fv * 2^ev, fv in [1, 2) (a zero or subnormal scale: ev = -126)
            const uint32_t e = __float_as_uint(vs) >> 23;
            ev[u] = (float)(int)max(e, 1u) - 127.f;
            fv[u] = e - 1u < 254u ? __uint_as_float((__float_as_uint(vs) & 0x7fffffu) | 0x3f800000u)
                                  : (e == 0u ? vs * 8.507059e37f : vs);
            vc[u] = fmaf(kCentre, vs, storage_to_float<kHalf>((unsigned short)(pr[u].y >> 16)));
            const bool in = base + item_row(u) < r1;
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                float dot;
                if (G == 4) dot = t < 2 ? c[u][h] : c[u][2 + h];
                else dot = t < 2 ? (t == 0 ? c[0][h] : c[0][2 + h]) : (t == 2 ? c[1][h] : c[1][2 + h]);
                sc[u][h] = in ? fmaf(ks * k_factor[h], dot, kz * q_sum[h]) : -INFINITY;
                grow |= sc[u][h] > st.m[h] + 6.f || sc[u][h] + ev[u] > st.m_w[h] + 6.f;
            }
        }
        // References move only when a step outgrows them by 2^6 (or on the first one), and by whole
        // powers of two: p = 2^(s - m), weights 2^(s + ev - m_w) stay below 2^7.
        if (__any_sync(0xffffffffu, grow)) {
            float fw[2] = {1.f, 1.f};
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                float mx = sc[0][h], mxw = sc[0][h] + ev[0];
                if (NT == 2) { mx = fmaxf(mx, sc[NT - 1][h]); mxw = fmaxf(mxw, sc[NT - 1][h] + ev[NT - 1]); }
                mx = fmaxf(st.m[h], ceilf(reduce<G>(mx, fmaxf)));
                mxw = fmaxf(st.m_w[h], ceilf(reduce<G>(mxw, fmaxf)));
                const float f = mx == -INFINITY ? 1.f : fast_exp2(st.m[h] - mx);
                fw[h] = mxw == -INFINITY ? 1.f : fast_exp2(st.m_w[h] - mxw);
                st.l[h] *= f;
                st.zacc[h] *= f;
                st.m[h] = mx;
                st.m_w[h] = mxw;
            }
            // (columns 2t and 2t + 1 of the accumulators are this lane's own heads)
#pragma unroll
            for (int s = 0; s < W::VS; ++s) {
                st.o[s][0] *= fw[0]; st.o[s][1] *= fw[NH - 1]; st.o[s][2] *= fw[0]; st.o[s][3] *= fw[NH - 1];
            }
        }
        uint32_t packed[NT][NH];             // (hi, lo) of a weight
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const float ref = st.m[h] == -INFINITY ? 0.f : st.m[h], ref_w = (st.m_w[h] == -INFINITY ? 0.f : st.m_w[h]) - 8.f;
#pragma unroll
            for (int u = 0; u < NT; ++u) {
                const float p = fast_exp2(sc[u][h] - ref);
                st.l[h] += p;
                st.zacc[h] = fmaf(p, vc[u], st.zacc[h]);
                // p * v scale as a multiple of 2^ref_w, below 2^15 (a power of two of its own, not an exponential of
                // its own: numerator and denominator of the softmax share the rounding of p)
                const float up = ev[u] + (ref - ref_w);
                float w = p * fv[u] * fast_exp2(fminf(up, 126.f));
                if (up > 126.f) w *= fast_exp2(fminf(up - 126.f, 126.f));
                const float hi = __half2float(__float2half_rn(w));
                packed[u][h] = pack_half2(w, (w - hi) * kLowScale);
            }
        }
#pragma unroll
        for (int tile = 0; tile < 2; ++tile) {
            uint32_t b[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {    // rows 2t, 2t + 1 (k = 0) and 2t + 8, 2t + 9 of the tile
                uint32_t x[2];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int src = 4 * (2 * t + r) + (G == 4 ? 2 * k + ((g >> 1) & 1) : 2 * tile + k);
                    const int u = G == 4 ? tile : 0;
                    x[r] = __shfl_sync(0xffffffffu, packed[u % NT][0], src);
                    if (NH == 2) {
                        const uint32_t y = __shfl_sync(0xffffffffu, packed[u % NT][NH - 1], src);
                        if (g & 1) x[r] = y;
                    }
                }
                b[k] = __byte_perm(x[0], x[1], pick);
            }
            uint32_t vw[4][VN];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                load_words<VW>(buf + 32 * RB + (8 * tile + t + 4 * (u >> 1) + 16 * (u & 1)) * RB + g * (VW ? VW * 4 : 2), vw[u]);
            // ---- O += (codes - kCentre)^T w: per MMA two channels of this lane's channel group, 16 rows
            // (pairs of rows 2t, 2t + 1 and 2t + 8, 2t + 9 share a word after a byte permutation)
#pragma unroll
            for (int j = 0; j < VN; ++j)
#pragma unroll
                for (int half = 0; half < (VW ? 2 : 1); ++half) {
                    const uint32_t x0 = __byte_perm(vw[0][j], vw[1][j], half ? 0x7632 : 0x5410);
                    const uint32_t x1 = __byte_perm(vw[2][j], vw[3][j], half ? 0x7632 : 0x5410);
#pragma unroll
                    for (int s = 0; s < PER / 2; ++s) {
                        const uint32_t a[4] = {Code<BITS>::pair(x0, 2 * s), Code<BITS>::pair(x0, 2 * s + 1),
                                               Code<BITS>::pair(x1, 2 * s), Code<BITS>::pair(x1, 2 * s + 1)};
                        mma16816(st.o[(j * 2 + half) * (PER / 2) + s], a, b[0], b[1]);
                    }
                }
        }
    }
    ptx::cp_async_wait<0>();
    __syncwarp();
}

template <bool kHalf, int D, int G>
__global__ void __launch_bounds__(kWarps * 32, 4)
decode_quant_kernel(int Hq, int Hkv, float scale_log2, const unsigned short *__restrict__ q,
                    const unsigned short *__restrict__ k_new, const unsigned short *__restrict__ v_new, QuantBlocks qb,
                    int32_t *lens, const zipvl_quant_cache *__restrict__ caches, int max_len, int chunk,
                    int n_chunks, float *__restrict__ ws, int *__restrict__ lens_ws, int32_t *status_word) {
    grid_launch_dependents();
    grid_dependency_wait(q, k_new, v_new, lens, caches, qb.k_hi, qb.v_hi, qb.k_lo, qb.v_lo, qb.p_hi, qb.p_lo);
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char *ring = smem + (threadIdx.x >> 5) * Ring<D>::kBytes;
    const int b = blockIdx.z, lane = threadIdx.x & 31;
    const int hkv = blockIdx.y * kWarps + (threadIdx.x >> 5);
    const bool first = blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0;
    const bool blocks_ok = request_blocks(caches, b, qb, lens);
    const int old_hi = blocks_ok ? lens[0] : 0, n_lo = blocks_ok ? lens[1] : 0;
    const bool room = blocks_ok && k_new != nullptr && old_hi >= 0 && old_hi < qb.cap_hi;
    if (first && blocks_ok && k_new != nullptr && !room) report(status_word, ZIPVL_DEV_CAPACITY);
    int n_hi = old_hi + (room ? 1 : 0);
    int total = n_hi + n_lo;
    if (!blocks_ok || n_hi < 0 || n_lo < 0 || n_hi > qb.cap_hi || n_lo > qb.cap_lo) {
        if (first) report(status_word, ZIPVL_DEV_BAD_INDEX);
        total = 0;
        n_hi = 0;
    }
    if (total > max_len) {
        if (first) report(status_word, ZIPVL_DEV_CAPACITY);
        total = max_len;
    }
    if (first) {                             // for the merge kernel, which writes the length
        lens_ws[2 * b] = old_hi + 1;
        lens_ws[2 * b + 1] = room ? 1 : 0;
    }
    if (hkv >= Hkv) return;
    // a chunk lies in one block: first those of the 4-bit rows, then those of the 2-bit ones
    const int rows4 = min(n_hi, total), chunks4 = (rows4 + chunk - 1) / chunk;
    const bool in4 = (int)blockIdx.x < chunks4;
    const int r0 = ((int)blockIdx.x - (in4 ? 0 : chunks4)) * chunk, r1 = min(in4 ? rows4 : total - rows4, r0 + chunk);
    float *dst = ws + (((long long)b * Hq + hkv * G) * n_chunks + blockIdx.x) * (D + 2);
    const long long head_pitch = (long long)n_chunks * (D + 2);
    // the appended row belongs to the chunk that ends with it (or, beyond the rows that count, to the last)
    const long long rh = (long long)old_hi * Hkv + hkv;
    NewRow fresh = {k_new + ((long long)b * Hkv + hkv) * D, v_new + ((long long)b * Hkv + hkv) * D, qb.k_hi + rh * (D / 2),
                    qb.v_hi + rh * (D / 2), qb.p_hi + rh * 4};
    const bool mine = room && in4 && old_hi >= r0 && old_hi < r1;
    if (room && old_hi >= rows4 && (int)blockIdx.x == n_chunks - 1) {
        uint32_t par;
        fresh.quantise<kHalf, D>(lane, par);
    }
    if (r0 >= r1) {
        if (lane < G) {                      // a chunk past the cache: an empty partial
            dst[lane * head_pitch] = -INFINITY;
            dst[lane * head_pitch + 1] = 0.f;
        }
        return;
    }
    const int g = lane >> 2, t = lane & 3;
    const unsigned short *qh = q + ((long long)b * Hq + hkv * G) * D;
    Warp<D, G> st;
    constexpr int VS = Warp<D, G>::VS, NH = Warp<D, G>::NH;
#pragma unroll
    for (int s = 0; s < VS; ++s)
#pragma unroll
        for (int e = 0; e < 4; ++e) st.o[s][e] = 0.f;
#pragma unroll
    for (int h = 0; h < NH; ++h) { st.m[h] = -INFINITY; st.m_w[h] = -INFINITY; st.l[h] = 0.f; st.zacc[h] = 0.f; }
    if (in4)
        run_block<4, kHalf, D, G>(st, qb.k_hi, qb.v_hi, qb.p_hi, r0, r1, Hkv, hkv, qh, scale_log2, ring, lane, mine ? &fresh : nullptr);
    else
        run_block<2, kHalf, D, G>(st, qb.k_lo, qb.v_lo, qb.p_lo, r0, r1, Hkv, hkv, qh, scale_log2, ring, lane);

    // ---- this chunk's (m, l, o): o = sum p * (code * v_scale + v_zero).  Lane t < 2 holds the hi parts of
    // heads 2t, 2t + 1, lane t + 2 their lo parts.
    auto add = [](float x, float y) { return x + y; };
#pragma unroll
    for (int h = 0; h < NH; ++h) {
        const float l = reduce<G>(st.l[h], add), z = reduce<G>(st.zacc[h], add);
        // from the accumulators' reference (and 2^8) to p's
        const float up = fast_exp2(st.m_w[h] - st.m[h] - 8.f);
        const bool write = t < 2 && 2 * t + h < G;
        float *row = dst + (2 * t + h) * head_pitch;
        if (write && g == 0) *reinterpret_cast<float2 *>(row) = make_float2(st.m[h], l);
#pragma unroll
        for (int s = 0; s < VS; ++s) {
            const float a = fmaf(__shfl_xor_sync(0xffffffffu, st.o[s][h], 2), 1.f / kLowScale, st.o[s][h]);
            const float c = fmaf(__shfl_xor_sync(0xffffffffu, st.o[s][2 + h], 2), 1.f / kLowScale, st.o[s][2 + h]);
            if (write) *reinterpret_cast<float2 *>(row + 2 + g * (D / 8) + 2 * s) = make_float2(fmaf(a, up, z), fmaf(c, up, z));
        }
    }
}

// Rows per warp, in whole steps.  An SM holds 16 of these warps.  One or two requests: at most one wave of
// them even if every request has max_len rows; a larger batch is ragged, and cutting it finer keeps the SMs busy when the
// shorter requests leave their last chunks empty.  24 against 14 warps per SM, the time over nine shapes of three head
// counts and lengths: 1.00 for one and two requests, 0.95 for three, 0.98, 0.94, 0.93, 0.95 for four, five, six and eight.
// With few heads neither fills the chip, and what counts is the number of partial results to merge: 64 at most
// (one request of 12000 rows, 4 heads of 64: 13.1 us at 375 chunks, 10.1 at 256, 9.2 at 128 and 64; 6 requests of
// 12000 rows, one head of 128: 19.1, 14.1, 12.3, 11.8; over 154 shapes 64 is 2% ahead of 128 and 256).
constexpr int kMaxChunks = 64;
constexpr int wave_warps(int B) { return B <= 2 ? 14 : 24; }
int quant_chunk(int B, int Hkv, int max_len) {
    const long long warps = 148 * wave_warps(B), rows = ((long long)B * Hkv * max_len + warps - 1) / warps;
    return (int)std::min<long long>(512, std::max<long long>(32, (std::max<long long>(rows, (max_len + kMaxChunks - 1) / kMaxChunks) + 31) / 32 * 32));
}
// (one more than the rows fill: either block ends with a part of a chunk)
int quant_chunks(int max_len, int chunk) { return (max_len + chunk - 1) / chunk + 1; }
// Chunks times query heads of all requests, for this problem or any smaller batch or length (see quant_chunk)
size_t quant_slots(int B, int Hq, int Hkv, int max_len) {
    const auto cut = [&](size_t rows) { return (size_t)B * Hq * ((max_len + rows - 1) / rows); };
    return std::max(cut(512), std::min(cut(32), (size_t)(Hq / Hkv) * 148 * wave_warps(B) + (size_t)B * Hq)) + (size_t)B * Hq;
}
size_t quant_partial_bytes(int B, int Hq, int Hkv, int D, int max_len) {
    const int chunk = quant_chunk(B, Hkv, max_len);
    return align256((size_t)B * Hq * quant_chunks(max_len, chunk) * (D + 2) * sizeof(float));
}

template <bool kHalf, int D>
zipvl_status run(const zipvl_decode_desc &d, float scale_log2, const void *q, const void *k_new,
                 const void *v_new, const QuantBlocks &qb, int32_t *lens, const zipvl_quant_cache *caches, int max_len,
                 void *out, void *ws, int32_t *status_word, cudaStream_t st) {
    const int Hq = d.n_q_heads, Hkv = d.n_kv_heads, G = Hq / Hkv, B = d.batch;
    const int chunk = quant_chunk(B, Hkv, max_len), n_chunks = quant_chunks(max_len, chunk);
    float *wsf = reinterpret_cast<float *>(ws);
    int *lens_ws = reinterpret_cast<int *>(reinterpret_cast<char *>(ws) + quant_partial_bytes(B, Hq, Hkv, D, max_len));
    auto *kernel = G == 1 ? decode_quant_kernel<kHalf, D, 1> : G == 2 ? decode_quant_kernel<kHalf, D, 2> : decode_quant_kernel<kHalf, D, 4>;
    constexpr int smem = kWarps * Ring<D>::kBytes;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return fail(ZIPVL_ERR_CUDA, "zipvl_decode_quant: smem opt-in: %s", cudaGetErrorString(e));
    e = launch_dependent(kernel, dim3(n_chunks, (Hkv + kWarps - 1) / kWarps, B), dim3(kWarps * 32), smem, st,
                                           Hq, Hkv, scale_log2, (const unsigned short *)q, (const unsigned short *)k_new,
                                           (const unsigned short *)v_new, qb, lens, caches, max_len, chunk, n_chunks, wsf,
                                           lens_ws, status_word);
    if (e != cudaSuccess) return fail(ZIPVL_ERR_CUDA, "zipvl_decode_quant: launch: %s", cudaGetErrorString(e));
    count_launches(1);
    return launch_decode_merge(d.dtype, D, Hq, B, n_chunks, wsf, lens_ws, lens, out, st, caches);
}

}  // namespace

zipvl_status launch_decode_quant(const zipvl_decode_desc &d, float scale_log2, const void *q, const void *k_new,
                                 const void *v_new, const QuantBlocks &qb, int32_t *lens,
                                 const zipvl_quant_cache *caches, int max_len, void *out, void *ws,
                                 int32_t *status_word, cudaStream_t st) {
    if (d.dtype == ZIPVL_F16)
        return d.head_dim == 128 ? run<true, 128>(d, scale_log2, q, k_new, v_new, qb, lens, caches, max_len, out, ws, status_word, st)
                                 : run<true, 64>(d, scale_log2, q, k_new, v_new, qb, lens, caches, max_len, out, ws, status_word, st);
    return d.head_dim == 128 ? run<false, 128>(d, scale_log2, q, k_new, v_new, qb, lens, caches, max_len, out, ws, status_word, st)
                             : run<false, 64>(d, scale_log2, q, k_new, v_new, qb, lens, caches, max_len, out, ws, status_word, st);
}

}  // namespace kvq

size_t decode_quant_ws_need(int B, int Hq, int Hkv, int D, int max_len) {
    return kvq::quant_partial_bytes(B, Hq, Hkv, D, max_len) + (size_t)2 * B * sizeof(int);
}
size_t decode_quant_ws_bytes(int B, int Hq, int Hkv, int D, int max_len) {
    return align256(kvq::quant_slots(B, Hq, Hkv, max_len) * (D + 2) * sizeof(float)) + (size_t)2 * B * sizeof(int);
}

}  // namespace zipvl
