// Decode over the kept cache (Algorithm 2; Eq. 4 append, Eq. 5 attention of one query
// token over the whole cache).  16-bit storage, head_dim 64, 96 or 128, 1 to 32 query heads per
// key/value head, contiguous and paged caches.
//
// What bounds it: HBM, as long as a cached row costs few instructions.  With G query heads sharing a
// row the CUDA cores need 2 G multiply-adds per element and fall behind from G = 3 on, so the
// contractions run on the tensor cores -- with mma.sync m16n8k16, whose operands are registers: the
// rows go from memory to the registers that feed the MMA, no shared memory, no barrier, no role for
// any warp but its own loop.  (A tcgen05 version with the G rows in a 128-row tile did 16 times
// the arithmetic for G = 7 and needed a ring, producers and an issuer: 4.2 TB/s sustained on 16 requests of
// 6K-30K rows, 28 heads on 4, against 5.6 here; one request of 732 rows: 8.6 -> 7.1 us.)
//   - S = K Q^T: A = 16 cached rows x 16 channels, B = 16 channels x 8 query heads.  The order
//     of the 16 contraction indices is free as long as both operands share it, so a lane loads 16
//     contiguous bytes of a row (four lanes 64) and they are the A registers of two MMAs;
//   - O^T = V^T P: A = 16 channels x 16 rows.  A lane loads 16 bytes (eight lanes 128) of rows 2t, 2t + 1, 2t + 8
//     and 2t + 9, two byte permutations pair up the rows of a channel, and the channels of a word are
//     rows g and g + 8 of the MMA.  P comes from S's accumulators by two 8 x 8 transpositions.
//     One query head per kv head (the CUDA cores keep up there, but their kernel needs more rows
//     in flight per step to do so): the head fills all columns of S, and its weight goes into
//     three columns as three numbers of eight bits, which is all 24 bits of it.  IEEE half ends at 2^-24, so there
//     the weights are multiplied up by 2^7, the second and third part by 2^8 and 2^16 more, and each part
//     is of what the one before it left: 24 bits down to 2^-23 and 2^-48 below, the largest weight being 1 or more.
//     The tensor core cuts its sums off instead of rounding them, so for one head, whose results are fp32 sums
//     of fp32 weights, every MMA starts a sum of its own and these are added in fp32.  Errors of the fp32 results against
//     64 bits, relative to the CUDA-core kernel's: 0.6 to 1.2 on N(0, 1) data at four query scales, up to 3.5
//     (1.7e-7 of the result) where the values share an offset; with running sums in the tensor core 1 to 57.
//     No slower: a step waits for the cache's rows (16 requests of 3K-24K rows: 520 us, one request of
//     2307 rows, eight layers: 97.5 us, either way);
//   - a lane holds the scores of two heads for two rows; running maxima move only when a tile outgrows them
//     (by 2^32, 2^8 for IEEE half: P is rounded to the storage type), so there is no reduction per tile;
//   - K of the warp's next tile is fetched as soon as S is computed, V as soon as O is: 16 loads of 16
//     bytes per lane in flight.  The warps of a CTA take every fourth tile of its chunk and are merged
//     through shared memory at the end; the chunks by decode_merge_kernel.
//   - more than eight heads: two to four tiles of eight, whose chains, votes and merges run side by side.  Two
//     CTAs fit an SM then, and their eight warps hold too few loads for HBM's latency: the rows of the step after
//     the next are fetched into L2 (0.93 of the time over 68 shapes of more than a wave, 0.87 to 1.01; 0.99 over 112 in
//     one wave).  From 25 heads of 128 channels on the warps no longer hide each other's latencies: 64 requests of
//     10K-20K rows on 2 kv heads, 24 heads 167 us (5.9 TB/s), 34 heads 188, 64 heads 246.
// Grid x is the kv head: the CTAs of one chunk run side by side and read whole rows of the cache together.
// A tile is 16 rows, chunks start at multiples of 16 and pages are at least 16 rows, so a paged
// cache costs one table look-up per tile.
#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace zipvl {
namespace {

using namespace ptx;

constexpr int kWarps = 4;         // (and of head tiles at most: each warp brings one into shared memory)
// rows of a CTA: the fewer CTAs share a row (kv heads), the more a partial weighs against the rows behind it.  Over 55 shapes
// of six head counts, half of these take 0.98 of the time (0.77 where a batch then fills its last wave, 1.09 on long
// caches), twice of them 1.01 (0.80 to 1.29).  (More than eight heads: from 512 on, see decode_mma_chunk.)
constexpr int max_rows(int G, int D) { return G > 8 ? 1536 : D == 64 ? 768 : G == 1 ? 1024 : 1536; }
constexpr int min_large(int G, int D) { return G > 8 ? 512 : max_rows(G, D); }
// (their registers; NT = 0: one query head per kv head, which spills at six CTAs of 64 channels: 16 requests of 10K-20K rows,
// 16 heads, paged 183 us against 157 at five)
__host__ __device__ constexpr int ctas_per_sm(int NT, int D) { return NT > 1 ? 2 : D == 64 ? (NT ? 6 : 5) : 3; }

template <bool kHalf>
__device__ __forceinline__ void mma16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    if (kHalf)
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                     : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
    else
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                     : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// d = a b, a sum of its own
template <bool kHalf>
__device__ __forceinline__ void mma16_new(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    if (kHalf)
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                     : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
    else
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                     : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ uint32_t transpose8(uint32_t x) {
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
// x to its leading eight bits, as the storage type holds them (a subnormal half holds fewer)
template <bool kHalf>
__device__ __forceinline__ float leading_bits(float x) {
    if (kHalf) {     // (2^-24 at least, of a positive number: a weight may meet an infinite value)
        const float y = __half2float(__float2half_rn(__uint_as_float(__float_as_uint(x) & 0xffff0000u)));
        return x > 0.f ? fmaxf(y, 5.9604645e-8f) : y;
    }
    return __bfloat162float(__float2bfloat16_rn(x));
}
template <int W>
__device__ __forceinline__ void load_row(const void *p, uint32_t (&w)[W]) {
    if constexpr (W == 4)
        asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(p));
    else
        asm volatile("ld.global.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "l"(p));
}
template <int W>
__device__ __forceinline__ void store_row(void *p, const uint32_t (&w)[W]) {
    if constexpr (W == 4) *reinterpret_cast<uint4 *>(p) = make_uint4(w[0], w[1], w[2], w[3]);
    else *reinterpret_cast<uint2 *>(p) = make_uint2(w[0], w[1]);
}

__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

struct DmArgs {
    int Hq, Hkv, max_len, chunk, n_chunks;
    float scale_log2;
    const char *q, *k_new, *v_new;
    char *k_cache, *v_cache;
    const int64_t *cache_off;
    PageArgs pg;
    const int32_t *capacity;
    int32_t *seq_lens;
    float *ws;
    int *lens;
    int32_t *status_word;
};

// NT: tiles of eight query heads; 0: one head per kv head
template <bool kHalf, bool kPaged, int D, int NT_>
__global__ void __launch_bounds__(kWarps * 32, ctas_per_sm(NT_, D))
decode_mma_kernel(DmArgs a) {
    constexpr bool kOne = NT_ == 0;
    constexpr int NT = kOne ? 1 : NT_;
    constexpr int KJ = D / 32;                       // 16-byte pieces of a K row per lane
    constexpr int VW = D % 64 ? 2 : 4;               // 32-bit words of a V piece
    constexpr int VJ = D / (16 * VW);                // pieces of a V row per lane
    constexpr int VS = VJ * VW;                      // MMAs per tile and head tile
    constexpr int RB = D * 2;                        // bytes of a row of one head
    constexpr float kGrow = kHalf ? 8.f : 32.f;
    // the three parts of a single head's weight, of eight bits each: multiplied up in IEEE half
    constexpr float kTop = kHalf ? 128.f : 1.f, kStep = kHalf ? 256.f : 1.f;
    constexpr int ET = NT > 1 ? 2 : 1;               // head tiles merged at a time
    __shared__ float sm_o[kWarps][8 * ET][D];
    __shared__ float sm_m[kWarps][8 * ET], sm_l[kWarps][8 * ET];
    __shared__ uint4 sm_q[NT > 2 ? NT * 8 * (D / 8) : 1];

    grid_launch_dependents();
    grid_dependency_wait(a.q, a.k_new, a.v_new, a.k_cache, a.v_cache, a.cache_off, a.capacity, a.seq_lens, a.pg.table);
    const int b = blockIdx.z, hkv = blockIdx.x, part = blockIdx.y, G = a.Hq / a.Hkv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const bool first = blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0;

    // ---- the query heads as B operand: head g's channels 32 j + 8 t .. + 7 are MMAs 2 j and 2 j + 1
    const char *qb = a.q + ((long long)b * a.Hq + (long long)hkv * G) * RB;
    auto q_piece = [&](int nt, int j) -> uint4 {
        const int h = kOne ? 0 : nt * 8 + g;
        return h < G ? *reinterpret_cast<const uint4 *>(qb + h * RB + j * 64 + t * 16) : make_uint4(0, 0, 0, 0);
    };
    uint4 qr[NT > 2 ? 1 : NT][KJ];
    if (NT <= 2) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int j = 0; j < KJ; ++j) qr[NT > 2 ? 0 : nt][j] = q_piece(nt, j);
    } else if (warp < NT) {
#pragma unroll
        for (int j = 0; j < KJ; ++j) sm_q[(warp * KJ + j) * 32 + lane] = q_piece(warp, j);
    }

    // A request whose length is negative or beyond its capacity, or whose cache offset breaks the
    // 16-byte alignment of the row loads, is skipped as a whole and reported.
    const int old_len = a.seq_lens[b], cap = a.capacity[b];
    const long long coff = kPaged ? 0ll : a.cache_off[b] * 2;
    const bool bad = old_len < 0 || old_len > cap || (coff & 15) != 0;
    if (bad && first) report(a.status_word, ZIPVL_DEV_BAD_INDEX);
    const bool appended = !bad && a.k_new != nullptr && old_len < cap;
    if (a.k_new != nullptr && !bad && !appended && first) report(a.status_word, ZIPVL_DEV_CAPACITY);
    int len = bad ? 0 : old_len + (appended ? 1 : 0);
    if (len > a.max_len) {
        if (first) report(a.status_word, ZIPVL_DEV_CAPACITY);
        len = a.max_len;
    }
    if (first) {
        a.lens[2 * b] = len;
        a.lens[2 * b + 1] = appended ? 1 : 0;
    }
    const int c0 = part * a.chunk, c1 = min(len, c0 + a.chunk);
    float *dst = a.ws + (((long long)b * a.Hq + hkv * G) * a.n_chunks + part) * (D + 2);
    const long long head_pitch = (long long)a.n_chunks * (D + 2);
    if (c0 >= len) {
        if ((int)threadIdx.x < G) {                  // a chunk past the request's length: an empty partial
            dst[threadIdx.x * head_pitch] = -INFINITY;
            dst[threadIdx.x * head_pitch + 1] = 0.f;
        }
        return;
    }
    const int new_row = appended ? old_len : -1;     // (== len when max_len cuts it off: never loaded)
    const long long pitch = (long long)a.Hkv * RB;
    const char *kb = a.k_cache + coff + (long long)hkv * RB, *vb = a.v_cache + coff + (long long)hkv * RB;
    const char *kn = a.k_new + ((long long)b * a.Hkv + hkv) * RB, *vn = a.v_new + ((long long)b * a.Hkv + hkv) * RB;
    // byte offset of the tile's first row; -1: its page is outside the pool (reported, the tile left out)
    auto tile_off = [&](int row) -> long long {
        if (!kPaged) return row * pitch;
        const int page = a.pg.table[(long long)b * a.pg.stride + (row >> a.pg.shift)];
        if (page < 0 || page >= a.pg.n_pages) { report(a.status_word, ZIPVL_DEV_BAD_INDEX); return -1; }
        return (((long long)page << a.pg.shift) + (row & ((1 << a.pg.shift) - 1))) * pitch;
    };

    float o[NT][VS][4], m[NT][2], l[NT][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
        for (int s = 0; s < VS; ++s)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[nt][s][e] = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) { m[nt][h] = -INFINITY; l[nt][h] = 0.f; }
    }
    uint32_t kr[2][KJ][4], vr[4][VJ][VW];
    // rows behind the last one are read as the last one (and weigh nothing)
    auto load_k = [&](int base, long long off) {
        off = off < 0 ? 0 : off;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int r = min(g + 8 * u, c1 - 1 - base);
            const char *p = (base + r == new_row ? kn : kb + off + r * pitch) + t * 16;
#pragma unroll
            for (int j = 0; j < KJ; ++j) load_row(p + j * 64, kr[u][j]);
        }
    };
    auto load_v = [&](int base, long long off) {
        off = off < 0 ? 0 : off;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = min(2 * t + (u & 1) + 8 * (u >> 1), c1 - 1 - base);
            const char *p = (base + r == new_row ? vn : vb + off + r * pitch) + g * (VW * 4);
#pragma unroll
            for (int j = 0; j < VJ; ++j) {
                if (2 * t + (u & 1) + 8 * (u >> 1) < c1 - base) load_row(p + j * (VW * 32), vr[u][j]);
                else
#pragma unroll
                    for (int w = 0; w < VW; ++w) vr[u][j][w] = 0u;
            }
        }
    };
    int base = c0 + warp * 16;
    long long off = -1, next_off = -1;
    if (base < c1) {
        off = tile_off(base);
        load_k(base, off);
        load_v(base, off);
    }
    if (NT > 2) __syncthreads();                     // the query heads are in shared memory
    for (; base < c1; base += kWarps * 16, off = next_off) {
        const bool more = base + kWarps * 16 < c1;
        next_off = more ? tile_off(base + kWarps * 16) : -1;
        const int rows = c1 - base;
        if (NT > 1 && rows > 2 * kWarps * 16) {      // the warp's tile after the next, into L2 (a lane: half a row of K and of V)
            const int row = lane >> 1;
            const long long far = kPaged ? tile_off(base + 2 * kWarps * 16) : off + 2 * kWarps * 16 * pitch;
            if (far >= 0 && 2 * kWarps * 16 + row < rows) {
                prefetch_l2(kb + far + row * pitch + (lane & 1) * (RB / 2));
                prefetch_l2(vb + far + row * pitch + (lane & 1) * (RB / 2));
            }
        }
        // Eq. 4: the appended row, stored by the lanes that hold its pieces
        if (off >= 0 && new_row >= base && new_row < min(base + 16, c1)) {
            const int r = new_row - base;
            if (g == (r & 7)) {
                char *p = const_cast<char *>(kb) + off + r * pitch + t * 16;
#pragma unroll
                for (int j = 0; j < KJ; ++j) {
                    if (r < 8) store_row(p + j * 64, kr[0][j]);
                    else store_row(p + j * 64, kr[1][j]);
                }
            }
            if (t == ((r & 7) >> 1)) {
                char *p = const_cast<char *>(vb) + off + r * pitch + g * (VW * 4);
                const int u = (r & 1) + 2 * (r >> 3);
#pragma unroll
                for (int j = 0; j < VJ; ++j)
#pragma unroll
                    for (int x = 0; x < 4; ++x)
                        if (x == u) store_row(p + j * (VW * 32), vr[x][j]);
            }
        }
        float c[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) c[nt][e] = 0.f;
#pragma unroll
        for (int j = 0; j < KJ; ++j)                 // (the head tiles' chains side by side)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                const uint4 qv = NT > 2 ? sm_q[(nt * KJ + j) * 32 + lane] : qr[NT > 2 ? 0 : nt][j];
                if (kOne && D == 64) {               // (two MMAs a sum: half the additions, 2-6% of a step)
                    float x[4];
                    mma16_new<kHalf>(x, kr[0][j][0], kr[1][j][0], kr[0][j][1], kr[1][j][1], qv.x, qv.y);
                    mma16<kHalf>(x, kr[0][j][2], kr[1][j][2], kr[0][j][3], kr[1][j][3], qv.z, qv.w);
#pragma unroll
                    for (int e = 0; e < 4; ++e) c[nt][e] += x[e];
                    continue;
                }
                if (kOne) {
                    float x[4], y[4];
                    mma16_new<kHalf>(x, kr[0][j][0], kr[1][j][0], kr[0][j][1], kr[1][j][1], qv.x, qv.y);
                    mma16_new<kHalf>(y, kr[0][j][2], kr[1][j][2], kr[0][j][3], kr[1][j][3], qv.z, qv.w);
#pragma unroll
                    for (int e = 0; e < 4; ++e) c[nt][e] += x[e] + y[e];
                    continue;
                }
                mma16<kHalf>(c[nt], kr[0][j][0], kr[1][j][0], kr[0][j][1], kr[1][j][1], qv.x, qv.y);
                mma16<kHalf>(c[nt], kr[0][j][2], kr[1][j][2], kr[0][j][3], kr[1][j][3], qv.z, qv.w);
            }
        if (more) load_k(base + kWarps * 16, next_off);
        if (off < 0) {                               // (uniform)
            if (more) load_v(base + kWarps * 16, next_off);
            continue;
        }
        // ---- weights of rows g and g + 8 for heads 2 t and 2 t + 1
        uint32_t pb[NT][2];
        bool grow = false;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
            for (int e = 0; e < 4; ++e) c[nt][e] = (g + 8 * (e >> 1) < rows) ? c[nt][e] * a.scale_log2 : -INFINITY;
            grow |= fmaxf(c[nt][0], c[nt][2]) > m[nt][0] + kGrow || fmaxf(c[nt][1], c[nt][3]) > m[nt][1] + kGrow;
        }
        if (__any_sync(0xffffffffu, grow)) {         // (one vote for all head tiles: between two of them nothing waits)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                float mx[2] = {fmaxf(c[nt][0], c[nt][2]), fmaxf(c[nt][1], c[nt][3])}, f[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int x = 4; x < 32; x <<= 1) mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], x));
                    mx[h] = fmaxf(mx[h], m[nt][h]);
                    f[h] = mx[h] == -INFINITY ? 1.f : fast_exp2(m[nt][h] - mx[h]);
                    m[nt][h] = mx[h];
                    l[nt][h] *= f[h];
                }
#pragma unroll
                for (int s = 0; s < VS; ++s) { o[nt][s][0] *= f[0]; o[nt][s][1] *= f[1]; o[nt][s][2] *= f[0]; o[nt][s][3] *= f[1]; }
            }
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const float r0 = m[nt][0] == -INFINITY ? 0.f : m[nt][0], r1 = m[nt][1] == -INFINITY ? 0.f : m[nt][1];
            if (kOne) {
                // every column holds the one head: columns 0, 1, 2 take the three parts of its weight
                const float p[2] = {fast_exp2(c[nt][0] - r0), fast_exp2(c[nt][2] - r0)};
                l[nt][0] += p[0] + p[1];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float x = p[u] * kTop, hi = leading_bits<kHalf>(x), y = (x - hi) * kStep, mid = leading_bits<kHalf>(y);
                    pb[nt][u] = transpose8(pack16<kHalf>(t == 0 ? hi : t == 1 ? (y - mid) * kStep : 0.f, t == 0 ? mid : 0.f));
                }
                continue;
            }
            const float p0 = fast_exp2(c[nt][0] - r0), p1 = fast_exp2(c[nt][1] - r1);
            const float p2 = fast_exp2(c[nt][2] - r0), p3 = fast_exp2(c[nt][3] - r1);
            l[nt][0] += p0 + p2;
            l[nt][1] += p1 + p3;
            c[nt][0] = p0; c[nt][1] = p1; c[nt][2] = p2; c[nt][3] = p3;
        }
        if (!kOne)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                pb[nt][0] = transpose8(pack16<kHalf>(c[nt][0], c[nt][1]));
                pb[nt][1] = transpose8(pack16<kHalf>(c[nt][2], c[nt][3]));
            }
#pragma unroll
        for (int j = 0; j < VJ; ++j)
#pragma unroll
            for (int w = 0; w < VW; ++w) {
                const uint32_t a0 = __byte_perm(vr[0][j][w], vr[1][j][w], 0x5410), a1 = __byte_perm(vr[0][j][w], vr[1][j][w], 0x7632);
                const uint32_t a2 = __byte_perm(vr[2][j][w], vr[3][j][w], 0x5410), a3 = __byte_perm(vr[2][j][w], vr[3][j][w], 0x7632);
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    float (&x)[4] = o[nt][j * VW + w];
                    if (kOne) {
                        float y[4];
                        mma16_new<kHalf>(y, a0, a1, a2, a3, pb[nt][0], pb[nt][1]);
#pragma unroll
                        for (int e = 0; e < 4; ++e) x[e] += y[e];
                    } else {
                        mma16<kHalf>(x, a0, a1, a2, a3, pb[nt][0], pb[nt][1]);
                    }
                }
            }
        if (more) load_v(base + kWarps * 16, next_off);
    }

    // ---- merge the warps, eight heads at a time (one head: the parts of its weights first)
    const auto channel = [&](int s) { return (s / VW) * (16 * VW) + g * (2 * VW) + (s % VW) * 2; };
    if (kOne) {
        // what the first parts alone make goes into a free place: an infinite value is infinite there, where the
        // parts that are zero or negative make it NaN
        if (t == 0)
#pragma unroll
            for (int s = 0; s < VS; ++s) *reinterpret_cast<float2 *>(&sm_o[warp][1][channel(s)]) = make_float2(o[0][s][0], o[0][s][2]);
#pragma unroll
        for (int s = 0; s < VS; ++s)
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
                const float part = fmaf(o[0][s][e + 1], 1.f / kStep, o[0][s][e]);         // columns 2 t, 2 t + 1
                o[0][s][e] = fmaf(__shfl_xor_sync(0xffffffffu, part, 1), 1.f / (kStep * kStep), part) * (1.f / kTop);
            }
    }
#pragma unroll
    for (int nt0 = 0; nt0 < NT; nt0 += ET) {
        if (nt0 > 0) __syncthreads();
#pragma unroll
        for (int nt = nt0; nt < (nt0 + ET < NT ? nt0 + ET : NT); ++nt)
#pragma unroll
            for (int h = 0; h < (kOne ? 1 : 2); ++h) {
#pragma unroll
                for (int x = 4; x < 32; x <<= 1) l[nt][h] += __shfl_xor_sync(0xffffffffu, l[nt][h], x);
                if (kOne && t > 0) continue;
                const int at = (nt - nt0) * 8 + 2 * t + h;
                if (g == 0) { sm_m[warp][at] = m[nt][h]; sm_l[warp][at] = l[nt][h]; }
#pragma unroll
                for (int s = 0; s < VS; ++s)
                    *reinterpret_cast<float2 *>(&sm_o[warp][at][channel(s)]) = make_float2(o[nt][s][h], o[nt][s][2 + h]);
            }
        __syncthreads();
        const int n_heads = min(8 * ET, G - nt0 * 8);
#pragma unroll(NT > 1 ? 2 : 1)
        for (int e = threadIdx.x; e < n_heads * (D / 2); e += kWarps * 32) {
            const int h = e / (D / 2), ch = 2 * (e % (D / 2));
            float M = -INFINITY, L = 0.f, x = 0.f, y = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) M = fmaxf(M, sm_m[w][h]);
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const float f = sm_m[w][h] == -INFINITY ? 0.f : fast_exp2(sm_m[w][h] - M);
                const float2 v = *reinterpret_cast<const float2 *>(&sm_o[w][h][ch]);
                L = fmaf(f, sm_l[w][h], L);
                x = fmaf(f, v.x, x);
                y = fmaf(f, v.y, y);
            }
            if (kOne && !(fabsf(x) + fabsf(y) < INFINITY)) {
                float u = 0.f, v = 0.f;
                for (int w = 0; w < kWarps; ++w) {
                    const float f = sm_m[w][h] == -INFINITY ? 0.f : fast_exp2(sm_m[w][h] - M);
                    u = fmaf(f, sm_o[w][1][ch], u);
                    v = fmaf(f, sm_o[w][1][ch + 1], v);
                }
                if (!(fabsf(u) < INFINITY)) x = u;
                if (!(fabsf(v) < INFINITY)) y = v;
            }
            float *p = dst + (nt0 * 8 + h) * head_pitch;
            *reinterpret_cast<float2 *>(p + 2 + ch) = make_float2(x, y);
            if (ch == 0) *reinterpret_cast<float2 *>(p) = make_float2(M, L);
        }
    }
}

template <bool kHalf, int D, int NT>
cudaError_t launch(const DmArgs &a, int B, cudaStream_t st) {
    const dim3 grid(a.Hkv, a.n_chunks, B), block(kWarps * 32);
    return a.pg.table ? launch_dependent(decode_mma_kernel<kHalf, true, D, NT>, grid, block, 0, st, a)
                      : launch_dependent(decode_mma_kernel<kHalf, false, D, NT>, grid, block, 0, st, a);
}
template <bool kHalf, int D>
cudaError_t launch(const DmArgs &a, int B, cudaStream_t st) {
    const int G = a.Hq / a.Hkv;
    return G == 1 ? launch<kHalf, D, 0>(a, B, st) : G <= 8 ? launch<kHalf, D, 1>(a, B, st) : G <= 16 ? launch<kHalf, D, 2>(a, B, st)
         : G <= 24 ? launch<kHalf, D, 3>(a, B, st) : launch<kHalf, D, 4>(a, B, st);
}
template <bool kHalf>
cudaError_t launch(const DmArgs &a, int B, int D, cudaStream_t st) {
    return D == 128 ? launch<kHalf, 128>(a, B, st) : D == 96 ? launch<kHalf, 96>(a, B, st) : launch<kHalf, 64>(a, B, st);
}

}  // namespace

bool decode_mma_supported(const zipvl_decode_desc &d) {
    const int G = d.n_q_heads / d.n_kv_heads;
    return (d.dtype == ZIPVL_BF16 || d.dtype == ZIPVL_F16) && (d.head_dim == 64 || d.head_dim == 96 || d.head_dim == 128) &&
           G <= 32;
}

// Rows per CTA.  One wave of CTAs where that gives each at most max_rows: every SM has its full share from
// the first moment (a second wave with a few CTAs costs a third of a short step: 332 against 377-430 us for
// four requests of 28K rows at 1.3 to 2.7 waves).  Longer problems: max_rows, dealt out by the
// scheduler.  (Cutting by the actual lengths, on the device, balances ragged batches but costs every
// CTA 2 us of dependent loads and sums: 91 -> 110 us for eight steps of one request of 2307 rows.)
int decode_mma_chunk(int B, int Hq, int Hkv, int D, int max_len) {
    const int nt = Hq == Hkv ? 0 : (Hq / Hkv + 7) / 8;
    const long long groups = (long long)B * Hkv, wave = 148 * ctas_per_sm(nt, D);
    const int n = (int)std::max(1ll, wave / groups);
    const auto tiles_of = [&](long long parts) { return (int)((max_len + parts - 1) / parts + 63) / 64 * 64; };
    // More than eight heads: an SM holds half the warps and a CTA's set-up and end weigh more, so a last wave that is nearly
    // empty costs most; six waves at least, in CTAs of 512 rows at least (16 requests of 10K-20K rows, 24 heads on 2: 1536 rows 72.5 us,
    // 768 62.7, 512 61.1, 384 64.8; 64 such requests, six waves of 1536 rows: 189.0, 189.6, 197.5, 214).
    const int G = Hq / Hkv, least = min_large(G, D), most = max_rows(G, D);
    const int large = G > 8 ? std::min(most, std::max(least, (int)(((groups * max_len) / (6 * wave) + 63) / 64 * 64))) : most;
    // (the last term: chunks are the grid's y, which ends at 65535)
    return std::max(std::min(large, std::max(64, tiles_of(n))), tiles_of(65535));
}

// Chunks times query heads of all requests, for this problem or any smaller batch or length: a chunk is no shorter than 64
// rows or max_rows allow, and in between there are no more of them than one wave (or one per request).
size_t decode_mma_slots(int B, int Hq, int Hkv, int D, int max_len) {
    const int G = Hq / Hkv, nt = G == 1 ? 0 : (G + 7) / 8;
    const auto cut = [&](size_t rows) { return (size_t)B * Hq * ((max_len + rows - 1) / rows); };
    const size_t wave = (size_t)G * std::max<size_t>(148 * ctas_per_sm(nt, D), (size_t)B * Hkv);
    return std::max(cut(min_large(G, D)), std::min(cut(64), wave));
}

zipvl_status launch_decode_mma(const zipvl_decode_desc &d, float scale_log2, const void *q, const void *k_new,
                               const void *v_new, void *k_cache, void *v_cache, const int64_t *cache_off, PageArgs pg,
                               const int32_t *capacity, int32_t *seq_lens, int max_len, float *partials, int *lens, void *out,
                               int32_t *status_word, cudaStream_t st) {
    const int B = d.batch, Hq = d.n_q_heads, Hkv = d.n_kv_heads;
    const int chunk = decode_mma_chunk(B, Hq, Hkv, d.head_dim, max_len), n_chunks = (max_len + chunk - 1) / chunk;
    const DmArgs a = {Hq, Hkv, max_len, chunk, n_chunks, scale_log2, (const char *)q, (const char *)k_new, (const char *)v_new,
                      (char *)k_cache, (char *)v_cache, cache_off, pg, capacity, seq_lens, partials, lens, status_word};
    const cudaError_t e = d.dtype == ZIPVL_F16 ? launch<true>(a, B, d.head_dim, st) : launch<false>(a, B, d.head_dim, st);
    if (e != cudaSuccess) return fail(ZIPVL_ERR_CUDA, "zipvl_decode: launch: %s", cudaGetErrorString(e));
    count_launches(1);
    return launch_decode_merge(d.dtype, d.head_dim, Hq, B, n_chunks, partials, lens, seq_lens, out, st);
}

}  // namespace zipvl
