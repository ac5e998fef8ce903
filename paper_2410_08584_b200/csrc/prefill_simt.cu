// Sparse causal prefill attention on CUDA cores (Algorithm 1, attention over
// Q[T], K[T], V[T]; Eq. 2 on the gathered tokens): the exact-fp32 path for
// fp32 tensors and the general-shape path for bf16 / fp16.  The tensor-core kernel in
// prefill_tc.cu takes over for the 16-bit shapes it supports.
//
// What bounds it: fp32 multiply-adds (4 d k^2/2 per head) where the layer is large, and
// the length of one CTA's serial chain of key tiles where it is small: the 1024-token, 4-head
// layer is 0.34 GFLOP (5 us of the FMA pipes), yet 64-row CTAs that each walked all their key
// tiles with one key per lane took 129 us on 52 of 148 SMs.  Hence
//   - register tiles: a thread owns 4 query rows x kBN / TX keys of S and 4 rows x D / TX
//     channels of O.  Rows and keys are interleaved over the threads (row = base + RG i, key = tx +
//     TX i) and the rows padded, so that the 16-byte reads are free of bank conflicts;
//   - a thread-block cluster per (query tile, head): its C CTAs take every C-th key tile and
//     merge their (m, l, O) through distributed shared memory, each CTA the rows 64 / C * rank...;
//   - K of the next tile is fetched (cp.async, by index) while P V runs, V while Q K^T runs.
// With the compaction inside: 129 + 3.4 -> 28 us on that layer.
//
// PADDED output: whoever stores row i also zero-fills the rows of the dropped tokens between
// T[i-1] and T[i] (and after the last kept token), so padding costs no extra launch.
// Compaction (fp32 only: the copy is the staged bits): the CTA that holds the key tile of its own
// query rows writes those K and V rows to the caches from shared memory.
#include <cooperative_groups.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace zipvl {
namespace {

namespace cg = cooperative_groups;

constexpr int kBM = 64;     // query rows per CTA

template <int D>
struct Shape {
    static constexpr int TX = D == 96 ? 8 : 16;        // threads along keys / channels
    static constexpr int kBN = D == 64 ? 64 : 32;       // keys per tile (two or three CTAs per SM)
    static constexpr int kThreads = kBM / 4 * TX;
    static constexpr int KPT = kBN / TX;                // keys of S per thread and row
    static constexpr int CPT = D / TX / 4;              // float4 of O per thread and row
    static constexpr int QP = D + 4, PP = kBN + TX;     // padded pitches
    static constexpr size_t kSmem = sizeof(float) * (kBM * QP + kBN * QP + kBN * D + kBM * PP) + sizeof(int) * (kBM + 1);
};

template <typename T, int D>
__global__ void __launch_bounds__(Shape<D>::kThreads)
prefill_simt_kernel(LayerArgs a, const T *__restrict__ q, const T *__restrict__ k,
                    const T *__restrict__ v, const int32_t *__restrict__ idx,
                    const int32_t *__restrict__ k_dev, int k_max, T *__restrict__ out, int out_mode,
                    T *__restrict__ kc, T *__restrict__ vc, int capacity, int32_t *__restrict__ len_out, int z0,
                    int32_t *status_word) {
    using S = Shape<D>;
    constexpr int TX = S::TX, kBN = S::kBN, NT = S::kThreads, KPT = S::KPT, CPT = S::CPT, QP = S::QP, PP = S::PP;
    constexpr bool kF32 = sizeof(T) == 4;
    constexpr int CH = D / 4;                           // 16-byte pieces of a row of floats
    constexpr int LPT = kBN * CH / NT;                  // pieces of a K (or V) tile per thread
    extern __shared__ __align__(16) float smem[];
    float *Qs = smem;                                   // [kBM][QP], later this CTA's O
    float *Ks = Qs + kBM * QP;                          // [kBN][QP]
    float *Vs = Ks + kBN * QP;                          // [kBN][D]
    float *Ps = Vs + kBN * D;                           // [kBM][PP], later (m, l) of the rows
    int *row_tok = reinterpret_cast<int *>(Ps + kBM * PP) + 1;   // tokens of rows -1 .. kBM - 1

    grid_launch_dependents();
    grid_dependency_wait(q, k, v, idx, k_dev);
    int n = *k_dev;
    const int rank = blockIdx.x, C = gridDim.x, h = blockIdx.y, z = z0 + (int)blockIdx.z, g = h / a.G;
    const int tid = threadIdx.x;
    if (n > k_max || n < 0) {
        if (rank == 0 && h == 0 && z == 0 && tid == 0) report(status_word, ZIPVL_DEV_CAPACITY);
        n = n < 0 ? 0 : k_max;
    }
    if (n == 0 && z == 0) {
        // nothing kept: every row is a dropped token's row
        if (out_mode == ZIPVL_OUT_PADDED)
            for (long long e = rank * NT + tid; e < (long long)a.L * D; e += C * NT)
                store_elem(out + ((e / D) * a.Hq + h) * D + (e % D), 0.f);
        if (kc != nullptr && h == 0 && rank == 0 && tid == 0) *len_out = 0;
    }
    // the longest rows first; tiles past the kept set leave at once (the whole cluster together)
    const int qt = (n + kBM - 1) / kBM - 1 - z;
    if (qt < 0) return;
    const int i0 = qt * kBM, i1 = min(n, i0 + kBM);
    const int n_kt = (i1 + kBN - 1) / kBN;              // key tiles up to the diagonal
    // A warp is 32 / TX row groups by TX key groups.  Neighbouring lanes share their key group and
    // every eight lanes hold two row groups: a 16-byte read of a row piece and one of a key piece then take
    // two cycles each instead of four (measured: pairs of equal addresses are merged).
    constexpr int RG = 32 / TX;
    const int lane = tid & 31, tx = (lane >> 1) % TX;
    const int rg = TX == 16 ? (lane & 1) : ((lane & 1) | (lane >> 4 << 1));
    const int ty = (tid >> 5) * RG + rg;
    const int row0 = (tid >> 5) * (4 * RG) + rg;        // + RG * i

    auto token = [&](int i) {
        if (i >= i1) return -1;
        const int t = idx[i];
        return (t < 0 || t >= a.L) ? -1 : t;
    };
    auto load_piece = [&](float *dst, const T *src, bool ok) {
        if constexpr (kF32) {
            ptx::cp_async16(ptx::smem_u32(dst), src, ok ? 16u : 0u);
        } else {
            float x[4] = {0.f, 0.f, 0.f, 0.f};
            if (ok)
                for (int u = 0; u < 4; ++u) x[u] = to_float(src[u]);
            *reinterpret_cast<float4 *>(dst) = make_float4(x[0], x[1], x[2], x[3]);
        }
    };
    int tok[LPT];                                       // tokens of the pieces of the tile to be loaded next
    auto look_up = [&](int kt) {
#pragma unroll
        for (int u = 0; u < LPT; ++u) tok[u] = kt < n_kt ? token(kt * kBN + (tid + u * NT) / CH) : -1;
    };
    auto load_k = [&]() {
#pragma unroll
        for (int u = 0; u < LPT; ++u) {
            const int e = tid + u * NT, r = e / CH, c = (e % CH) * 4;
            load_piece(Ks + r * QP + c, k + (long long)max(tok[u], 0) * a.kv_stride + (long long)g * D + c, tok[u] >= 0);
        }
        ptx::cp_async_commit();
    };
    auto load_v = [&](const int (&t)[LPT]) {
#pragma unroll
        for (int u = 0; u < LPT; ++u) {
            const int e = tid + u * NT, r = e / CH, c = (e % CH) * 4;
            load_piece(Vs + r * D + c, v + (long long)max(t[u], 0) * a.kv_stride + (long long)g * D + c, t[u] >= 0);
        }
        ptx::cp_async_commit();
    };

    // the rows' tokens once, into shared memory (an index load per use would put one L2 latency
    // after another in front of the first tile and behind the last one)
    look_up(rank);
    if (tid <= kBM) {
        const int i = i0 + tid - 1;
        const int t = i < 0 || i >= i1 ? -1 : idx[i];
        row_tok[tid - 1] = t < a.L ? t : -1;
        if (tid > 0 && i < i1 && rank == 0 && (t < 0 || t >= a.L)) report(status_word, ZIPVL_DEV_BAD_INDEX);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kBM * CH / NT; ++u) {
        const int e = tid + u * NT, r = e / CH, c = (e % CH) * 4, t = row_tok[r];
        load_piece(Qs + r * QP + c, q + (long long)max(t, 0) * a.q_stride + (long long)h * D + c, t >= 0);
    }
    load_k();
    int tok_v[LPT];
#pragma unroll
    for (int u = 0; u < LPT; ++u) tok_v[u] = tok[u];
    load_v(tok_v);

    float m[4], l[4];
    float4 o[4][CPT];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m[i] = -INFINITY;
        l[i] = 0.f;
#pragma unroll
        for (int c = 0; c < CPT; ++c) o[i][c] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const int lim = min(n, capacity);
    for (int kt = rank; kt < n_kt; kt += C) {
        const bool more = kt + C < n_kt;
        // does this tile hold the K and V rows of this CTA's own tokens, and is it this head's to copy?
        const bool keep = kF32 && kc != nullptr && h % a.G == 0 && kt * kBN >= i0;
        auto copy_out = [&](const float *src, int pitch, T *dst) {
#pragma unroll
            for (int u = 0; u < LPT; ++u) {
                const int e = tid + u * NT, r = e / CH, c = (e % CH) * 4, i = kt * kBN + r;
                if (i < lim && tok_v[u] >= 0)
                    *reinterpret_cast<float4 *>(reinterpret_cast<float *>(dst) + ((long long)i * a.Hkv + g) * D + c) =
                        *reinterpret_cast<const float4 *>(src + r * pitch + c);
            }
        };
        ptx::cp_async_wait<1>();                        // K is in (V may still be on its way)
        __syncthreads();
        if (more) look_up(kt + C);
        float s[4][KPT];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < KPT; ++j) s[i][j] = 0.f;
#pragma unroll 4
        for (int c = 0; c < CH; ++c) {
            float4 x[4], y[KPT];
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float4 *>(Qs + (row0 + RG * i) * QP + 4 * c);
#pragma unroll
            for (int j = 0; j < KPT; ++j) y[j] = *reinterpret_cast<const float4 *>(Ks + (tx + TX * j) * QP + 4 * c);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < KPT; ++j) {
                    s[i][j] = fmaf(x[i].x, y[j].x, s[i][j]);
                    s[i][j] = fmaf(x[i].y, y[j].y, s[i][j]);
                    s[i][j] = fmaf(x[i].z, y[j].z, s[i][j]);
                    s[i][j] = fmaf(x[i].w, y[j].w, s[i][j]);
                }
        }
        if (keep) copy_out(Ks, QP, kc);
        __syncthreads();                                // K has been read
        if (more) load_k();
        // online softmax: the TX threads of a row are in one warp
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int qi = i0 + row0 + RG * i;
            float mx = m[i];
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                s[i][j] = (kt * kBN + tx + TX * j <= qi) ? s[i][j] * a.scale_log2 : -INFINITY;   // causal inside T
                mx = fmaxf(mx, s[i][j]);
            }
#pragma unroll
            for (int off = TX; off > 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            const float ref = mx == -INFINITY ? 0.f : mx;
            const float sc = fast_exp2(m[i] - ref);
            float sum = 0.f;
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                const float p = fast_exp2(s[i][j] - ref);
                sum += p;
                Ps[(row0 + RG * i) * PP + tx + TX * j] = p;
            }
            m[i] = mx;
            l[i] = l[i] * sc + sum;                     // this thread's share of the row
#pragma unroll
            for (int c = 0; c < CPT; ++c) { o[i][c].x *= sc; o[i][c].y *= sc; o[i][c].z *= sc; o[i][c].w *= sc; }
        }
        if (more) ptx::cp_async_wait<1>(); else ptx::cp_async_wait<0>();   // V is in
        __syncthreads();
        // Keys behind the warp's last row weigh nothing and are left out: 0 x Inf would reach rows that do not see
        // that key (rows of a warp are 4 RG consecutive ones, a multiple of four).
        const int seen = min(kBN, i0 + ((tid >> 5) + 1) * (4 * RG) - kt * kBN);
#pragma unroll 2
        for (int j = 0; j < seen; j += 4) {
            float4 p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = *reinterpret_cast<const float4 *>(Ps + (row0 + RG * i) * PP + j);
#pragma unroll
            for (int jj = 0; jj < 4; ++jj)
#pragma unroll
                for (int c = 0; c < CPT; ++c) {
                    const float4 y = *reinterpret_cast<const float4 *>(Vs + (j + jj) * D + (tx + TX * c) * 4);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float w = jj == 0 ? p[i].x : jj == 1 ? p[i].y : jj == 2 ? p[i].z : p[i].w;
                        o[i][c].x = fmaf(w, y.x, o[i][c].x);
                        o[i][c].y = fmaf(w, y.y, o[i][c].y);
                        o[i][c].z = fmaf(w, y.z, o[i][c].z);
                        o[i][c].w = fmaf(w, y.w, o[i][c].w);
                    }
                }
        }
        if (keep) copy_out(Vs, D, vc);
        __syncthreads();                                // V and P have been read
        if (more) {
#pragma unroll
            for (int u = 0; u < LPT; ++u) tok_v[u] = tok[u];
            load_v(tok_v);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int off = TX; off > 1; off >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);
    if (rank >= n_kt) {                                 // (no key tile of its own: its first loads were empty)
        ptx::cp_async_wait<0>();
        __syncthreads();
    }

    // one row of the output, TX threads wide, by the thread that holds its channels; then the gap in
    // front of it (an entry that is out of range or not below its successor is read as "no gap")
    auto store_row = [&](int i, float inv, const float4 (&x)[CPT]) {
        const int t = row_tok[i - i0];
        if (t < 0) return;
        const bool padded = out_mode == ZIPVL_OUT_PADDED;
        auto put = [&](long long row, bool zero) {
            T *dst = out + (row * a.Hq + h) * D;
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const float4 w = zero ? make_float4(0.f, 0.f, 0.f, 0.f)
                                      : make_float4(x[c].x * inv, x[c].y * inv, x[c].z * inv, x[c].w * inv);
                T *p = dst + (tx + TX * c) * 4;
                if constexpr (kF32) {
                    *reinterpret_cast<float4 *>(p) = w;
                } else {
                    store_elem(p, w.x); store_elem(p + 1, w.y); store_elem(p + 2, w.z); store_elem(p + 3, w.w);
                }
            }
        };
        put(padded ? t : i, false);
        if (padded) {
            int lo = 0;
            if (i > 0) {
                const int tp = row_tok[i - i0 - 1];
                lo = (tp >= 0 && tp < t) ? tp + 1 : t;
            }
            for (int z = lo; z < t; ++z) put(z, true);
            if (i == n - 1)
                for (int z = t + 1; z < a.L; ++z) put(z, true);
        }
    };
    if (C == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int qi = i0 + row0 + RG * i;
            if (qi < i1) store_row(qi, l[i] > 0.f ? 1.f / l[i] : 0.f, o[i]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = row0 + RG * i;
#pragma unroll
            for (int c = 0; c < CPT; ++c) *reinterpret_cast<float4 *>(Qs + r * QP + (tx + TX * c) * 4) = o[i][c];
            if (tx == 0) *reinterpret_cast<float2 *>(Ps + 2 * r) = make_float2(m[i], l[i]);
        }
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();
        const int per = kBM / C;                        // rows this CTA merges
        for (int r = rank * per + ty; r < (rank + 1) * per; r += NT / TX) {
            if (i0 + r >= i1) break;
            float M = -INFINITY, sum = 0.f;
            float2 ml[8];
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                ml[p] = p < C ? *reinterpret_cast<const float2 *>(cl.map_shared_rank(Ps, p) + 2 * r)
                              : make_float2(-INFINITY, 0.f);
                M = fmaxf(M, ml[p].x);
            }
            float4 x[CPT];
#pragma unroll
            for (int c = 0; c < CPT; ++c) x[c] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                if (p >= C) break;
                const float w = ml[p].y > 0.f ? fast_exp2(ml[p].x - M) : 0.f;
                sum = fmaf(w, ml[p].y, sum);
                const float *src = cl.map_shared_rank(Qs, p) + r * QP;
#pragma unroll
                for (int c = 0; c < CPT; ++c) {
                    const float4 y = *reinterpret_cast<const float4 *>(src + (tx + TX * c) * 4);
                    x[c].x = fmaf(w, y.x, x[c].x);
                    x[c].y = fmaf(w, y.y, x[c].y);
                    x[c].z = fmaf(w, y.z, x[c].z);
                    x[c].w = fmaf(w, y.w, x[c].w);
                }
            }
            store_row(i0 + r, sum > 0.f ? 1.f / sum : 0.f, x);
        }
        cl.sync();                                      // nobody leaves while its shared memory is read
    }
    if (kF32 && kc != nullptr && h == 0 && z == 0 && rank == 0 && tid == 0) {
        *len_out = lim;
        if (n > capacity) report(status_word, ZIPVL_DEV_CAPACITY);
    }
}

template <typename T, int D>
zipvl_status run(const LayerArgs &a, const void *q, const void *k, const void *v,
                 const int32_t *idx, const int32_t *k_dev, int k_max, void *out, int out_mode, void *kc, void *vc,
                 int capacity, int32_t *len_out, int32_t *status_word, cudaStream_t st) {
    static_assert(Shape<D>::kSmem <= 120 * 1024, "");
    const int tiles = (k_max + kBM - 1) / kBM;
    // CTAs per (query tile, head): as many as keep the launch within about two CTAs per SM (a wave),
    // so that short layers use every SM and long ones keep whole rows in one CTA; no more than
    // a row has key tiles.
    int C = 1;
    while (C < 8 && 2 * C <= tiles && (long long)tiles * a.Hq * 2 * C <= 360) C *= 2;
    // Clusters of two and four: each CTA gets an SM to itself (by its shared-memory request), which takes the longest rows,
    // started first, off the critical path.  Attention with compaction, shared and alone, in us: two CTAs: 4 heads x 64, 1500
    // tokens 60.8, 51.4, 2300 tokens 119, 79; 16 x 128, 400 tokens 50, 35; no shape of 13 slower.  Four: 4 x 64, 1024 tokens 35.2, 27.6;
    // 4 x 128 61.0, 45.7; 2 x 64, 2300 64.5, 50.2; but where a CTA has one key tile or a third wave comes: 12 x 64, 200 tokens 12.3, 17.2;
    // 8 x 64, 700 27.5, 35.6.  Eight (short chains): 4 x 64, 700 tokens 22.5, 32.5; 1 x 64, 2300 35.7, 41.7.
    const long long ctas = (long long)tiles * a.Hq * C;
    const bool alone = C == 2 || (C == 4 && (ctas <= 148 || (ctas <= 296 && tiles > C)));
    const size_t smem = alone ? (size_t)120 * 1024 : Shape<D>::kSmem;
    cudaError_t e = cudaFuncSetAttribute(prefill_simt_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         120 * 1024);
    if (e != cudaSuccess) return fail(ZIPVL_ERR_CUDA, "sparse_prefill: smem opt-in: %s", cudaGetErrorString(e));
    // (the grid's z ends at 65535, which a prompt of four million tokens has more tiles than)
    for (int z0 = 0; z0 < tiles; z0 += 65535) {
        e = launch_cluster(prefill_simt_kernel<T, D>, dim3(C, a.Hq, tiles - z0 < 65535 ? tiles - z0 : 65535),
                           dim3(Shape<D>::kThreads), smem, st, C, a, (const T *)q, (const T *)k, (const T *)v, idx, k_dev, k_max,
                           (T *)out, out_mode, (T *)kc, (T *)vc, capacity, len_out, z0, status_word);
        if (e != cudaSuccess) return fail(ZIPVL_ERR_CUDA, "sparse_prefill: launch: %s", cudaGetErrorString(e));
        count_launches(1);
    }
    return check_launch("zipvl_sparse_prefill");
}

}  // namespace

zipvl_status launch_prefill_simt(const LayerArgs &a, int dtype, const void *q, const void *k,
                                 const void *v, const int32_t *idx, const int32_t *k_dev,
                                 int k_max, void *out, int out_mode, void *kc, void *vc, int capacity,
                                 int32_t *len_out, int32_t *status_word, cudaStream_t st) {
#define ZIPVL_RUN(T, HD) \
    if (a.D == HD) return run<T, HD>(a, q, k, v, idx, k_dev, k_max, out, out_mode, kc, vc, capacity, len_out, status_word, st)
    if (dtype == ZIPVL_F32) {
        ZIPVL_RUN(float, 64);
        ZIPVL_RUN(float, 96);
        ZIPVL_RUN(float, 128);
    } else if (dtype == ZIPVL_F16) {
        ZIPVL_RUN(__half, 64);
        ZIPVL_RUN(__half, 96);
        ZIPVL_RUN(__half, 128);
    } else {
        ZIPVL_RUN(__nv_bfloat16, 64);
        ZIPVL_RUN(__nv_bfloat16, 96);
        ZIPVL_RUN(__nv_bfloat16, 128);
    }
#undef ZIPVL_RUN
    return fail(ZIPVL_ERR_UNSUPPORTED, "sparse_prefill: head_dim %d", a.D);
}

}  // namespace zipvl
