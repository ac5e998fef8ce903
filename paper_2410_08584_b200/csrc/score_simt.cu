// Probe scoring on CUDA cores: exact fp32 FMA path (fp32 tensors) and the
// general-shape path for bf16 / fp16.  Supplementary Eq. A with the causal mask of
// Eq. 2, column sums of Eq. 6, normalisation of Eq. 8.
//
// A column sum of a row-softmax needs every row's final max and denominator,
// so the contraction runs twice and the attention matrix never leaves the SM:
//   pass 1  one thread per probe row, keys streamed through shared memory:
//           per (head, key chunk, probe) running max m and sum l (base 2);
//   pass 2  one thread per key, probe rows streamed through shared memory:
//           column sum of exp2(s - m_r) / l_r over the probes that see the key;
//   pass 3  sum over heads in fixed order, nnz by binary search, normalise.
// Nothing uses float atomics, so results repeat bit for bit.
//
// Short fp32 layers (kClusterKeys x 8 keys, 128 probes) take one sweep instead of two: a cluster of
// eight CTAs holds the scores of 32 probes against all keys of a head in registers, exchanges the row
// statistics through distributed shared memory and adds up the columns from the exponentials
// it already has.  The 1024-token, 4-head layer is 34 MFLOP of scores: what counts is the number
// of SMs at work (64 instead of 16) and the length of a thread's chain (2 x 4 register tiles over
// 128 keys instead of a dot product per key): 56 -> 9 us with the sum over heads.
#include <cooperative_groups.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace zipvl {
namespace {

constexpr int kChunk = 256;   // keys per pass-1 block
constexpr int kKeyTile = 32;  // keys staged in shared memory at a time
constexpr int kProbeTile = 32;
constexpr int kThreads = 128;

template <typename T, int D>
__global__ void __launch_bounds__(kThreads)
score_stats_kernel(LayerArgs a, const T *__restrict__ q, const T *__restrict__ k,
                   const int32_t *__restrict__ probe_pos, int P, int n_chunks,
                   float2 *__restrict__ stats, int32_t *status_word) {
    __shared__ __align__(16) float Ks[kKeyTile][D];
    const int chunk = blockIdx.x, h = blockIdx.y, g = h / a.G;
    const int r = blockIdx.z * kThreads + threadIdx.x;
    const int j0 = chunk * kChunk, j1 = min(a.L, j0 + kChunk);

    int c = -1;
    if (r < P) {
        c = probe_pos[r];
        if (c < 0 || c >= a.L) {
            if (chunk == 0 && h == 0) report(status_word, ZIPVL_DEV_BAD_INDEX);
            c = -1;
        }
    }
    float qr[D];
    if (c >= 0) {
        const T *qp = q + (long long)c * a.q_stride + (long long)h * D;
#pragma unroll
        for (int t = 0; t < D; t += 8) {
            float x[8];
            load8(qp + t, x);
#pragma unroll
            for (int u = 0; u < 8; ++u) qr[t + u] = x[u] * a.scale_log2;
        }
    } else {
#pragma unroll
        for (int t = 0; t < D; ++t) qr[t] = 0.f;
    }

    float m = -INFINITY, l = 0.f;
    for (int jt = j0; jt < j1; jt += kKeyTile) {
        __syncthreads();
        // stage keys jt .. jt+31 of kv head g as floats
        for (int e = threadIdx.x; e < kKeyTile * (D / 8); e += kThreads) {
            const int row = e / (D / 8), col = (e % (D / 8)) * 8;
            float x[8];
            if (jt + row < j1) {
                load8(k + (long long)(jt + row) * a.kv_stride + (long long)g * D + col, x);
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = 0.f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) Ks[row][col + u] = x[u];
        }
        __syncthreads();
        const int jend = min(min(j1, jt + kKeyTile), c + 1);  // causal: keys <= c
        for (int j = jt; j < jend; ++j) {
            const float4 *kr = reinterpret_cast<const float4 *>(Ks[j - jt]);
            float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
            for (int t = 0; t < D / 4; ++t) {
                const float4 kv = kr[t];
                s0 = fmaf(qr[4 * t], kv.x, s0);
                s1 = fmaf(qr[4 * t + 1], kv.y, s1);
                s2 = fmaf(qr[4 * t + 2], kv.z, s2);
                s3 = fmaf(qr[4 * t + 3], kv.w, s3);
            }
            const float s = (s0 + s1) + (s2 + s3);
            if (s > m) {
                l *= fast_exp2(m - s);
                m = s;
            }
            l += fast_exp2(s - m);
        }
    }
    if (r < P) stats[((long long)h * n_chunks + chunk) * P + r] = make_float2(m, l);
}

template <typename T, int D>
__global__ void __launch_bounds__(kThreads)
score_colsum_kernel(LayerArgs a, const T *__restrict__ q, const T *__restrict__ k,
                    const int32_t *__restrict__ probe_pos, int P, int n_chunks,
                    const float2 *__restrict__ stats, float *__restrict__ partial) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *Qs = reinterpret_cast<float *>(smem_raw);      // [kProbeTile][D]
    float *Ms = Qs + kProbeTile * D;                       // [P] merged row max
    float *Il = Ms + P;                                    // [P] 1 / merged row sum
    int *Pos = reinterpret_cast<int *>(Il + P);            // [P]

    const int h = blockIdx.y, g = h / a.G;
    const int jb = blockIdx.x * kThreads, j = jb + threadIdx.x;

    // merge the per-chunk row statistics of this head
    for (int r = threadIdx.x; r < P; r += kThreads) {
        int c = probe_pos[r];
        if (c < 0 || c >= a.L) c = -1;
        Pos[r] = c;
        float M = -INFINITY;
        for (int ch = 0; ch < n_chunks; ++ch)
            M = fmaxf(M, stats[((long long)h * n_chunks + ch) * P + r].x);
        float Lsum = 0.f;
        for (int ch = 0; ch < n_chunks; ++ch) {
            const float2 s = stats[((long long)h * n_chunks + ch) * P + r];
            if (s.y > 0.f) Lsum += s.y * fast_exp2(s.x - M);
        }
        Ms[r] = M;
        Il[r] = Lsum > 0.f ? 1.f / Lsum : 0.f;
    }

    float kr[D];
    if (j < a.L) {
        const T *kp = k + (long long)j * a.kv_stride + (long long)g * D;
#pragma unroll
        for (int t = 0; t < D; t += 8) {
            float x[8];
            load8(kp + t, x);
#pragma unroll
            for (int u = 0; u < 8; ++u) kr[t + u] = x[u] * a.scale_log2;
        }
    } else {
#pragma unroll
        for (int t = 0; t < D; ++t) kr[t] = 0.f;
    }
    __syncthreads();

    float colsum = 0.f;
    for (int rt = 0; rt < P; rt += kProbeTile) {
        const int rend = min(P, rt + kProbeTile);
        // if every probe of the tile sits before this block's first key, no key
        // of the block is visible to the tile (uniform over the block)
        int tile_max = -1;
        for (int r = rt; r < rend; ++r) tile_max = max(tile_max, Pos[r]);
        if (tile_max < jb) continue;
        __syncthreads();
        for (int e = threadIdx.x; e < kProbeTile * (D / 8); e += kThreads) {
            const int row = e / (D / 8), col = (e % (D / 8)) * 8;
            float x[8];
            const int c = (rt + row < P) ? Pos[rt + row] : -1;
            if (c >= 0) {
                load8(q + (long long)c * a.q_stride + (long long)h * D + col, x);
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = 0.f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) Qs[row * D + col + u] = x[u];
        }
        __syncthreads();
        for (int r = rt; r < rend; ++r) {
            if (Pos[r] < j) continue;       // causal mask (also skips invalid probes)
            const float4 *qv = reinterpret_cast<const float4 *>(Qs + (r - rt) * D);
            float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
            for (int t = 0; t < D / 4; ++t) {
                const float4 x = qv[t];
                s0 = fmaf(kr[4 * t], x.x, s0);
                s1 = fmaf(kr[4 * t + 1], x.y, s1);
                s2 = fmaf(kr[4 * t + 2], x.z, s2);
                s3 = fmaf(kr[4 * t + 3], x.w, s3);
            }
            const float s = (s0 + s1) + (s2 + s3);
            colsum += fast_exp2(s - Ms[r]) * Il[r];
        }
    }
    if (j < a.L) partial[(long long)h * a.L + j] = colsum;
}

constexpr int kClThreads = 256, kClProbes = 32, kClTile = 64;
constexpr int kClusterKeys = 4 * kClTile;   // keys a CTA can hold: 4 tiles x 8 scores in registers per thread

// grid (8 CTAs of a cluster, head, tile of 32 probes); NS = 64-key tiles per CTA.
// A thread owns rows row0 + 2 i (i < 2) and keys tx + 16 j (j < 4) of every tile; rows are padded by
// 16 bytes so that the float4 reads of a warp (2 rows, 16 keys) are conflict-free, and lanes 2i, 2i + 1
// share their keys (pairs of equal addresses make a 16-byte read two cycles instead of four).
template <int D, int NS>
__global__ void __launch_bounds__(kClThreads)
score_cluster_kernel(LayerArgs a, const float *__restrict__ q, const float *__restrict__ k,
                     const int32_t *__restrict__ probe_pos, int P, int keys_per_cta, float *__restrict__ partial,
                     int32_t *status_word) {
    constexpr int QP = D + 4, CH = D / 4;
    extern __shared__ __align__(16) float smem[];
    float *Qs = smem;                                   // [32][QP]
    float *Ks = Qs + kClProbes * QP;                    // two tiles [64][QP]
    float *part = Ks + 2 * kClTile * QP;                // column sums [8 warps][NS * 64]
    float *weight = part + 8 * NS * kClTile;            // [32]
    float2 *stat = reinterpret_cast<float2 *>(weight + kClProbes);   // [32] this CTA's (m, l)
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();

    grid_launch_dependents();
    grid_dependency_wait(q, k, probe_pos);
    const int rank = blockIdx.x, h = blockIdx.y, z = blockIdx.z, g = h / a.G;
    const int tid = threadIdx.x, tx = (tid & 31) >> 1, warp = tid >> 5;
    const int row0 = warp * 4 + (tid & 1);
    const int j0 = rank * keys_per_cta, j1 = min(a.L, j0 + keys_per_cta);

    auto load_keys = [&](int t) {
        float *dst = Ks + (t & 1) * kClTile * QP;
        for (int e = tid; e < kClTile * CH; e += kClThreads) {
            const int r = e / CH, c = (e % CH) * 4, j = j0 + t * kClTile + r;
            ptx::cp_async16(ptx::smem_u32(dst + r * QP + c), k + (long long)(j < j1 ? j : 0) * a.kv_stride + (long long)g * D + c,
                            j < j1 ? 16u : 0u);
        }
        ptx::cp_async_commit();
    };
    auto position = [&](int r) {                        // of probe r of this tile; -1: none or out of range
        const int p = z * kClProbes + r;
        const int c = p < P ? probe_pos[p] : -1;
        return c < a.L ? c : -1;
    };
    for (int e = tid; e < kClProbes * CH; e += kClThreads) {
        const int r = e / CH, c = (e % CH) * 4, pos = position(r);
        if (pos < 0 && c == 0 && h == 0 && rank == 0 && z * kClProbes + r < P) report(status_word, ZIPVL_DEV_BAD_INDEX);
        ptx::cp_async16(ptx::smem_u32(Qs + r * QP + c), q + (long long)max(pos, 0) * a.q_stride + (long long)h * D + c,
                        pos >= 0 ? 16u : 0u);
    }
    load_keys(0);
    if (NS > 1) load_keys(1);
    const int pos[2] = {position(row0), position(row0 + 2)};

    float s[NS][2][4];
#pragma unroll
    for (int t = 0; t < NS; ++t) {
        if (t + 1 < NS) ptx::cp_async_wait<1>(); else ptx::cp_async_wait<0>();
        __syncthreads();
        const float *kt = Ks + (t & 1) * kClTile * QP;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) s[t][i][j] = 0.f;
#pragma unroll 4
        for (int c = 0; c < CH; ++c) {
            float4 x[2], y[4];
#pragma unroll
            for (int i = 0; i < 2; ++i) x[i] = *reinterpret_cast<const float4 *>(Qs + (row0 + 2 * i) * QP + 4 * c);
#pragma unroll
            for (int j = 0; j < 4; ++j) y[j] = *reinterpret_cast<const float4 *>(kt + (tx + 16 * j) * QP + 4 * c);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    s[t][i][j] = fmaf(x[i].x, y[j].x, s[t][i][j]);
                    s[t][i][j] = fmaf(x[i].y, y[j].y, s[t][i][j]);
                    s[t][i][j] = fmaf(x[i].z, y[j].z, s[t][i][j]);
                    s[t][i][j] = fmaf(x[i].w, y[j].w, s[t][i][j]);
                }
        }
        if (t + 2 < NS) {
            __syncthreads();
            load_keys(t + 2);
        }
    }
    // row statistics over this CTA's keys; s becomes exp2(s - m)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        float m = -INFINITY;
#pragma unroll
        for (int t = 0; t < NS; ++t)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int key = j0 + t * kClTile + tx + 16 * j;
                s[t][i][j] = (key < j1 && key <= pos[i]) ? s[t][i][j] * a.scale_log2 : -INFINITY;
                m = fmaxf(m, s[t][i][j]);
            }
#pragma unroll
        for (int off = 16; off > 1; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        const float ref = m == -INFINITY ? 0.f : m;
        float l = 0.f;
#pragma unroll
        for (int t = 0; t < NS; ++t)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                s[t][i][j] = fast_exp2(s[t][i][j] - ref);
                l += s[t][i][j];
            }
#pragma unroll
        for (int off = 16; off > 1; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        if (tx == 0) stat[row0 + 2 * i] = make_float2(m, l);
    }
    cl.sync();
    if (tid < kClProbes) {                              // what this CTA's exponentials of row tid count for
        float2 st[8];
        float M = -INFINITY, sum = 0.f;
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            st[p] = *(cl.map_shared_rank(stat, p) + tid);
            M = fmaxf(M, st[p].x);
        }
#pragma unroll
        for (int p = 0; p < 8; ++p)
            if (st[p].y > 0.f) sum += st[p].y * fast_exp2(st[p].x - M);
        const float2 own = stat[tid];
        weight[tid] = own.y > 0.f ? fast_exp2(own.x - M) / sum : 0.f;
    }
    cl.sync();                                          // (also: nobody leaves while its statistics are read)
    const float w0 = weight[row0], w1 = weight[row0 + 2];
#pragma unroll
    for (int t = 0; t < NS; ++t)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float v = s[t][0][j] * w0 + s[t][1][j] * w1;
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            if (!(tid & 1)) part[warp * NS * kClTile + t * kClTile + tx + 16 * j] = v;
        }
    __syncthreads();
    for (int e = tid; e < NS * kClTile; e += kClThreads) {
        if (j0 + e >= j1) break;
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) v += part[w * NS * kClTile + e];
        partial[((long long)h * gridDim.z + z) * a.L + j0 + e] = v;
    }
}

// first r with probe_pos[r] >= x (probe_pos ascending)
__device__ __forceinline__ int lower_bound(const int32_t *p, int n, int x) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (p[mid] < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// n_part: partial rows to add up, in order (heads, or heads x probe tiles)
__global__ void score_finalize_kernel(int L, int Hq, int n_part, int P, const float *__restrict__ partial,
                                      const int32_t *__restrict__ probe_pos,
                                      float *__restrict__ acc, float *__restrict__ norm) {
    grid_launch_dependents();
    grid_dependency_wait(partial, probe_pos);
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= L) return;
    float s = 0.f;
#pragma unroll 8
    for (int h = 0; h < n_part; ++h) s += partial[(long long)h * L + j];
    // structural nnz: probes at positions j .. L-1
    const int nnz = lower_bound(probe_pos, P, L) - lower_bound(probe_pos, P, j);
    acc[j] = s;
    norm[j] = nnz > 0 ? s / ((float)Hq * (float)nnz) : 0.f;
}

}  // namespace

__global__ void sum_to_double_kernel(int L, const float *__restrict__ x, double *__restrict__ out) {
    __shared__ double sh[1024];
    double s = 0.0;
    for (int j = threadIdx.x; j < L; j += blockDim.x) s += (double)x[j];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0];
}

constexpr int kClMaxProbes = 128;
static bool use_cluster(int L, int P) { return L <= 8 * kClusterKeys && P <= kClMaxProbes; }

size_t score_simt_ws_bytes(int L, int Hq, int P) {
    const size_t n_chunks = (L + kChunk - 1) / kChunk;
    size_t stats = (size_t)Hq * n_chunks * P * sizeof(float2);
    stats = (stats + 255) & ~(size_t)255;
    // Room for every shorter row and smaller number of probes too: a buffer sized for the largest serves all.  The
    // one-sweep kernels need most at their own limits and nothing beyond.
    const int cl = L < 8 * kClusterKeys ? L : 8 * kClusterKeys, cp = P < kClMaxProbes ? P : kClMaxProbes;
    const size_t cluster = (size_t)Hq * ((cp + kClProbes - 1) / kClProbes) * cl * sizeof(float);
    const size_t two_pass = stats + (size_t)Hq * L * sizeof(float);
    return cluster > two_pass ? cluster : two_pass;
}

template <int D, int NS>
static zipvl_status run_cluster(const LayerArgs &a, const float *q, const float *k, const int32_t *probe_pos, int P,
                                float *acc, float *norm, double *total, float *partial, int32_t *status_word,
                                cudaStream_t st) {
    const size_t smem = sizeof(float) * ((kClProbes + 2 * kClTile) * (D + 4) + 8 * NS * kClTile + 3 * kClProbes);
    cudaError_t e = cudaFuncSetAttribute(score_cluster_kernel<D, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return fail(ZIPVL_ERR_CUDA, "score: smem opt-in: %s", cudaGetErrorString(e));
    const int nz = (P + kClProbes - 1) / kClProbes;
    e = launch_cluster(score_cluster_kernel<D, NS>, dim3(8, a.Hq, nz), dim3(kClThreads), smem, st, 8, a, q, k, probe_pos, P,
                       (a.L + 7) / 8, partial, status_word);
    if (e == cudaSuccess)
        e = launch_dependent(score_finalize_kernel, dim3((a.L + 63) / 64), dim3(64), 0, st, a.L, a.Hq, a.Hq * nz, P,
                             partial, probe_pos, acc, norm);
    if (e != cudaSuccess) return fail(ZIPVL_ERR_CUDA, "score: launch: %s", cudaGetErrorString(e));
    if (total) sum_to_double_kernel<<<1, 1024, 0, st>>>(a.L, acc, total);
    count_launches(total ? 3 : 2);
    return check_launch("zipvl_score");
}

template <int D>
static zipvl_status run_cluster(const LayerArgs &a, const float *q, const float *k, const int32_t *probe_pos, int P,
                                float *acc, float *norm, double *total, float *partial, int32_t *status_word,
                                cudaStream_t st) {
    const int keys = (a.L + 7) / 8;
    if (keys <= kClTile) return run_cluster<D, 1>(a, q, k, probe_pos, P, acc, norm, total, partial, status_word, st);
    if (keys <= 2 * kClTile) return run_cluster<D, 2>(a, q, k, probe_pos, P, acc, norm, total, partial, status_word, st);
    return run_cluster<D, 4>(a, q, k, probe_pos, P, acc, norm, total, partial, status_word, st);
}

template <typename T, int D>
static zipvl_status run(const LayerArgs &a, const void *q, const void *k,
                        const int32_t *probe_pos, int P, float *acc, float *norm, double *total,
                        void *ws, int32_t *status_word, cudaStream_t st) {
    const int n_chunks = (a.L + kChunk - 1) / kChunk;
    size_t stats_bytes = (size_t)a.Hq * n_chunks * P * sizeof(float2);
    stats_bytes = (stats_bytes + 255) & ~(size_t)255;
    float2 *stats = reinterpret_cast<float2 *>(ws);
    float *partial = reinterpret_cast<float *>(reinterpret_cast<char *>(ws) + stats_bytes);

    dim3 g1(n_chunks, a.Hq, (P + kThreads - 1) / kThreads);
    score_stats_kernel<T, D><<<g1, kThreads, 0, st>>>(a, (const T *)q, (const T *)k, probe_pos, P,
                                                     n_chunks, stats, status_word);
    const size_t smem = (size_t)kProbeTile * D * sizeof(float) + (size_t)P * 12;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(score_colsum_kernel<T, D>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return fail(ZIPVL_ERR_CUDA, "score: smem opt-in: %s", cudaGetErrorString(e));
    }
    dim3 g2((a.L + kThreads - 1) / kThreads, a.Hq);
    score_colsum_kernel<T, D><<<g2, kThreads, smem, st>>>(a, (const T *)q, (const T *)k, probe_pos,
                                                         P, n_chunks, stats, partial);
    score_finalize_kernel<<<(a.L + 255) / 256, 256, 0, st>>>(a.L, a.Hq, a.Hq, P, partial, probe_pos, acc,
                                                            norm);
    if (total) sum_to_double_kernel<<<1, 1024, 0, st>>>(a.L, acc, total);
    count_launches(total ? 4 : 3);
    return check_launch("zipvl_score");
}

zipvl_status launch_score_simt(const LayerArgs &a, int dtype, const void *q, const void *k,
                               const int32_t *probe_pos, int P, float *acc, float *norm,
                               double *total, void *ws, int32_t *status_word, cudaStream_t st) {
    if (P > 8192) return fail(ZIPVL_ERR_UNSUPPORTED, "score: n_probe %d > 8192", P);
    if (dtype == ZIPVL_F32 && use_cluster(a.L, P)) {
        // one sweep: every (head, 32 probes) is one cluster whose scores fit the registers of its CTAs
        auto *one = a.D == 64 ? run_cluster<64> : a.D == 96 ? run_cluster<96> : a.D == 128 ? run_cluster<128> : nullptr;
        if (one)
            return one(a, (const float *)q, (const float *)k, probe_pos, P, acc, norm, total, (float *)ws, status_word, st);
    }
    if (dtype == ZIPVL_F32) {
        if (a.D == 64) return run<float, 64>(a, q, k, probe_pos, P, acc, norm, total, ws, status_word, st);
        if (a.D == 96) return run<float, 96>(a, q, k, probe_pos, P, acc, norm, total, ws, status_word, st);
        if (a.D == 128) return run<float, 128>(a, q, k, probe_pos, P, acc, norm, total, ws, status_word, st);
    } else if (dtype == ZIPVL_F16) {
        if (a.D == 64) return run<__half, 64>(a, q, k, probe_pos, P, acc, norm, total, ws, status_word, st);
        if (a.D == 96) return run<__half, 96>(a, q, k, probe_pos, P, acc, norm, total, ws, status_word, st);
        if (a.D == 128) return run<__half, 128>(a, q, k, probe_pos, P, acc, norm, total, ws, status_word, st);
    } else {
        if (a.D == 64) return run<__nv_bfloat16, 64>(a, q, k, probe_pos, P, acc, norm, total, ws, status_word, st);
        if (a.D == 96) return run<__nv_bfloat16, 96>(a, q, k, probe_pos, P, acc, norm, total, ws, status_word, st);
        if (a.D == 128) return run<__nv_bfloat16, 128>(a, q, k, probe_pos, P, acc, norm, total, ws, status_word, st);
    }
    return fail(ZIPVL_ERR_UNSUPPORTED, "score: head_dim %d", a.D);
}

}  // namespace zipvl
