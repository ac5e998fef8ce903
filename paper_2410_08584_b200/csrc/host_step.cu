// Algorithm 1 (and one step of Algorithm 2) from and to HOST buffers: zipvl_prefill_layer_host,
// zipvl_layer_step_host.
//
// What bounds it: the bus.  A 2944-token, 32-head layer copies 72 MB in and about 62 MB out at some 54 GB/s each
// way; its kernels take 0.14 ms.  One direction after the other the call took 2.77 ms, now 1.90.  The order here
// lets the two directions overlap:
//   - K goes first; beside it a small kernel fetches the probe rows of Q (and the decode step's
//     rows) straight from pinned host memory, so that the token set is known when K has landed;
//   - from then on K[T] goes out while V and Q come in, V[T] behind it;
//   - Q comes in groups of heads (rows of a group are 2 KB or so, which a strided copy moves at
//     the full rate), the attention of a group runs as soon as it is there, and its output goes out while
//     the next group comes in.
// Three streams (in, run, out) joined by events; the host waits twice, for k and for the end.
#include <cuda.h>
#include <math.h>

#include <mutex>

#include "common.cuh"
#include "tc.cuh"

namespace zipvl {
namespace {

constexpr int kMaxDevices = 64, kMaxGroups = 8, kKeptContexts = 4;

// Device scratch comes from a memory pool of the library's own
// (one per device, created on first use) whose release threshold is unlimited: the
// few hundred MB a call needs are then handed back to the pool, not to the driver, when
// the call ends, and the next call gets them again at once.  With the device's default
// pool every call paid for mapping and unmapping that memory (16 ms against 2.7 ms per
// call on a 2944-token layer).  zipvl_release_host_scratch() gives the memory back.
cudaMemPool_t g_host_pool[kMaxDevices] = {};
std::mutex g_host_mutex;        // pools and contexts

cudaError_t host_pool(int dev, cudaMemPool_t *pool) {
    std::lock_guard<std::mutex> lock(g_host_mutex);
    if (!g_host_pool[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        cudaError_t e = cudaMemPoolCreate(&p, &props);
        if (e != cudaSuccess) return e;
        unsigned long long keep = ~0ull;
        e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) { cudaMemPoolDestroy(p); return e; }
        g_host_pool[dev] = p;
    }
    *pool = g_host_pool[dev];
    return cudaSuccess;
}

// What a call needs besides memory: made on first use, one per call in flight, at most kKeptContexts per
// device kept for later calls (making them takes longer than a short layer).
struct HostContext {
    cudaStream_t in = nullptr, run = nullptr, out = nullptr;
    cudaEvent_t alloc = nullptr, k_in = nullptr, v_in = nullptr, chosen = nullptr, told = nullptr, k_kept = nullptr,
                v_kept = nullptr, decoded = nullptr, q_in[kMaxGroups] = {}, done[kMaxGroups] = {};
    int32_t *misc = nullptr;    // pinned

    cudaError_t create() {
        cudaError_t e = cudaSuccess;
        for (cudaStream_t *s : {&in, &run, &out})
            if (e == cudaSuccess) e = cudaStreamCreateWithFlags(s, cudaStreamNonBlocking);
        each([&](cudaEvent_t &ev) { if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming); });
        if (e == cudaSuccess) e = cudaHostAlloc((void **)&misc, 64, cudaHostAllocDefault);
        return e;
    }
    void destroy() {
        each([](cudaEvent_t &ev) { if (ev) cudaEventDestroy(ev); });
        for (cudaStream_t s : {in, run, out})
            if (s) cudaStreamDestroy(s);
        if (misc) cudaFreeHost(misc);
    }
    template <typename F>
    void each(F f) {
        for (cudaEvent_t *ev : {&alloc, &k_in, &v_in, &chosen, &told, &k_kept, &v_kept, &decoded}) f(*ev);
        for (int i = 0; i < kMaxGroups; ++i) { f(q_in[i]); f(done[i]); }
    }
};
// (a fixed array: nothing that may throw behind a C entry)
struct KeptContexts {
    HostContext at[kKeptContexts];
    int n;
} g_host_context[kMaxDevices];

cudaError_t take_context(int dev, HostContext *c) {
    {
        std::lock_guard<std::mutex> lock(g_host_mutex);
        KeptContexts &kept = g_host_context[dev];
        if (kept.n > 0) {
            *c = kept.at[--kept.n];
            return cudaSuccess;
        }
    }
    const cudaError_t e = c->create();
    if (e != cudaSuccess) { c->destroy(); *c = HostContext(); }
    return e;
}
void give_context(int dev, HostContext &c) {
    {
        std::lock_guard<std::mutex> lock(g_host_mutex);
        KeptContexts &kept = g_host_context[dev];
        if (kept.n < kKeptContexts) {
            kept.at[kept.n++] = c;
            return;
        }
    }
    c.destroy();
}

// The device's address of pinned host memory [p, p + bytes); nullptr for any other memory.  The whole range has to
// lie in one allocation: two pinned ranges may have memory between them that the GPU cannot read.
const void *mapped(const void *p, size_t bytes) {
    if (!p) return nullptr;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (at.type != cudaMemoryTypeHost || !at.devicePointer || ((uintptr_t)at.devicePointer & 15u)) return nullptr;
    static const auto attribute = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPoint("cuPointerGetAttribute", &f, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<CUresult (*)(void *, CUpointer_attribute, CUdeviceptr)>(f);
    }();
    CUdeviceptr start = 0;
    size_t size = 0;
    const CUdeviceptr first = (CUdeviceptr)(uintptr_t)at.devicePointer;
    if (!attribute || attribute(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, first) != CUDA_SUCCESS ||
        attribute(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, first) != CUDA_SUCCESS)
        return nullptr;
    return first >= start && bytes <= size && first - start <= size - bytes ? at.devicePointer : nullptr;
}

// Small inputs read over the bus by the GPU itself.  Block r < P: probe row r of Q into its place; the blocks
// behind: the three rows of the decode step.  Block 0 also copies the positions and sets the
// call's words: [0] k, [1] cache length, [2] status, [3] cache capacity, [4..] offset 0.
struct SmallInputs {
    const uint4 *q, *rows[3];
    const int32_t *probe;
    uint4 *q_dev, *rows_dev[3];
    int32_t *probe_dev, *misc;
    int L, P, cap, q_chunks, row_chunks[3];   // 16-byte chunks of a row
};
__global__ void __launch_bounds__(256) fetch_small_inputs_kernel(SmallInputs s) {
    if (blockIdx.x == 0) {
        if (threadIdx.x < 8) s.misc[threadIdx.x] = threadIdx.x == 3 ? s.cap : 0;
        if (s.probe)
            for (int i = threadIdx.x; i < s.P; i += 256) s.probe_dev[i] = s.probe[i];
    }
    const int r = blockIdx.x;
    if (r < s.P) {
        if (!s.q) return;
        const int t = s.probe[r];
        if (t < 0 || t >= s.L) return;                       // (reported by the scoring)
        const uint4 *src = s.q + (long long)t * s.q_chunks;
        uint4 *dst = s.q_dev + (long long)t * s.q_chunks;
        for (int i = threadIdx.x; i < s.q_chunks; i += 256) dst[i] = src[i];
    } else {
        const int j = r - s.P;
        if (j < 3 && s.rows[j])
            for (int i = threadIdx.x; i < s.row_chunks[j]; i += 256) s.rows_dev[j][i] = s.rows[j][i];
    }
}

}  // namespace
}  // namespace zipvl

using namespace zipvl;

extern "C" {

zipvl_status zipvl_release_host_scratch(void) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return fail(ZIPVL_ERR_CUDA, "zipvl_release_host_scratch: no current device");
    std::lock_guard<std::mutex> lock(g_host_mutex);
    KeptContexts &kept = g_host_context[dev];
    while (kept.n > 0) kept.at[--kept.n].destroy();
    if (g_host_pool[dev]) {
        const cudaError_t e = cudaMemPoolTrimTo(g_host_pool[dev], 0);
        if (e != cudaSuccess)
            return fail(ZIPVL_ERR_CUDA, "zipvl_release_host_scratch: %s", cudaGetErrorString(e));
    }
    return ZIPVL_OK;
}

zipvl_status zipvl_prefill_layer_host(const zipvl_layer *layer, const void *q, const void *k,
                                      const void *v, const int32_t *probe_pos, int32_t n_probe,
                                      float tau, int32_t *k_out, int32_t *idx_out, void *out,
                                      void *k_cache_out, void *v_cache_out) {
    return zipvl_layer_step_host(layer, q, k, v, probe_pos, n_probe, tau, k_out, idx_out, out,
                                 k_cache_out, v_cache_out, nullptr, nullptr, nullptr, nullptr);
}

#define ZIPVL_CUDA(call)                                                                   \
    do {                                                                                   \
        const cudaError_t e_ = (call);                                                     \
        if (e_ != cudaSuccess)                                                             \
            return fail(ZIPVL_ERR_CUDA, "prefill_layer_host: %s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)
#define ZIPVL_CALL(call)                           \
    do {                                           \
        const zipvl_status s_ = (call);            \
        if (s_ != ZIPVL_OK) return s_;             \
    } while (0)

zipvl_status zipvl_layer_step_host(const zipvl_layer *layer, const void *q, const void *k,
                                   const void *v, const int32_t *probe_pos, int32_t n_probe,
                                   float tau, int32_t *k_out, int32_t *idx_out, void *out,
                                   void *k_cache_out, void *v_cache_out, const void *q_new,
                                   const void *k_new, const void *v_new, void *decode_out) {
    LayerArgs a{};
    zipvl_status status = check_layer("zipvl_layer_step_host", layer, &a);
    if (status != ZIPVL_OK) return status;
    if (!q || !k || !v || !probe_pos || n_probe < 1)
        return fail(ZIPVL_ERR_INVALID_ARG, "zipvl_layer_step_host: NULL input or n_probe < 1");
    if (layer->q_stride_tok || layer->kv_stride_tok)
        return fail(ZIPVL_ERR_UNSUPPORTED, "zipvl_layer_step_host: contiguous tensors only");
    const bool with_decode = (q_new != nullptr);
    if (with_decode && (!k_new || !v_new || !decode_out))
        return fail(ZIPVL_ERR_INVALID_ARG, "zipvl_layer_step_host: the decode step needs q_new, k_new, v_new and decode_out");
    if (with_decode && a.G > 8)
        return fail(ZIPVL_ERR_UNSUPPORTED, "zipvl_layer_step_host: more than 8 query heads per kv head");
    const size_t eb = elem_bytes(layer->dtype);
    const size_t qb = (size_t)a.L * a.Hq * a.D * eb, kb = (size_t)a.L * a.Hkv * a.D * eb;
    const size_t ws_score = zipvl_workspace_bytes(ZIPVL_OP_SCORE, layer, n_probe, 1);
    const size_t ws_pf = zipvl_workspace_bytes(ZIPVL_OP_SPARSE_PREFILL, layer, 0, 1);
    size_t ws_b = ws_score > ws_pf ? ws_score : ws_pf;
    if (ws_b < select_ws_bytes()) ws_b = select_ws_bytes();
    // the decode step runs on the cache this call has just compacted: capacity L + 1 rows
    const size_t ws_dec = with_decode ? align256(decode_ws_bytes(1, a.Hq, a.D, a.L + 1, a.Hkv, layer->dtype)) : 0;
    if (ws_b < ws_dec) ws_b = ws_dec;
    const size_t qn_b = (size_t)a.Hq * a.D * eb, kn_b = (size_t)a.Hkv * a.D * eb;
    // one stream-ordered allocation carved into pieces
    size_t off = 0;
    auto carve = [&](size_t bytes) { size_t o = off; off += align256(bytes); return o; };
    const size_t o_q = carve(qb), o_k = carve(kb), o_v = carve(kb), o_out = carve(qb),
                 o_kc = carve(kb + kn_b), o_vc = carve(kb + kn_b), o_probe = carve((size_t)n_probe * 4),
                 o_qn = carve(qn_b), o_kn = carve(kn_b), o_vn = carve(kn_b), o_dec = carve(qn_b),
                 o_acc = carve((size_t)a.L * 4), o_norm = carve((size_t)a.L * 4),
                 o_idx = carve((size_t)a.L * 4), o_misc = carve(256), o_ws = carve(ws_b);

    // what the GPU can read by itself
    const void *m_probe = mapped(probe_pos, (size_t)n_probe * 4);
    const void *m_q = m_probe ? mapped(q, qb) : nullptr;
    const void *m_new[3] = {with_decode ? mapped(q_new, qn_b) : nullptr, with_decode ? mapped(k_new, kn_b) : nullptr,
                            with_decode ? mapped(v_new, kn_b) : nullptr};
    // Groups of heads for Q and the output: pinned on both sides (a strided copy of pageable memory goes
    // row by row), whole kv heads, rows of 1 KB or more, 2 MB or more per copy.
    const bool tc = prefill_tc_supported(a, layer->dtype);
    int groups = (tc && m_q && (!out || mapped(out, qb))) ? kMaxGroups / 2 : 1;
    while (groups > 1 && (a.Hkv % groups || (size_t)(a.Hq / groups) * a.D * eb < 1024 || qb / groups < ((size_t)2 << 20)))
        groups /= 2;
    const int hn = a.Hq / groups;
    const size_t row_b = (size_t)a.Hq * a.D * eb, part_b = (size_t)hn * a.D * eb;

    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return fail(ZIPVL_ERR_CUDA, "zipvl_layer_step_host: no current device");
    HostContext c;
    cudaMemPool_t pool = nullptr;
    char *base = nullptr;
    ZIPVL_CUDA(host_pool(dev, &pool));
    ZIPVL_CUDA(take_context(dev, &c));
    auto body = [&]() -> zipvl_status {
        ZIPVL_CUDA(cudaMallocFromPoolAsync((void **)&base, off, pool, c.run));
        ZIPVL_CUDA(cudaEventRecord(c.alloc, c.run));
        ZIPVL_CUDA(cudaStreamWaitEvent(c.in, c.alloc, 0));
        int32_t *d_misc = (int32_t *)(base + o_misc), *d_idx = (int32_t *)(base + o_idx);
        int32_t *d_probe = (int32_t *)(base + o_probe);
        auto up = [&](size_t o, const void *src, size_t bytes) {
            return cudaMemcpyAsync(base + o, src, bytes, cudaMemcpyHostToDevice, c.in);
        };
        // ---- in: what the token set depends on first
        const size_t o_new[3] = {o_qn, o_kn, o_vn}, new_b[3] = {qn_b, kn_b, kn_b};
        const void *p_new[3] = {q_new, k_new, v_new};
        SmallInputs si{};
        si.q = (const uint4 *)m_q;
        si.probe = (const int32_t *)m_probe;
        si.q_dev = (uint4 *)(base + o_q);
        si.probe_dev = d_probe;
        si.misc = d_misc;
        si.L = a.L; si.P = n_probe; si.cap = a.L + 1;
        si.q_chunks = (int)(row_b / 16);
        for (int i = 0; i < 3; ++i) {
            si.rows[i] = (const uint4 *)m_new[i];
            si.rows_dev[i] = (uint4 *)(base + o_new[i]);
            si.row_chunks[i] = (int)(new_b[i] / 16);
            if (with_decode && !m_new[i]) ZIPVL_CUDA(up(o_new[i], p_new[i], new_b[i]));
        }
        if (!m_probe) ZIPVL_CUDA(up(o_probe, probe_pos, (size_t)n_probe * 4));
        ZIPVL_CUDA(up(o_k, k, kb));
        if (!m_q) ZIPVL_CUDA(up(o_q, q, qb));
        ZIPVL_CUDA(cudaEventRecord(c.k_in, c.in));
        fetch_small_inputs_kernel<<<n_probe + 3, 256, 0, c.run>>>(si);
        count_launches(1);
        ZIPVL_CALL(check_launch("zipvl_layer_step_host"));
        ZIPVL_CUDA(cudaStreamWaitEvent(c.run, c.k_in, 0));
        // ---- run: token set
        ZIPVL_CALL(zipvl_score(layer, base + o_q, base + o_k, d_probe, n_probe, (float *)(base + o_acc),
                               (float *)(base + o_norm), nullptr, base + o_ws, ws_b, d_misc + 2, c.run));
        ZIPVL_CALL(zipvl_select(a.L, (float *)(base + o_acc), (float *)(base + o_norm), tau, 0, 0, d_misc, d_idx, nullptr,
                                base + o_ws, ws_b, d_misc + 2, c.run));
        ZIPVL_CUDA(cudaEventRecord(c.chosen, c.run));
        ZIPVL_CUDA(cudaStreamWaitEvent(c.out, c.chosen, 0));
        ZIPVL_CUDA(cudaMemcpyAsync(c.misc, d_misc, 16, cudaMemcpyDeviceToHost, c.out));
        ZIPVL_CUDA(cudaEventRecord(c.told, c.out));
        // ---- in: V, then Q by groups of heads.  The copies write the probe rows of Q again, so they wait for the kernels
        // that fetched and read them (which are done while V comes in, unless its heads are few)
        ZIPVL_CUDA(up(o_v, v, kb));
        ZIPVL_CUDA(cudaEventRecord(c.v_in, c.in));
        if (m_q) ZIPVL_CUDA(cudaStreamWaitEvent(c.in, c.chosen, 0));
        if (m_q)
            for (int g = 0; g < groups; ++g) {
                if (groups == 1) ZIPVL_CUDA(up(o_q, q, qb));
                else
                    ZIPVL_CUDA(cudaMemcpy2DAsync(base + o_q + g * part_b, row_b, (const char *)q + g * part_b, row_b, part_b,
                                                 a.L, cudaMemcpyHostToDevice, c.in));
                ZIPVL_CUDA(cudaEventRecord(c.q_in[g], c.in));
            }
        // ---- run: caches, decode step, attention group by group
        ZIPVL_CALL(launch_compact(a, (int)eb, base + o_k, nullptr, d_idx, d_misc, a.L, base + o_kc, nullptr, a.L, d_misc + 1,
                                  d_misc + 2, c.run));
        ZIPVL_CUDA(cudaEventRecord(c.k_kept, c.run));
        ZIPVL_CUDA(cudaStreamWaitEvent(c.run, c.v_in, 0));
        ZIPVL_CALL(launch_compact(a, (int)eb, base + o_v, nullptr, d_idx, d_misc, a.L, base + o_vc, nullptr, a.L, d_misc + 1,
                                  d_misc + 2, c.run));
        ZIPVL_CUDA(cudaEventRecord(c.v_kept, c.run));
        if (with_decode) {
            // Algorithm 2 on the cache just built: d_misc[1] holds its length, d_misc[3] its
            // capacity, d_misc + 4 (8-byte aligned) the one request's offset 0
            zipvl_decode_desc dd = {1, a.Hq, a.Hkv, a.D, layer->dtype, layer->softmax_scale};
            ZIPVL_CALL(zipvl_decode(&dd, base + o_qn, base + o_kn, base + o_vn, base + o_kc, base + o_vc,
                                    (const int64_t *)(d_misc + 4), d_misc + 3, d_misc + 1, a.L + 1, base + o_dec,
                                    base + o_ws, ws_b, d_misc + 2, c.run));
            ZIPVL_CUDA(cudaEventRecord(c.decoded, c.run));
        }
        for (int g = 0; g < groups; ++g) {
            if (m_q) ZIPVL_CUDA(cudaStreamWaitEvent(c.run, c.q_in[g], 0));
            a.h0 = g * hn;
            a.hn = hn;
            ZIPVL_CALL(tc ? launch_prefill_tc(a, base + o_q, base + o_k, base + o_v, d_idx, d_misc, a.L, base + o_out,
                                              ZIPVL_OUT_PADDED, nullptr, nullptr, 0, nullptr, base + o_ws, d_misc + 2, c.run)
                          : launch_prefill_simt(a, layer->dtype, base + o_q, base + o_k, base + o_v, d_idx, d_misc, a.L,
                                                base + o_out, ZIPVL_OUT_PADDED, nullptr, nullptr, 0, nullptr, d_misc + 2, c.run));
            ZIPVL_CUDA(cudaEventRecord(c.done[g], c.run));
        }
        // ---- out
        auto down = [&](void *dst, size_t o, size_t bytes) {
            return cudaMemcpyAsync(dst, base + o, bytes, cudaMemcpyDeviceToHost, c.out);
        };
        if (idx_out) ZIPVL_CUDA(down(idx_out, o_idx, (size_t)a.L * 4));
        ZIPVL_CUDA(cudaEventSynchronize(c.told));
        const int kept_rows = c.misc[0];
        const size_t kept = (size_t)(kept_rows < 0 ? 0 : kept_rows > a.L ? a.L : kept_rows) * a.Hkv * a.D * eb;
        ZIPVL_CUDA(cudaStreamWaitEvent(c.out, c.k_kept, 0));
        if (k_cache_out) ZIPVL_CUDA(down(k_cache_out, o_kc, kept));
        ZIPVL_CUDA(cudaStreamWaitEvent(c.out, c.v_kept, 0));
        if (v_cache_out) ZIPVL_CUDA(down(v_cache_out, o_vc, kept));
        if (with_decode) {
            ZIPVL_CUDA(cudaStreamWaitEvent(c.out, c.decoded, 0));
            ZIPVL_CUDA(down(decode_out, o_dec, qn_b));
        }
        for (int g = 0; g < groups; ++g) {
            ZIPVL_CUDA(cudaStreamWaitEvent(c.out, c.done[g], 0));
            if (!out) continue;
            if (groups == 1) ZIPVL_CUDA(down(out, o_out, qb));
            else
                ZIPVL_CUDA(cudaMemcpy2DAsync((char *)out + g * part_b, row_b, base + o_out + g * part_b, row_b, part_b, a.L,
                                             cudaMemcpyDeviceToHost, c.out));
        }
        ZIPVL_CUDA(cudaMemcpyAsync(c.misc, d_misc, 16, cudaMemcpyDeviceToHost, c.out));
        // (everything on `in` and `run` is in front of it; the free too is over when the call returns, so that
        // zipvl_release_host_scratch finds the memory in the pool)
        ZIPVL_CUDA(cudaFreeAsync(base, c.out));
        base = nullptr;
        ZIPVL_CUDA(cudaStreamSynchronize(c.out));
        if (k_out) *k_out = kept_rows;
        if (c.misc[2] != 0)
            return fail(c.misc[2] & ZIPVL_DEV_TIMEOUT ? ZIPVL_ERR_TIMEOUT : ZIPVL_ERR_BAD_INDEX,
                        "prefill_layer_host: device status word = %d", c.misc[2]);
        return ZIPVL_OK;
    };
    status = body();
    if (status != ZIPVL_OK) {                           // nothing may still be using the buffers
        for (cudaStream_t s : {c.in, c.run, c.out}) cudaStreamSynchronize(s);
        if (base) cudaFreeAsync(base, c.out);
        cudaStreamSynchronize(c.out);
    }
    give_context(dev, c);
    return status;
}

}  // extern "C"
