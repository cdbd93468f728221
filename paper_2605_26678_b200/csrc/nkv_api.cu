// C ABI of the nkv library: argument checking, workspace carving and launch order.
#include <math.h>
#include <new>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <cuda.h>

#include "nkv_common.cuh"
#include "nkv_hostrange.h"

using namespace nkv;

constexpr int kHostSlots = 4;   // staging slots of nkv_compress_host, a stream each

struct nkv_handle {
    int device;
    int sm_count;
    int64_t launches;
    int timing;
    int timing_valid;
    int key_pass;     // NKV_KEY_PASS_*: which kernels make the two key passes
    cudaEvent_t ev[NKV_NUM_STAGES + 1];
    cudaStream_t copy_streams[kHostSlots];
    int* chunk_status;   // pinned: the status code of every step of nkv_compress_host
    int64_t chunk_capacity;
    int64_t host_in, host_out;   // bytes that the last nkv_compress_host moved to the device and back
    int inject_status;   // tests: status code planted in chunk `inject_chunk` of nkv_compress_host
    int inject_chunk;
};

constexpr int64_t kHostSteps = 4096;   // steps of nkv_compress_host that the first status buffer holds

namespace {

constexpr size_t kAlign = 256;
size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

bool params_ok(const nkv_params* p) {
    if (!p) return false;
    if (p->n_sink < 0 || p->block_div < 1 || p->block_min < 1 || p->block_max < p->block_min) return false;
    if (!(p->top_frac > 0.0 && p->top_frac <= 1.0)) return false;
    // a prior of zero switches its scale off (the single-anchor and no-current ablations); one must remain
    double prior_sum = 0.0;
    for (int k = 0; k < 3; ++k) {
        if (!(p->prior[k] >= 0.0) || !isfinite(p->prior[k])) return false;
        prior_sum += p->prior[k];
    }
    if (!(prior_sum > 0.0)) return false;
    if (!isfinite(p->beta) || !isfinite(p->tau) || !isfinite(p->kappa)) return false;
    if (!(p->safeguard >= 0.0 && p->safeguard <= 1.0)) return false;
    if (p->gate_mode < NKV_GATE_SURPRISE || p->gate_mode > NKV_GATE_MAX) return false;
    return true;
}

int64_t block_size(int64_t N, const nkv_params* p) {
    int64_t b = N / p->block_div;
    if (b < p->block_min) b = p->block_min;
    if (b > p->block_max) b = p->block_max;
    return b;
}

int64_t keep_count(int64_t N, double r) { return (int64_t)floor((1.0 - r) * (double)N); }

// Workspace carving shared by every entry point.
struct Layout {
    size_t status, mm, inv_norm, mu_s, mu_e, inv_s, inv_e, a_raw, a_star, hist, total;
};

// Rows of the per-token arrays start on 16-byte boundaries, so that ragged lengths keep the four-wide accesses.
int64_t padded_row(int64_t N) { return (N + 3) & ~(int64_t)3; }

Layout make_layout(int64_t units, int64_t N, int64_t d, int64_t nb) {
    Layout L;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        size_t at = o;
        o += align_up(bytes);
        return at;
    };
    const size_t row = (size_t)padded_row(N) * 4;
    L.status = take(kStatusWords * sizeof(int));
    L.mm = take((size_t)units * 6 * 4);      // cleared together with the status words in front of it
    L.inv_norm = take((size_t)units * row);
    L.mu_s = take((size_t)units * d * 4);
    L.mu_e = take((size_t)units * nb * d * 4);
    L.inv_s = take((size_t)units * 4);
    L.inv_e = take((size_t)units * nb * 4);
    L.a_raw = take((size_t)units * 3 * row);
    L.a_star = take((size_t)units * row);
    L.hist = take(score_hist_bytes(units));
    L.total = o;
    return L;
}
size_t cleared_bytes(const Layout& L, int64_t units) { return L.mm + (size_t)units * 6 * 4; }

int check_tensor(const nkv_tensor* t) {
    if (!t || !t->ptr) return NKV_ERR_INVALID_ARG;
    if (t->dtype != NKV_BF16 && t->dtype != NKV_F32 && t->dtype != NKV_F16) return NKV_ERR_UNSUPPORTED;
    if (t->d != 64 && t->d != 128) return NKV_ERR_UNSUPPORTED;
    if (t->G < 1 || t->H < 1 || t->N < 1) return NKV_ERR_INVALID_ARG;
    if (t->N > (int64_t)1 << 24 || t->G * t->H > (int64_t)1 << 24) return NKV_ERR_UNSUPPORTED;
    if (t->stride_n != t->d) return NKV_ERR_UNSUPPORTED;
    const int64_t eb = t->dtype == NKV_F32 ? 4 : 2;
    if (t->stride_h < t->N * t->d || t->stride_g < t->H * t->N * t->d) {
        // strides may be permuted (for instance heads outermost); only require non-overlap of rows
        if (t->stride_h < 1 || t->stride_g < 1) return NKV_ERR_INVALID_ARG;
    }
    if (((uintptr_t)t->ptr) % 16 != 0 || (t->stride_h * eb) % 16 != 0 || (t->stride_g * eb) % 16 != 0)
        return NKV_ERR_INVALID_ARG;
    return NKV_OK;
}

// The bound that calls on keys have always had (heads once lay on gridDim.y).
int check_units(int64_t units) { return units > 65535 ? NKV_ERR_UNSUPPORTED : NKV_OK; }

TensorView view_of(const nkv_tensor* t) {
    TensorView v;
    v.ptr = t->ptr;
    v.stride_g = t->stride_g;
    v.stride_h = t->stride_h;
    v.H = (int)t->H;
    v.N = (int)t->N;
    v.d = (int)t->d;
    return v;
}

int resolve_params(const nkv_params* p, int64_t N, ScoreParams* sp) {
    if (!params_ok(p)) return NKV_ERR_INVALID_ARG;
    // W = 1 makes the current anchor the key itself: a_c is the constant -1 and its per-head min-max would
    // normalise rounding noise, so the smallest window is 2
    if (p->window < 2 || p->window > kMaxWindow) return NKV_ERR_UNSUPPORTED;
    sp->window = p->window;
    sp->n_sink = p->n_sink;
    sp->block = (int)block_size(N, p);
    sp->nblocks = (int)((N + sp->block - 1) / sp->block);
    sp->gate_mode = p->gate_mode;
    int64_t m = (int64_t)floor(p->top_frac * (double)N);
    sp->top_m = (int)(m < 1 ? 1 : m);
    for (int k = 0; k < 3; ++k) sp->log_prior[k] = (float)log(p->prior[k]);
    sp->beta = (float)p->beta;
    sp->tau = (float)p->tau;
    sp->kappa = (float)p->kappa;
    sp->raw_row = sp->inv_row = padded_row(N);   // in the workspace
    return NKV_OK;
}

int check_ws(const void* ws, size_t ws_bytes, size_t need) {
    if (!ws || ((uintptr_t)ws) % kAlign != 0 || ws_bytes < need) return NKV_ERR_WORKSPACE;
    return NKV_OK;
}

template <typename T>
T* at(void* ws, size_t off) { return reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(ws) + off); }

// With NKV_TRACE set in the environment a failing CUDA call is named on stderr.  The call's error does not stay behind as the
// runtime's last one: launches that ask for it would take it for theirs.
int cuda_failed(cudaError_t e, const char* what, int line) {
    cudaGetLastError();
    static const bool trace = getenv("NKV_TRACE") != nullptr;
    if (trace) fprintf(stderr, "nkv: %s (nkv_api.cu:%d): %s\n", what, line, cudaGetErrorString(e));
    return NKV_ERR_CUDA;
}

#define CU(expr)                                                     \
    do {                                                             \
        cudaError_t e__ = (expr);                                    \
        if (e__ != cudaSuccess) return cuda_failed(e__, #expr, __LINE__); \
    } while (0)

// The workspace arrays of the key passes.
struct Bufs {
    float *inv_norm, *mu_s, *mu_e, *inv_s, *inv_e, *a_raw;
    uint32_t* mm;
};
Bufs bufs_at(void* ws, const Layout& L) {
    Bufs b;
    b.inv_norm = at<float>(ws, L.inv_norm);
    b.mu_s = at<float>(ws, L.mu_s);
    b.mu_e = at<float>(ws, L.mu_e);
    b.inv_s = at<float>(ws, L.inv_s);
    b.inv_e = at<float>(ws, L.inv_e);
    b.a_raw = at<float>(ws, L.a_raw);
    b.mm = at<uint32_t>(ws, L.mm);
    return b;
}

// Whether the tensor form of a key pass is the better one where both are there.  It is bound by the read of the keys (the
// first pass: by half the FMA form's instructions), but its roles take 1 to 2 us longer to get going.  Whole calls with both
// passes in the FMA form / the second / none, H = 8, r = 0.75, bf16, us:
//     d = 64    17 MB of keys 52 / 54 / 56   33 MB 69 / 70 / 69   67 MB 106 / 100 / 99 (64 x 8192), 99 / 102 / 102 (128 x 4096)
//     d = 128   17 MB 53 / 54 / 54           33 MB 66 / 62 / 62   67 MB 98 / 84 / 84
// With keys that are not in L2, 41 MB of 16 x 8 x 2500 x 64 at r = 0.5: 84.7 with the second pass in FMA form, 85.5 with none.
// (For d = 64 the two forms of the second pass are within a percent or two of each other from 33 to 67 MB: where its line lies
// between them matters little.)
constexpr int kFirstPassKb = 192, kSecondPassKb64 = 320, kSecondPassKb128 = 192;   // of keys per SM
bool tensor_pays(const nkv_handle* h, const TensorView& kv, int G, const ScoreParams& sp, int kb) {
    const int64_t bytes = (int64_t)G * kv.H * kv.N * kv.d * 2;
    return h->key_pass == NKV_KEY_PASS_TENSOR || !stream_path_supported(sp) || bytes >= (int64_t)h->sm_count * kb * 1024;
}

// The second pass over the keys: a_s and a_e of every token from the anchors.
int anchor_scores(nkv_handle* h, const TensorView& kv, int dtype, int G, const ScoreParams& sp, const float* mu_s, const float* mu_e,
                  const float* inv_norm, const Bufs& B, float* a_raw, int* status, cudaStream_t st) {
    const bool tensor = h->key_pass != NKV_KEY_PASS_FMA && tensor_pays(h, kv, G, sp, kv.d == 64 ? kSecondPassKb64 : kSecondPassKb128) &&
                        anchor_dots_supported(kv, dtype, sp);
    if (tensor)
        CU(launch_anchor_dots(kv, dtype, G, sp, mu_s, mu_e, inv_norm, B.inv_s, B.inv_e, a_raw, B.mm, status, h->sm_count, st,
                              &h->launches));
    else
        CU(launch_stream_b(kv, dtype, G, sp, mu_s, mu_e, inv_norm, B.inv_s, B.inv_e, a_raw, B.mm, status, h->sm_count, st,
                           &h->launches));
    return NKV_OK;
}

// The two passes over the keys (Sections 2.1-2.3): afterwards the workspace holds 1/||k||, the anchors, the
// three raw anomalies and their per-head min/max keys (which start out cleared).  `mark` is called once between the passes (stage
// timing).
template <typename Mark>
int key_scan(nkv_handle* h, const TensorView& kv, int dtype, int G, const ScoreParams& sp, const Bufs& B, int* status,
             cudaStream_t st, Mark&& mark) {
    const int units = G * kv.H, N = kv.N, d = kv.d;
    // (sizes first: the other two encode a tensor map to ask the driver, which a call that small does not need)
    const bool tensor_a = h->key_pass != NKV_KEY_PASS_FMA && tensor_pays(h, kv, G, sp, kFirstPassKb) &&
                          gram_pass_supported(kv, dtype, sp) && anchor_dots_supported(kv, dtype, sp);
    if (!tensor_a && !stream_path_supported(sp)) {
        CU(launch_anchor_sums(kv, dtype, G, sp, B.mu_e, B.inv_norm, st, &h->launches));
        CU(launch_anchor_means(units, N, d, sp, B.mu_e, B.mu_s, B.inv_e, B.inv_s, st, &h->launches));
        CU(mark());
        CU(launch_scan_scores(kv, dtype, G, sp, B.mu_s, B.mu_e, B.inv_norm, B.inv_s, B.inv_e, B.a_raw, B.mm, st,
                              &h->launches));
        return NKV_OK;
    }
    // pass A: norms, block sums and the current-memory anomaly; pass B: the two anchor anomalies
    if (tensor_a)
        CU(launch_gram_pass(kv, dtype, G, sp, nullptr, B.mu_e, B.inv_norm, B.a_raw, B.mm, status, h->sm_count, st, &h->launches));
    else
        CU(launch_stream_a(kv, dtype, G, sp, B.mu_e, B.inv_norm, B.a_raw, B.mm, status, h->sm_count, st, &h->launches));
    CU(launch_anchor_means(units, N, d, sp, B.mu_e, B.mu_s, B.inv_e, B.inv_s, st, &h->launches));
    CU(mark());
    return anchor_scores(h, kv, dtype, G, sp, B.mu_s, B.mu_e, B.inv_norm, B, B.a_raw, status, st);
}

// Staging of nkv_compress_host: the groups of a chunk are halved where possible, so that twice as many slots keep the
// copy engines busy in both directions while kernels run.
constexpr int kHostGatherCtas = 32;
constexpr double kHostRowsShare = 0.6;
struct HostSlot {
    size_t K, V, K_out, V_out, idx, offsets, budgets, ws, total;
};
struct HostPlan {
    int64_t groups;   // per slot
    int slots;
    HostSlot slot;
};
HostSlot host_slot(int64_t c, int64_t H, int64_t N, int64_t d, int dtype, int64_t keep, const nkv_params* params) {
    const size_t eb = dtype == NKV_F32 ? 4 : 2;
    const int64_t b = block_size(N, params);
    HostSlot s;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += align_up(bytes);
        return at;
    };
    s.K = take((size_t)c * H * N * d * eb);
    s.V = take((size_t)c * H * N * d * eb);
    s.K_out = take((size_t)c * H * keep * d * eb);
    s.V_out = take((size_t)c * H * keep * d * eb);
    s.idx = take((size_t)c * H * keep * 4);
    s.offsets = take((size_t)c * (H + 1) * 4);
    s.budgets = take((size_t)c * H * 4);
    s.ws = o;
    s.total = o + make_layout(c * H, N, d, (N + b - 1) / b).total;
    return s;
}
HostPlan host_plan(int64_t H, int64_t N, int64_t d, int dtype, int64_t keep, const nkv_params* params, int64_t groups_per_chunk) {
    HostPlan p;
    p.slots = groups_per_chunk >= 2 ? kHostSlots : 2;
    p.groups = groups_per_chunk >= 2 ? groups_per_chunk / 2 : 1;
    p.slot = host_slot(p.groups, H, N, d, dtype, keep, params);
    return p;
}

// The address at which the current device reads [p, p + bytes) of host memory in place; null when it cannot.
const void* device_address(const void* p, size_t bytes) {
    return readable_in_place(p, bytes, [](const void* q, HostRange* r) {
        using GetAttribute = CUresult (*)(void*, CUpointer_attribute, CUdeviceptr);
        static const GetAttribute attribute = [] {   // looked up once (the library does not link against the driver)
            void* f = nullptr;
            cudaDriverEntryPointQueryResult found;
            if (cudaGetDriverEntryPoint("cuPointerGetAttribute", &f, cudaEnableDefault, &found) != cudaSuccess ||
                found != cudaDriverEntryPointSuccess)
                f = nullptr;
            return reinterpret_cast<GetAttribute>(f);
        }();
        cudaPointerAttributes a;
        if (cudaPointerGetAttributes(&a, q) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        if (!attribute || a.type != cudaMemoryTypeHost || !a.devicePointer) return false;
        CUdeviceptr start = 0;
        size_t size = 0;
        const CUdeviceptr at = reinterpret_cast<CUdeviceptr>(a.devicePointer);
        if (attribute(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, at) != CUDA_SUCCESS ||
            attribute(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, at) != CUDA_SUCCESS)
            return false;
        *r = {static_cast<const unsigned char*>(a.devicePointer), static_cast<uintptr_t>(start), size};
        return true;
    });
}

// ordered min/max keys -> floats (lo_s, hi_s, lo_e, hi_e, lo_c, hi_c per head)
__global__ void minmax_floats_kernel(int n, const uint32_t* keys, float* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = ord_float((i & 1) ? keys[i] : ~keys[i]);
}

}  // namespace

extern "C" {

const char* nkv_version(void) { return "nkv 0.1 (sm_100a)"; }

const char* nkv_status_string(int status) {
    switch (status) {
        case NKV_OK: return "ok";
        case NKV_ERR_INVALID_ARG: return "invalid argument";
        case NKV_ERR_UNSUPPORTED: return "unsupported dtype, head_dim, window or layout";
        case NKV_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case NKV_ERR_CUDA: return "CUDA runtime error";
        case NKV_ERR_TIMEOUT: return "device-side bounded wait ran out";
        case NKV_ERR_DEVICE_CHECK: return "device-side self-check failed";
        default: return "unknown status";
    }
}

int nkv_default_params(nkv_params* p) {
    if (!p) return NKV_ERR_INVALID_ARG;
    p->window = 64;
    p->n_sink = 4;
    p->block_div = 32;
    p->block_min = 128;
    p->block_max = 256;
    p->gate_mode = NKV_GATE_SURPRISE;
    p->top_frac = 0.10;
    p->prior[0] = 0.4;
    p->prior[1] = 0.4;
    p->prior[2] = 0.2;
    p->beta = 3.0;
    p->tau = 0.60;
    p->kappa = 10.0;
    p->safeguard = 0.20;
    return NKV_OK;
}

int64_t nkv_block_size(int64_t N, const nkv_params* p) {
    if (N < 1 || !params_ok(p)) return -1;
    return block_size(N, p);
}
int64_t nkv_num_blocks(int64_t N, const nkv_params* p) {
    if (N < 1 || !params_ok(p)) return -1;
    const int64_t b = block_size(N, p);
    return (N + b - 1) / b;
}
int64_t nkv_keep_per_head(int64_t N, double r) {
    if (N < 1 || !(r >= 0.0 && r < 1.0)) return -1;
    return keep_count(N, r);
}
int64_t nkv_safeguard_count(int64_t N, double r, const nkv_params* p) {
    if (N < 1 || !(r >= 0.0 && r < 1.0) || !params_ok(p)) return -1;
    const int64_t k = keep_count(N, r);
    int64_t s = (int64_t)floor(p->safeguard * (double)k);
    return s > k ? k : s;
}
int64_t nkv_top_count(int64_t N, const nkv_params* p) {
    if (N < 1 || !params_ok(p)) return -1;
    int64_t m = (int64_t)floor(p->top_frac * (double)N);
    return m < 1 ? 1 : m;
}

int nkv_create(nkv_handle** out, int device) {
    if (!out) return NKV_ERR_INVALID_ARG;
    *out = nullptr;
    int count = 0, previous = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || device < 0 || device >= count) return NKV_ERR_CUDA;
    CU(cudaGetDevice(&previous));
    CU(cudaSetDevice(device));
    struct Restore {   // the caller's current device is left as it was
        int dev;
        ~Restore() { cudaSetDevice(dev); }
    } restore{previous};
    nkv_handle* h = new (std::nothrow) nkv_handle();
    if (!h) return NKV_ERR_INVALID_ARG;
    memset(h, 0, sizeof(*h));
    h->device = device;
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) {
        delete h;
        return NKV_ERR_CUDA;
    }
    h->sm_count = prop.multiProcessorCount;
    h->key_pass = NKV_KEY_PASS_AUTO;
    if (configure_scan_kernels() != cudaSuccess || configure_stream_kernels() != cudaSuccess ||
        configure_gram_kernels() != cudaSuccess ||
        configure_dots_kernels() != cudaSuccess || configure_select_kernels() != cudaSuccess) {
        delete h;
        return NKV_ERR_CUDA;
    }
    for (int i = 0; i <= NKV_NUM_STAGES; ++i)
        if (cudaEventCreate(&h->ev[i]) != cudaSuccess) {
            delete h;
            return NKV_ERR_CUDA;
        }
    if (cudaMallocHost(reinterpret_cast<void**>(&h->chunk_status), kHostSteps * sizeof(int)) != cudaSuccess) {
        delete h;
        return NKV_ERR_CUDA;
    }
    h->chunk_capacity = kHostSteps;
    for (int i = 0; i < kHostSlots; ++i) {
        if (cudaStreamCreateWithFlags(&h->copy_streams[i], cudaStreamNonBlocking) != cudaSuccess) {
            delete h;
            return NKV_ERR_CUDA;
        }
    }
    *out = h;
    return NKV_OK;
}

int nkv_destroy(nkv_handle* h) {
    if (!h) return NKV_ERR_INVALID_ARG;
    for (int i = 0; i <= NKV_NUM_STAGES; ++i) cudaEventDestroy(h->ev[i]);
    for (int i = 0; i < kHostSlots; ++i) cudaStreamDestroy(h->copy_streams[i]);
    cudaFreeHost(h->chunk_status);
    delete h;
    return NKV_OK;
}

int nkv_workspace_bytes(const nkv_handle* h, int64_t G, int64_t H, int64_t N, int64_t d, int32_t dtype,
                        const nkv_params* params, size_t* out_bytes) {
    (void)dtype;
    if (!h || !out_bytes || G < 1 || H < 1 || N < 1 || d < 1 || !params_ok(params)) return NKV_ERR_INVALID_ARG;
    const int64_t b = block_size(N, params);
    *out_bytes = make_layout(G * H, N, d, (N + b - 1) / b).total;
    return NKV_OK;
}

int nkv_anchors(nkv_handle* h, const nkv_tensor* K, const nkv_params* params, float* mu_s, float* mu_e,
                float* inv_norm, float* mu_c_opt, void* ws, size_t ws_bytes, void* stream) {
    if (!h || !mu_s || !mu_e || !inv_norm) return NKV_ERR_INVALID_ARG;
    int rc = check_tensor(K);
    if (rc) return rc;
    ScoreParams sp;
    if ((rc = resolve_params(params, K->N, &sp))) return rc;
    if ((rc = check_ws(ws, ws_bytes, align_up(kStatusWords * sizeof(int))))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const TensorView kv = view_of(K);
    const int units = (int)(K->G * K->H);
    sp.inv_row = K->N;
    CU(launch_anchor_sums(kv, K->dtype, (int)K->G, sp, mu_e, inv_norm, st, &h->launches));
    CU(launch_anchor_means(units, (int)K->N, (int)K->d, sp, mu_e, mu_s, nullptr, nullptr, st, &h->launches));
    if (mu_c_opt) CU(launch_window_means(kv, K->dtype, (int)K->G, sp, inv_norm, mu_c_opt, st, &h->launches));
    return NKV_OK;
}

int nkv_score(nkv_handle* h, const nkv_tensor* K, const float* mu_s, const float* mu_e, const float* inv_norm,
              const nkv_params* params, float* a_raw_opt, float* a_star, float* head_stats_opt, void* ws,
              size_t ws_bytes, void* stream) {
    if (!h || !mu_s || !mu_e || !inv_norm || !a_star) return NKV_ERR_INVALID_ARG;
    int rc = check_tensor(K);
    if (rc) return rc;
    if ((rc = check_units(K->G * K->H))) return rc;
    ScoreParams sp;
    if ((rc = resolve_params(params, K->N, &sp))) return rc;
    const int units = (int)(K->G * K->H);
    const Layout L = make_layout(units, K->N, K->d, sp.nblocks);
    if ((rc = check_ws(ws, ws_bytes, L.total))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const TensorView kv = view_of(K);
    sp.inv_row = K->N;
    if (a_raw_opt) sp.raw_row = K->N;
    float* a_raw = a_raw_opt ? a_raw_opt : at<float>(ws, L.a_raw);
    CU(cudaMemsetAsync(ws, 0, cleared_bytes(L, units), st));
    const Bufs B = bufs_at(ws, L);
    const int G = (int)K->G;
    CU(launch_anchor_norms(units, (int)K->d, sp, mu_s, mu_e, B.inv_s, B.inv_e, st, &h->launches));
    // two passes on the tensor cores against one that keeps a window sum per lane group: 58 + 56 us against 257 at
    // 28 x 8 heads of 4133 x 128 bf16 keys
    if (h->key_pass != NKV_KEY_PASS_FMA && gram_pass_supported(kv, K->dtype, sp) && anchor_dots_supported(kv, K->dtype, sp)) {
        CU(launch_gram_pass(kv, K->dtype, G, sp, inv_norm, nullptr, nullptr, a_raw, B.mm, at<int>(ws, L.status), h->sm_count, st,
                            &h->launches));
        if ((rc = anchor_scores(h, kv, K->dtype, G, sp, mu_s, mu_e, inv_norm, B, a_raw, at<int>(ws, L.status), st))) return rc;
    } else {
        CU(launch_scan_scores(kv, K->dtype, G, sp, mu_s, mu_e, inv_norm, B.inv_s, B.inv_e, a_raw, B.mm, st, &h->launches));
    }
    CU(launch_head_scores(units, (int)K->N, sp, a_raw, at<uint32_t>(ws, L.mm), a_star, head_stats_opt,
                          at<int>(ws, L.status), st, &h->launches));
    return NKV_OK;
}

int nkv_budget(nkv_handle* h, const float* a_star, int64_t G, int64_t H, int64_t N, double r,
               const nkv_params* params, int32_t* budgets, float* thresholds_opt, void* ws, size_t ws_bytes,
               void* stream) {
    if (!h || !a_star || !budgets || G < 1 || H < 1 || N < 1 || !params_ok(params)) return NKV_ERR_INVALID_ARG;
    if (!(r >= 0.0 && r < 1.0)) return NKV_ERR_INVALID_ARG;
    if (H > 64 || N > (int64_t)1 << 24 || H * N > (int64_t)1 << 30) return NKV_ERR_UNSUPPORTED;
    const int64_t k = keep_count(N, r);
    if (k < 1 || k > N) return NKV_ERR_INVALID_ARG;
    const int64_t n_safe = nkv_safeguard_count(N, r, params);
    int rc = check_ws(ws, ws_bytes, align_up(kStatusWords * sizeof(int)) + align_up((size_t)G * H * 8));
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    CU(cudaMemsetAsync(ws, 0, kStatusWords * sizeof(int), st));
    CU(launch_budget((int)G, (int)H, (int)N, (int)k, (int)n_safe, a_star, budgets, thresholds_opt, at<int>(ws, 0), st,
                     &h->launches));
    return NKV_OK;
}

int nkv_select(nkv_handle* h, const float* a_star, const int32_t* budgets, int64_t G, int64_t H, int64_t N,
               int64_t idx_capacity, int32_t* idx, int32_t* head_offsets, int32_t* ranks_opt, void* ws,
               size_t ws_bytes, void* stream) {
    if (!h || !a_star || !budgets || !idx || !head_offsets || G < 1 || H < 1 || N < 1 || idx_capacity < 1)
        return NKV_ERR_INVALID_ARG;
    if (N > (int64_t)1 << 24 || G * H > (int64_t)1 << 24) return NKV_ERR_UNSUPPORTED;
    int rc = check_ws(ws, ws_bytes, align_up(kStatusWords * sizeof(int)));
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    CU(cudaMemsetAsync(ws, 0, kStatusWords * sizeof(int), st));
    CU(launch_select((int)G, (int)H, (int)N, idx_capacity, a_star, budgets, idx, head_offsets, at<int>(ws, 0), st,
                     &h->launches));
    if (ranks_opt) {
        if (G * H > 65535) return NKV_ERR_UNSUPPORTED;
        CU(launch_ranks((int)(G * H), (int)N, a_star, ranks_opt, st, &h->launches));
    }
    return NKV_OK;
}

int nkv_compact(nkv_handle* h, const nkv_tensor* K, const nkv_tensor* V, const int32_t* idx,
                const int32_t* head_offsets, int64_t idx_capacity, void* K_out, void* V_out, int32_t mode, void* ws,
                size_t ws_bytes, void* stream) {
    (void)ws;
    (void)ws_bytes;
    if (!h || !idx || !head_offsets || idx_capacity < 1) return NKV_ERR_INVALID_ARG;
    int rc = check_tensor(K);
    if (rc) return rc;
    if ((rc = check_tensor(V))) return rc;
    if (V->G != K->G || V->H != K->H || V->N != K->N) return NKV_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int kb = K->dtype == NKV_F32 ? 4 : 2, vb = V->dtype == NKV_F32 ? 4 : 2;
    if (mode == NKV_OUT_OF_PLACE) {
        if (!K_out || !V_out || ((uintptr_t)K_out) % 16 || ((uintptr_t)V_out) % 16) return NKV_ERR_INVALID_ARG;
        CU(launch_gather(view_of(K), kb, view_of(V), vb, (int)K->G, idx, head_offsets, idx_capacity, K_out, V_out,
                         0, st, &h->launches));
    } else if (mode == NKV_IN_PLACE) {
        if (K_out || V_out) return NKV_ERR_INVALID_ARG;
        CU(launch_gather_in_place(view_of(K), kb, view_of(V), vb, (int)K->G, idx, head_offsets, idx_capacity, st,
                                  &h->launches));
    } else {
        return NKV_ERR_INVALID_ARG;
    }
    return NKV_OK;
}

// `host_v`: V lies in host memory that the device can read; its retained rows are fetched over the bus from there.
static int compress(nkv_handle* h, const nkv_tensor* K, const nkv_tensor* V, double r, const nkv_params* params, void* K_out,
                    void* V_out, int32_t* idx, int32_t* head_offsets, int32_t* budgets, float* a_star_opt, void* ws,
                    size_t ws_bytes, cudaStream_t st, bool host_v) {
    if (!h || !K_out || !V_out || !idx || !head_offsets || !budgets) return NKV_ERR_INVALID_ARG;
    int rc = check_tensor(K);
    if (rc) return rc;
    if ((rc = check_tensor(V))) return rc;
    if (V->G != K->G || V->H != K->H || V->N != K->N) return NKV_ERR_INVALID_ARG;
    if (!(r >= 0.0 && r < 1.0)) return NKV_ERR_INVALID_ARG;
    if (K->H > 64 || K->H * K->N > (int64_t)1 << 30) return NKV_ERR_UNSUPPORTED;
    if ((rc = check_units(K->G * K->H))) return rc;
    if (((uintptr_t)K_out) % 16 || ((uintptr_t)V_out) % 16) return NKV_ERR_INVALID_ARG;
    ScoreParams sp;
    if ((rc = resolve_params(params, K->N, &sp))) return rc;
    const int64_t keep = keep_count(K->N, r);
    if (keep < 1 || keep > K->N) return NKV_ERR_INVALID_ARG;
    const int64_t n_safe = nkv_safeguard_count(K->N, r, params);
    const int G = (int)K->G, H = (int)K->H, N = (int)K->N, d = (int)K->d;
    const int units = G * H;
    const Layout L = make_layout(units, N, d, sp.nblocks);
    if ((rc = check_ws(ws, ws_bytes, L.total))) return rc;
    const TensorView kv = view_of(K), vv = view_of(V);
    const int kb = K->dtype == NKV_F32 ? 4 : 2, vb = V->dtype == NKV_F32 ? 4 : 2;
    float* a_star = a_star_opt ? a_star_opt : at<float>(ws, L.a_star);
    const int64_t star_row = a_star_opt ? N : padded_row(N);
    int* status = at<int>(ws, L.status);
    const bool timing = h->timing != 0;
    int stage = 0;
    auto mark = [&]() -> cudaError_t {
        if (!timing) return cudaSuccess;
        return cudaEventRecord(h->ev[stage++], st);
    };

    CU(cudaMemsetAsync(ws, 0, cleared_bytes(L, units), st));
    CU(mark());
    const Bufs B = bufs_at(ws, L);
    if ((rc = key_scan(h, kv, K->dtype, G, sp, B, status, st, mark))) return rc;
    CU(mark());
    CU(launch_score_to_select(G, H, N, sp, (int)keep, (int)n_safe, B.a_raw, B.mm, a_star, star_row, at<int>(ws, L.hist), budgets, idx,
                              (int64_t)H * keep, head_offsets, status, st, &h->launches));
    CU(mark());
    CU(mark());   // the budget and select stages are part of that call
    CU(mark());
    CU(launch_gather(kv, kb, vv, vb, G, idx, head_offsets, (int64_t)H * keep, K_out, host_v ? nullptr : V_out, 0, st,
                     &h->launches));
    // a few CTAs keep more reads on the bus than it takes to fill it, and leave the SMs to the kernels of other chunks
    if (host_v)
        CU(launch_gather(kv, kb, vv, vb, G, idx, head_offsets, (int64_t)H * keep, nullptr, V_out, kHostGatherCtas, st,
                         &h->launches));
    CU(mark());
    if (timing) h->timing_valid = 1;
    return NKV_OK;
}

int nkv_compress(nkv_handle* h, const nkv_tensor* K, const nkv_tensor* V, double r, const nkv_params* params,
                 void* K_out, void* V_out, int32_t* idx, int32_t* head_offsets, int32_t* budgets,
                 float* a_star_opt, void* ws, size_t ws_bytes, void* stream) {
    return compress(h, K, V, r, params, K_out, V_out, idx, head_offsets, budgets, a_star_opt, ws, ws_bytes, (cudaStream_t)stream,
                    false);
}

int nkv_host_staging_bytes(const nkv_handle* h, int64_t H, int64_t N, int64_t d, int32_t dtype, double r,
                           const nkv_params* params, int64_t groups_per_chunk, size_t* out_bytes) {
    if (!h || !out_bytes || H < 1 || N < 1 || d < 1 || groups_per_chunk < 1 || !params_ok(params))
        return NKV_ERR_INVALID_ARG;
    if (!(r >= 0.0 && r < 1.0)) return NKV_ERR_INVALID_ARG;
    const int64_t keep = keep_count(N, r);
    if (keep < 1) return NKV_ERR_INVALID_ARG;
    const HostPlan p = host_plan(H, N, d, dtype, keep, params, groups_per_chunk);
    *out_bytes = p.slots * p.slot.total;
    return NKV_OK;
}

int nkv_compress_host(nkv_handle* h, const nkv_tensor* Kh, const nkv_tensor* Vh, double r, const nkv_params* params,
                      void* K_out_host, void* V_out_host, int32_t* idx_host, int32_t* head_offsets_host,
                      int32_t* budgets_host, int64_t groups_per_chunk, void* dev, size_t dev_bytes) {
    if (!h || !K_out_host || !V_out_host || !idx_host || !head_offsets_host || !budgets_host) return NKV_ERR_INVALID_ARG;
    int rc = check_tensor(Kh);
    if (rc) return rc;
    if ((rc = check_tensor(Vh))) return rc;
    if (Vh->G != Kh->G || Vh->H != Kh->H || Vh->N != Kh->N || Vh->d != Kh->d || Vh->dtype != Kh->dtype)
        return NKV_ERR_INVALID_ARG;
    // the host path copies whole groups: require densely packed groups
    if (Kh->stride_h != Kh->N * Kh->d || Kh->stride_g != Kh->H * Kh->N * Kh->d || Vh->stride_h != Kh->stride_h ||
        Vh->stride_g != Kh->stride_g)
        return NKV_ERR_UNSUPPORTED;
    size_t need = 0;
    if ((rc = nkv_host_staging_bytes(h, Kh->H, Kh->N, Kh->d, Kh->dtype, r, params, groups_per_chunk, &need))) return rc;
    if ((rc = check_ws(dev, dev_bytes, need))) return rc;
    const int64_t G = Kh->G, H = Kh->H, N = Kh->N, d = Kh->d;
    const int64_t keep = keep_count(N, r);
    const size_t eb = Kh->dtype == NKV_F32 ? 4 : 2;
    const HostPlan p = host_plan(H, N, d, Kh->dtype, keep, params, groups_per_chunk);
    const size_t grp_in = (size_t)H * N * d * eb, grp_out = (size_t)H * keep * d * eb;
    // Only the retained rows of V are needed on the device.  Where the device can read V in place (pinned memory) the
    // gather kernel fetches them from there, which spares the bus the others.  16 x 8 heads of 8192 x 64 bf16 keys: with
    // a quarter of the rows kept 5.34 -> 3.52 ms, with half 5.67 -> 4.92, with three quarters 6.06 -> 6.60, where one
    // copy is the better way; the two meet between 0.6 and 0.7 of the rows.  The same with rows of 256 and
    // 512 bytes: half of the rows kept 9.79 / 11.35 and 18.9 / 22.3 ms, 0.6 of them 11.05 / 11.58 and 21.5 / 22.8, 0.7 12.29 / 11.78
    // and 23.9 / 23.2 (in place / copied).
    const void* v_mapped = (double)keep <= kHostRowsShare * (double)N ? device_address(Vh->ptr, (size_t)G * grp_in) : nullptr;

    const int64_t steps = (G + p.groups - 1) / p.groups;
    if (steps > h->chunk_capacity) {
        int* more = nullptr;
        CU(cudaMallocHost(reinterpret_cast<void**>(&more), steps * sizeof(int)));
        cudaFreeHost(h->chunk_status);
        h->chunk_status = more;
        h->chunk_capacity = steps;
    }

    h->host_in = G * (int64_t)(grp_in + (v_mapped ? grp_out : grp_in));
    h->host_out = G * (int64_t)(2 * grp_out + (H * keep + 2 * H + 1) * 4);
    int result = NKV_OK;
    int64_t step = 0;
    for (int64_t g0 = 0; g0 < G && result == NKV_OK; g0 += p.groups, ++step) {
        cudaStream_t st = h->copy_streams[step % p.slots];
        const int64_t gc = (G - g0 < p.groups) ? (G - g0) : p.groups;
        unsigned char* base = reinterpret_cast<unsigned char*>(dev) + (size_t)(step % p.slots) * p.slot.total;
        unsigned char *dK = base + p.slot.K, *dV = base + p.slot.V, *dKo = base + p.slot.K_out, *dVo = base + p.slot.V_out;
        int32_t* dIdx = reinterpret_cast<int32_t*>(base + p.slot.idx);
        int32_t* dOff = reinterpret_cast<int32_t*>(base + p.slot.offsets);
        int32_t* dBud = reinterpret_cast<int32_t*>(base + p.slot.budgets);
        void* dWs = base + p.slot.ws;
        // the slot's previous groups finished all their copies before this stream reaches here (same stream)
        if (cudaMemcpyAsync(dK, (const unsigned char*)Kh->ptr + g0 * grp_in, gc * grp_in, cudaMemcpyHostToDevice, st) !=
                cudaSuccess ||
            (!v_mapped && cudaMemcpyAsync(dV, (const unsigned char*)Vh->ptr + g0 * grp_in, gc * grp_in, cudaMemcpyHostToDevice,
                                          st) != cudaSuccess)) {
            result = NKV_ERR_CUDA;
            break;
        }
        nkv_tensor dk = *Kh, dv = *Vh;
        dk.ptr = dK;
        dv.ptr = v_mapped ? const_cast<unsigned char*>((const unsigned char*)v_mapped) + g0 * grp_in : dV;
        dk.G = dv.G = gc;
        rc = compress(h, &dk, &dv, r, params, dKo, dVo, dIdx, dOff, dBud, nullptr, dWs, p.slot.total - p.slot.ws, st,
                      v_mapped != nullptr);
        if (rc) {
            result = rc;
            break;
        }
        if (h->inject_status && g0 / groups_per_chunk == h->inject_chunk &&
            cudaMemcpyAsync(dWs, &h->inject_status, sizeof(int), cudaMemcpyHostToDevice, st) != cudaSuccess) {
            result = NKV_ERR_CUDA;
            break;
        }
        if (cudaMemcpyAsync((unsigned char*)K_out_host + g0 * grp_out, dKo, gc * grp_out, cudaMemcpyDeviceToHost, st) !=
                cudaSuccess ||
            cudaMemcpyAsync((unsigned char*)V_out_host + g0 * grp_out, dVo, gc * grp_out, cudaMemcpyDeviceToHost, st) !=
                cudaSuccess ||
            cudaMemcpyAsync(idx_host + g0 * H * keep, dIdx, gc * H * keep * 4, cudaMemcpyDeviceToHost, st) !=
                cudaSuccess ||
            cudaMemcpyAsync(head_offsets_host + g0 * (H + 1), dOff, gc * (H + 1) * 4, cudaMemcpyDeviceToHost, st) !=
                cudaSuccess ||
            cudaMemcpyAsync(budgets_host + g0 * H, dBud, gc * H * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaMemcpyAsync(h->chunk_status + step, static_cast<int*>(dWs) + kStatusCode, sizeof(int), cudaMemcpyDeviceToHost, st) !=
                cudaSuccess) {
            result = NKV_ERR_CUDA;
            break;
        }
    }
    for (int i = 0; i < kHostSlots; ++i)
        if (cudaStreamSynchronize(h->copy_streams[i]) != cudaSuccess) result = result ? result : NKV_ERR_CUDA;
    // the status of every step was copied out before its slot was reused: report the first failure
    for (int64_t i = 0; i < step && result == NKV_OK; ++i)
        if (h->chunk_status[i] != 0) result = h->chunk_status[i] == NKV_ERR_TIMEOUT ? NKV_ERR_TIMEOUT : NKV_ERR_DEVICE_CHECK;
    if (result == NKV_ERR_CUDA) cudaGetLastError();
    return result;
}

int nkv_last_device_status(nkv_handle* h, const void* ws, void* stream) {
    if (!h || !ws) return NKV_ERR_INVALID_ARG;
    int words[4] = {0, 0, 0, 0};
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return NKV_ERR_CUDA;
    if (cudaMemcpy(words, ws, sizeof(words), cudaMemcpyDeviceToHost) != cudaSuccess) return NKV_ERR_CUDA;
    if (words[kStatusCode] == NKV_ERR_TIMEOUT) return NKV_ERR_TIMEOUT;
    if (words[kStatusCode] != 0) return NKV_ERR_DEVICE_CHECK;
    return NKV_OK;
}

int nkv_set_timing(nkv_handle* h, int enable) {
    if (!h) return NKV_ERR_INVALID_ARG;
    h->timing = enable ? 1 : 0;
    h->timing_valid = 0;
    return NKV_OK;
}

int nkv_get_stage_ms(nkv_handle* h, float* ms_out) {
    if (!h || !ms_out || !h->timing_valid) return NKV_ERR_INVALID_ARG;
    if (cudaEventSynchronize(h->ev[NKV_NUM_STAGES]) != cudaSuccess) return NKV_ERR_CUDA;
    for (int i = 0; i < NKV_NUM_STAGES; ++i)
        if (cudaEventElapsedTime(&ms_out[i], h->ev[i], h->ev[i + 1]) != cudaSuccess) return NKV_ERR_CUDA;
    return NKV_OK;
}

int nkv_host_bytes(const nkv_handle* h, int64_t* in, int64_t* out) {
    if (!h || !in || !out) return NKV_ERR_INVALID_ARG;
    *in = h->host_in;
    *out = h->host_out;
    return NKV_OK;
}

int64_t nkv_launch_count(const nkv_handle* h) { return h ? h->launches : -1; }

int nkv_key_scan(nkv_handle* h, const nkv_tensor* K, const nkv_params* params, float* inv_norm, float* mu_s,
                 float* mu_e, float* a_raw, float* minmax, void* ws, size_t ws_bytes, void* stream) {
    if (!h || !inv_norm || !mu_s || !mu_e || !a_raw || !minmax) return NKV_ERR_INVALID_ARG;
    int rc = check_tensor(K);
    if (rc) return rc;
    if ((rc = check_units(K->G * K->H))) return rc;
    ScoreParams sp;
    if ((rc = resolve_params(params, K->N, &sp))) return rc;
    const int G = (int)K->G, N = (int)K->N, d = (int)K->d, units = (int)(K->G * K->H);
    const Layout L = make_layout(units, N, d, sp.nblocks);
    if ((rc = check_ws(ws, ws_bytes, L.total))) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    CU(cudaMemsetAsync(ws, 0, cleared_bytes(L, units), st));
    auto no_mark = []() -> cudaError_t { return cudaSuccess; };
    if ((rc = key_scan(h, view_of(K), K->dtype, G, sp, bufs_at(ws, L), at<int>(ws, L.status), st, no_mark))) return rc;
    const size_t row = (size_t)padded_row(N) * 4, out_row = (size_t)N * 4;
    CU(cudaMemcpyAsync(mu_s, at<float>(ws, L.mu_s), (size_t)units * d * 4, cudaMemcpyDeviceToDevice, st));
    CU(cudaMemcpyAsync(mu_e, at<float>(ws, L.mu_e), (size_t)units * sp.nblocks * d * 4, cudaMemcpyDeviceToDevice, st));
    CU(cudaMemcpy2DAsync(inv_norm, out_row, at<float>(ws, L.inv_norm), row, out_row, units, cudaMemcpyDeviceToDevice, st));
    CU(cudaMemcpy2DAsync(a_raw, out_row, at<float>(ws, L.a_raw), row, out_row, (size_t)units * 3, cudaMemcpyDeviceToDevice, st));
    minmax_floats_kernel<<<(units * 6 + 255) / 256, 256, 0, st>>>(units * 6, at<uint32_t>(ws, L.mm), minmax);
    ++h->launches;
    CU(cudaGetLastError());
    return NKV_OK;
}

int nkv_debug_set(nkv_handle* h, int what, int64_t value) {
    if (!h) return NKV_ERR_INVALID_ARG;
    switch (what) {
        case NKV_DEBUG_INJECT_HOST_STATUS:   // value = chunk * 16 + status code (0 clears)
            if (value < 0) return NKV_ERR_INVALID_ARG;
            h->inject_status = (int)(value & 15);
            h->inject_chunk = (int)(value >> 4);
            return NKV_OK;
        default:
            return NKV_ERR_INVALID_ARG;
    }
}

int nkv_debug_wait_probe(nkv_handle* h, int64_t polls, void* ws, size_t ws_bytes, void* stream) {
    if (!h || polls < 1 || polls > (1 << 16)) return NKV_ERR_INVALID_ARG;
    int rc = check_ws(ws, ws_bytes, align_up(kStatusWords * sizeof(int)));
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    CU(cudaMemsetAsync(ws, 0, kStatusWords * sizeof(int), st));
    CU(launch_wait_probe(static_cast<int*>(ws), (uint32_t)polls, st, &h->launches));
    return NKV_OK;
}

int nkv_set_key_passes(nkv_handle* h, int mode) {
    if (!h || mode < NKV_KEY_PASS_AUTO || mode > NKV_KEY_PASS_TENSOR) return NKV_ERR_INVALID_ARG;
    h->key_pass = mode;
    return NKV_OK;
}

}  // extern "C"
