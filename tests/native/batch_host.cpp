// The host code of batches and of the serving loop (vjb_batch.cu) without a GPU:
// device memory is host memory, a context is its sizes and its round state, and
// a launched graph counts one round for every job that takes part.  The job of
// kFailing samples reports a kernel error flag in its second round.  Built with
// checked standard containers; prints "ok".
#include <cstdlib>

#include "vjb_batch.cu"

constexpr int kFailing = 13;

#define CHECK(x)                                                              \
    do {                                                                      \
        if (!(x)) {                                                           \
            printf("line %d: %s (%s)\n", __LINE__, #x, g_err);                \
            exit(1);                                                          \
        }                                                                     \
    } while (0)

// ---- the runtime, on host memory ----------------------------------------------------
namespace {
JobDesc *g_jobs;
BatchMeta *g_meta;
BatchSeen *g_seen;
template <class H>
H handle() { return reinterpret_cast<H>(uintptr_t(64)); }

void one_round() {
    for (int j = 0; j < g_meta->njobs; ++j) {
        RoundState *rs = g_jobs[j].rs;
        if (rs->status == VJB_OK && !rs->flags && rs->rounds < g_jobs[j].round_target) {
            rs->rounds += 1;
            if (g_jobs[j].lay.n == kFailing && rs->rounds == 2) {
                rs->flags |= kFlagWaitTimeout;
                g_meta->flags |= kFlagWaitTimeout;
            }
        }
        g_seen->job[j] = JobSeen{rs->status, rs->rounds, rs->flags, 0};
    }
    g_seen->flags = g_meta->flags;
}
CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int x, size_t n, cudaStream_t) { memset(d, x, n); return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) {
    memset(p, 0, sizeof *p);
    p->multiProcessorCount = 4;
    p->sharedMemPerBlockOptin = 232448;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *q) {
    *fn = reinterpret_cast<void *>(encode);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = handle<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) { *s = handle<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = handle<cudaGraph_t>(); return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *a, int *b) { *a = *b = 0; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = handle<cudaGraphExec_t>(); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { one_round(); return cudaSuccess; }
}

// ---- the rest of the library, as far as batches use it --------------------------------
namespace vjb {
thread_local char g_err[512];
int fail(int code, const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof g_err, fmt, ap);
    va_end(ap);
    return code;
}
int ensure_stump_cap(vjb_ctx *c, int need) {
    if (need > c->stump_cap) {
        free(c->d_stumps);
        c->d_stumps = static_cast<vjb_stump *>(calloc((size_t)need, sizeof(vjb_stump)));
        c->stump_cap = need;
    }
    return VJB_OK;
}
JobDesc job_desc(const vjb_ctx *c) {
    JobDesc J{};
    J.nfeat = c->nfeat;
    J.lay.n = c->n;
    J.rs = c->d_rs;
    return J;
}
int validate_labels(const uint8_t *, int) { return VJB_OK; }
int screen_max_warps(int) { return 16; }
cudaError_t set_screen_smem_limit(int) { return cudaSuccess; }
cudaError_t set_bscreen_smem_limit(int) { return cudaSuccess; }
size_t bscreen_smem_bytes(const SearchShape &, int) { return 0; }
WeightLayout make_layout(int n, bool) { return WeightLayout{n, 0, 0, n + 1, 0}; }
int update_grid(int n) { return (n + 255) / 256; }
cudaError_t launch_bbegin(JobDesc *jobs, BatchMeta *meta, cudaStream_t) { g_jobs = jobs; g_meta = meta; return cudaSuccess; }
cudaError_t launch_bscreen(const BatchMaps &, const JobDesc *, const WorkItem *, BatchMeta *, int, const SearchShape &, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_bshortlist(const JobDesc *, BatchMeta *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_brescan(const JobDesc *, BatchMeta *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_bupdate_a(const JobDesc *, BatchMeta *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_bupdate_b(const JobDesc *, BatchMeta *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_bend(const JobDesc *, const BatchMeta *, BatchSeen *seen, cudaStream_t) { g_seen = seen; return cudaSuccess; }
}  // namespace vjb

extern "C" {
const char *vjb_last_error(void) { return g_err; }
int vjb_create(vjb_ctx **out, int device, void *stream) {
    *out = new vjb_ctx();
    (*out)->device = device;
    (*out)->stream = static_cast<cudaStream_t>(stream);
    return VJB_OK;
}
void vjb_destroy(vjb_ctx *c) {
    c->free_all();
    delete c;
}
int vjb_load_windows(vjb_ctx *c, const uint8_t *, const uint8_t *, int32_t n, int32_t h, int32_t w) {
    c->n = n;
    c->h = h;
    c->w = w;
    c->d_w = static_cast<float *>(calloc((size_t)n, sizeof(float)));
    c->d_rs = static_cast<RoundState *>(calloc(1, sizeof(RoundRecord)));
    return ensure_stump_cap(c, 1);
}
int vjb_build_integral(vjb_ctx *) { return VJB_OK; }
int vjb_enumerate_haar(vjb_ctx *c, int64_t *count, vjb_feature *) {
    *count = c->nfeat = haar_count(c->w, c->h);
    return VJB_OK;
}
int vjb_get_info(vjb_ctx *c, vjb_info *out) {
    memset(out, 0, sizeof *out);
    out->rounds_done = c->d_rs->rounds;
    out->status = c->d_rs->status;
    out->device_flags = c->d_rs->flags;
    return VJB_OK;
}
int vjb_get_weights(vjb_ctx *, float *) { return VJB_OK; }
}

// ---- the cases -----------------------------------------------------------------------
static int32_t add(vjb_batch *b, int n, int rounds) {
    std::vector<uint8_t> px((size_t)n * 16), y((size_t)n);
    int32_t id = -1;
    CHECK(vjb_batch_add_job(b, px.data(), y.data(), n, 4, 4, rounds, &id) == VJB_OK);
    return id;
}

// An error flag is reported until the job that set it leaves, and no longer.
static void flags() {
    vjb_batch *b = nullptr;
    CHECK(vjb_batch_create(&b, 0, nullptr, 1 << 20) == VJB_OK);
    const int32_t good = add(b, 10, 5), bad = add(b, kFailing, 5);
    int32_t ran = -1, done = 0, status = 0;
    CHECK(vjb_batch_train(b, 100, &ran) == VJB_EDEVICE);
    CHECK(vjb_batch_job_state(b, good, &done, &status) == VJB_OK && done == 5 && status == VJB_OK);
    CHECK(vjb_batch_job_state(b, bad, &done, &status) == VJB_OK && done == 2 && status == VJB_EDEVICE);
    CHECK(vjb_batch_train(b, 100, &ran) == VJB_EDEVICE);  // the job is still there
    CHECK(vjb_batch_remove_job(b, bad) == VJB_OK);
    CHECK(vjb_batch_train(b, 100, &ran) == VJB_OK && ran == 0);
    add(b, 11, 3);
    CHECK(vjb_batch_train(b, 100, &ran) == VJB_OK && ran == 3);
    vjb_batch_destroy(b);
}

// Jobs of 2, 5 and 8 rounds served in one step: how many take part in each round.
static void step_counts() {
    vjb_server *s = nullptr;
    CHECK(vjb_server_create(&s, 0, 1 << 20, 8) == VJB_OK);
    std::vector<uint8_t> px(20 * 16), y(20);
    int64_t id[3];
    const int32_t rounds[3] = {2, 5, 8};
    for (int k = 0; k < 3; ++k) CHECK(vjb_server_submit(s, px.data(), y.data(), 20, 4, 4, rounds[k], &id[k]) == VJB_OK);
    vjb_server_summary sum;
    do {
        CHECK(vjb_server_step(s, 0, nullptr) == VJB_OK);
        CHECK(vjb_server_stats(s, &sum) == VJB_OK);
    } while (sum.training < 3);
    int32_t ran = 0;
    CHECK(vjb_server_step(s, 8, &ran) == VJB_OK && ran == 8);
    float ms[8];
    int32_t jobs[8];
    CHECK(vjb_server_round_times(s, 0, 8, ms, jobs) == VJB_OK);
    const int32_t expected[8] = {3, 3, 2, 2, 2, 1, 1, 1};
    for (int k = 0; k < 8; ++k) CHECK(jobs[k] == expected[k]);
    CHECK(vjb_server_stats(s, &sum) == VJB_OK && sum.job_rounds == 15 && sum.done == 3);
    for (int k = 0; k < 3; ++k) {
        vjb_request_info r;
        CHECK(vjb_server_request(s, id[k], &r) == VJB_OK && r.rounds_done == rounds[k] && r.rounds_timed == rounds[k]);
    }
    vjb_server_destroy(s);
}

int main(int argc, char **argv) {
    if (argc == 2 && !strcmp(argv[1], "flags")) flags();
    else if (argc == 2 && !strcmp(argv[1], "step_counts")) step_counts();
    else return 2;
    printf("ok\n");
    return 0;
}
