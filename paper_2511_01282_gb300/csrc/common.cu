// common.cu -- error reporting, version and launch accounting of the library.
#include <atomic>
#include <mutex>

#include "common.cuh"

namespace rs {

static thread_local char g_err[1024] = "";
static std::atomic<uint64_t> g_launches{0};

void set_error(const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof g_err, fmt, ap);
    va_end(ap);
}

void clear_error() { g_err[0] = 0; }

void count_launch(int n) { g_launches.fetch_add((uint64_t)n, std::memory_order_relaxed); }

int num_sms() {
    static std::mutex mu;
    static int cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    std::lock_guard<std::mutex> lk(mu);
    if (!cache[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 148;
        cache[dev] = n;
    }
    return cache[dev];
}

unsigned long long context_id() {
    typedef int (*ctx_get_current_t)(void **);
    typedef int (*ctx_get_id_t)(void *, unsigned long long *);
    static std::once_flag once;
    static ctx_get_current_t get_current = nullptr;
    static ctx_get_id_t get_id = nullptr;
    std::call_once(once, [] {
        void *a = nullptr, *b = nullptr;
        cudaDriverEntryPointQueryResult qa, qb;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 12000, cudaEnableDefault, &qa) ==
                cudaSuccess && qa == cudaDriverEntryPointSuccess &&
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &qb) == cudaSuccess &&
            qb == cudaDriverEntryPointSuccess) {
            get_current = reinterpret_cast<ctx_get_current_t>(a);
            get_id = reinterpret_cast<ctx_get_id_t>(b);
        }
    });
    if (!get_current || !get_id) return 0;
    void *ctx = nullptr;
    unsigned long long id = 0;
    if (get_current(&ctx) != 0 || !ctx || get_id(ctx, &id) != 0) return 0;
    return id;
}

long long l2_bytes() {
    static std::mutex mu;
    static long long cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 128ll << 20;
    std::lock_guard<std::mutex> lk(mu);
    if (!cache[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrL2CacheSize, dev) != cudaSuccess || n <= 0) n = 128 << 20;
        cache[dev] = n;
    }
    return cache[dev];
}

}  // namespace rs

extern "C" {

const char *rs_last_error(void) { return rs::g_err; }

const char *rs_version(void) { return "respec-gb300 0.1 (sm_103a)"; }

uint64_t rs_launch_count(void) { return rs::g_launches.load(); }

}  // extern "C"
