// Host check of the serving context (csrc/ph0_serve.cu) against a fake of the
// CUDA calls it makes (serve_fake_cuda.cpp): a cloud whose launch fails part of the way has kernels
// queued on its stream, so its device memory must not go to another cloud
// before that stream was waited for.  The fake keeps, for every stream, the
// device ranges its queued work uses until the stream is synchronized, and
// counts uses of such a range from another stream.
//   serve_failure_check first : the first launch of a cloud fails
//   serve_failure_check again : its second one, with the complete sort, does
// Prints "clouds failed overlaps".
#include <atomic>
#include <chrono>
#include <cstdio>
#include <string>
#include <thread>
#include <vector>

#include "ph0_common.cuh"

// the fake (serve_fake_cuda.cpp)
void fake_use(const void *p, size_t bytes, cudaStream_t s);
extern std::atomic<int> g_overlaps;
extern std::atomic<bool> g_ready;

namespace {
constexpr int kBad = 40;  // points of the cloud whose launch fails
bool g_again = false;
std::atomic<int> g_launches{0};
}  // namespace

// ---- the library's other units ----
namespace ph0 {
cudaError_t prepare_small_kernel() { return cudaSuccess; }
cudaError_t launch_small(const SmallTask *, const int32_t *, uint32_t *, int, cudaStream_t) { return cudaSuccess; }
int small_max_n() { return 8; }
int small_max_d() { return 8; }
int sm_count() { return 4; }
int barcodes_whole(const float *, int64_t n, int32_t, int64_t, ph0_bar *, ph0_inf_bar *, void *ws, size_t ws_bytes,
                   void *stream, const ph0_tuning *, bool full) {
    fake_use(ws, ws_bytes, static_cast<cudaStream_t>(stream));
    Header *h = static_cast<Header *>(ws);
    h->status = PH0_OK;
    h->inf_vertex = 0;
    h->fixup_fallback = g_again && n == kBad ? 1 : 0;
    ++g_launches;
    return n == kBad && full == g_again ? PH0_ECUDA : PH0_OK;
}
}  // namespace ph0

extern "C" {
size_t ph0_workspace_bytes(int64_t n, int32_t) { return (size_t(512) << 10) + size_t(n) * 1024; }
}

int main(int argc, char **argv) {
    g_again = argc > 1 && std::string(argv[1]) == "again";
    // room for clouds of 39 and 40 points at a time, or for a large one
    const int d = 9;  // beyond small_max_d: every cloud on a stream of its own
    auto bytes = [&](int n) {
        return ph0::align_up(size_t(n) * d * 4, 256) + ph0::align_up(size_t(n - 1) * sizeof(ph0_bar), 256) +
               ph0::align_up(ph0_workspace_bytes(n, d), 256) + 256;
    };
    ph0_options opt{};
    opt.host_budget = size_t(8) << 20;
    opt.streams = 2;
    opt.small_max_n = 8;
    opt.batch_max = 1;
    opt.mem_budget = bytes(kBad - 1) + bytes(kBad);  // above the least that is accepted, 1 MiB
    int big = kBad;
    while (bytes(big + 1) <= opt.mem_budget) ++big;
    ph0_ctx *c = nullptr;
    if (ph0_ctx_create(&opt, &c) != PH0_OK) return 2;
    std::vector<float> x(size_t(big) * d, 0.0f);
    // first: the bad cloud's stream is free at once, and the next cloud, on
    // the next stream, needs its room.  again: a good cloud on the first
    // stream, the bad one on the second, both ready at once, and a large one
    // that needs the room of both
    const int sizes[3] = {g_again ? kBad - 1 : kBad, g_again ? kBad : big, big};
    g_ready = !g_again;
    for (int i = 0; i < 3; ++i) {
        if (ph0_submit(c, x.data(), sizes[i], d, uint64_t(i + 1)) != PH0_OK) return 3;
        while (g_again && i < 2 && g_launches < i + 1) std::this_thread::sleep_for(std::chrono::milliseconds(1));
    }
    std::this_thread::sleep_for(std::chrono::milliseconds(20));
    g_ready = true;
    int clouds = 0, failed = 0;
    for (int t = 0; t < 400 && clouds < 3; ++t) {
        ph0_result r[4];
        int32_t got = 0;
        ph0_poll(c, r, 4, &got, 10);
        for (int i = 0; i < got; ++i) failed += r[i].status != PH0_OK;
        clouds += got;
    }
    ph0_ctx_destroy(c);
    std::printf("%d %d %d\n", clouds, failed, g_overlaps.load());
    return 0;
}
