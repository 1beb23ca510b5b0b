// The upload of the sieve form's tables from several host threads at once, with the
// copies to the device replaced by a recorder that reads its source slowly. Prints the
// number of uploads and how many of them changed while they were read or differ from a
// single thread's.
#include <cuda_runtime.h>

#include <chrono>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>

static std::mutex g_mu;
static std::vector<std::vector<unsigned char>> g_seen[2];   // by table, told apart by their sizes
static size_t g_bytes[2] = {0, 0};
static int g_torn = 0;

static cudaError_t record_upload(const void *src, size_t bytes)
{
    std::vector<unsigned char> a((const unsigned char *)src, (const unsigned char *)src + bytes);
    std::this_thread::sleep_for(std::chrono::microseconds(50));
    const bool torn = std::memcmp(a.data(), src, bytes) != 0;
    std::lock_guard<std::mutex> g(g_mu);
    g_torn += torn;
    for (int k = 0; k < 2; ++k)
        if (g_bytes[k] == 0 || g_bytes[k] == bytes) {
            g_bytes[k] = bytes;
            g_seen[k].push_back(std::move(a));
            break;
        }
    return cudaSuccess;
}

#define cudaMemcpyToSymbol(symbol, src, bytes) record_upload(src, bytes)
#include "../../paper_2403_00306_gb300/csrc/pms_sieve.cu"
#undef cudaMemcpyToSymbol

int main()
{
    constexpr int kThreads = 8, kUploads = 100;
    std::vector<std::thread> th;
    for (int t = 0; t < kThreads; ++t)
        th.emplace_back([] {
            for (int u = 0; u < kUploads; ++u)
                pms::sieve_init_tables();
        });
    for (auto &t : th)
        t.join();
    pms::sieve_init_tables();   // alone: the last of each table
    int uploads = 0, wrong = g_torn;
    for (const auto &seen : g_seen) {
        uploads += (int)seen.size();
        for (const auto &s : seen)
            wrong += s != seen.back();
    }
    std::printf("%d %d\n", uploads, wrong);
    return 0;
}
