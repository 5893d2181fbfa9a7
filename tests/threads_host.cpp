/* Host threads that make one decode call each, over and over, at the same
 * time (test_gpu_zthreads.py): in native code, because threads of the
 * interpreter spend most of their time waiting for its lock. */
#include <atomic>
#include <cstdint>
#include <thread>
#include <vector>

struct Call {
    void *handle; /* orbg_code, or orbg_codeset with batched */
    const float *llr;
    int64_t blocks;
    uint8_t *cw;
    uint32_t *q;
    uint8_t *ab;
    void *stream;
};

typedef int (*Plain)(const void *, const float *, int64_t, uint32_t, uint8_t *, uint32_t *,
                     uint8_t *, void *);
typedef int (*Batched)(const void *, const int32_t *, const int64_t *, const float *, int64_t,
                       uint32_t, uint8_t *, const int64_t *, uint32_t *, uint8_t *, void *);

/* refused[i]: how many of thread i's calls did not return 0 */
extern "C" void calls_together(void *plain, void *batched, uint32_t cap, const Call *c,
                               int threads, int calls, int *refused)
{
    std::atomic<int> ready{0};
    std::vector<std::thread> all;
    for (int i = 0; i < threads; i++)
        all.emplace_back([&, i] {
            refused[i] = 0;
            ready++;
            while (ready.load() < threads)
                ;
            for (int k = 0; k < calls; k++) {
                const int rc =
                    plain ? ((Plain)plain)(c[i].handle, c[i].llr, c[i].blocks, cap, c[i].cw,
                                           c[i].q, c[i].ab, c[i].stream)
                          : ((Batched)batched)(c[i].handle, nullptr, nullptr, c[i].llr,
                                               c[i].blocks, cap, c[i].cw, nullptr, c[i].q,
                                               c[i].ab, c[i].stream);
                refused[i] += rc != 0;
            }
        });
    for (auto &t : all)
        t.join();
}
