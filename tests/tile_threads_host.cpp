// Two host threads that call the library side by side, each on its own decoder and
// stream: plain BP, the training forward and backward in turn.  Returns the number
// of calls that did not return BSD_OK.
#include <cstdint>
#include <thread>

#include "bsd.h"

struct Api {
    decltype(&bsd_bp_llr) llr;
    decltype(&bsd_unrolled_forward) forward;
    decltype(&bsd_unrolled_backward) backward;
};
struct Job {
    bsd_decoder* llr_dec;
    bsd_decoder* dec;
    const uint32_t* synd;
    const uint32_t* errs;
    int64_t B;
    int32_t T, ckpt;
    const float* w;
    const float* grad_loss;
    float* llr;
    float* loss;
    float* grad;
    void* work;
    int64_t work_bytes;
    void* stream;
};

extern "C" int tile_threads(const Api* api, const Job* jobs, int calls)
{
    int failed[2] = {0, 0};
    auto run = [&](int k) {
        const Job& j = jobs[k];
        for (int n = 0; n < calls; ++n) {
            const int rc = n % 3 == 0 ? api->llr(j.llr_dec, j.synd, j.B, j.T, j.llr, nullptr, j.stream)
                         : n % 3 == 1 ? api->forward(j.dec, j.synd, j.errs, j.B, j.T, j.ckpt, j.w, j.loss, nullptr, j.work,
                                                     j.work_bytes, j.stream)
                                      : api->backward(j.dec, j.B, j.T, j.ckpt, j.w, j.grad_loss, j.grad, j.work,
                                                      j.work_bytes, j.stream);
            failed[k] += rc != BSD_OK;
        }
    };
    std::thread other(run, 1);
    run(0);
    other.join();
    return failed[0] + failed[1];
}
