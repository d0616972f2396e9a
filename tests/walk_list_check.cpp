// Host check of the walk's list (walk_list.cuh): 32 lanes as threads that run one at a time, each until the next
// barrier, first to last or last to first -- an order that the program allows wherever lanes don't meet.  Every lane
// has to sum the entries as they were, and the rest has to arrive at the front.
#define __host__
#define __device__
#define __forceinline__ inline
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <thread>
#include <vector>
struct alignas(16) float4 { float x, y, z, w; };
#include "walk_list.cuh"

struct Turns {  // whose turn it is: lane after lane up to the barrier, then the next round
    std::mutex m;
    std::condition_variable cv;
    int at = 0;  // place in the order
    void wait(int place) {
        std::unique_lock<std::mutex> l(m);
        cv.wait(l, [&] { return at == place; });
    }
    void pass() {
        std::lock_guard<std::mutex> l(m);
        at = (at + 1) % 32;
        cv.notify_all();
    }
};

struct Warp {
    Turns *t;
    int id, place;
    uint32_t lane() const { return (uint32_t)id; }
    void sync() const {
        t->pass();
        t->wait(place);
    }
};

int main() {
    constexpr uint32_t CHUNK = 128, CAP = 256;
    int bad = 0;
    for (uint32_t n0 : {0u, 1u, 127u, 128u, 129u, 131u, 160u, 250u, 255u, 256u})
        for (uint32_t step : {1u, 4u, 32u})  // lanes that share a member's quads
            for (int down = 0; down < 2; down++) {
                alignas(16) static float lx[4 * CAP];
                auto value = [&](uint32_t e) { return (float)(e * 7 % 251 + 1); };
                for (uint32_t a = 0; a < 4; a++)
                    for (uint32_t e = 0; e < CAP; e++) lx[a * CAP + e] = e < n0 ? value(e) + 300.0f * a : -1e6f;
                Turns turns;
                std::vector<double> sum(32, 0.0);
                std::vector<uint32_t> left(32), full(32);
                std::vector<std::thread> lanes;
                for (int id = 0; id < 32; id++)
                    lanes.emplace_back([&, id] {
                        const Warp w{&turns, id, down ? 31 - id : id};
                        w.t->wait(w.place);
                        uint32_t n = n0;
                        full[id] = flush_chunks<CHUNK>(lx, CAP, n, w, [&](uint32_t k0, uint32_t k1) {
                            for (uint32_t k = k0 + id % step; k < k1; k += step)
                                for (uint32_t a = 0; a < 4; a++)
                                    for (uint32_t j = 0; j < 4; j++) sum[id] += lx[a * CAP + 4 * k + j];
                        });
                        left[id] = n;
                        w.t->pass();
                    });
                for (auto &t : lanes) t.join();
                const uint32_t chunks = n0 / CHUNK;
                for (int id = 0; id < 32; id++) {
                    double want = 0.0;
                    for (uint32_t k = id % step; k < chunks * (CHUNK / 4); k += step)
                        for (uint32_t a = 0; a < 4; a++)
                            for (uint32_t j = 0; j < 4; j++) want += value(4 * k + j) + 300.0f * a;
                    if (sum[id] != want || left[id] != n0 % CHUNK || full[id] != chunks)
                        if (bad++ < 10) printf("n %u step %u down %d lane %d: %.0f, not %.0f\n", n0, step, down, id, sum[id], want);
                }
                for (uint32_t a = 0; a < 4; a++)
                    for (uint32_t e = 0; e < n0 % CHUNK; e++)
                        if (lx[a * CAP + e] != value(chunks * CHUNK + e) + 300.0f * a && bad++ < 10)
                            printf("n %u step %u down %d: entry %u is not moved\n", n0, step, down, e);
            }
    // a window's entries: slot list_n - w0 + e, also where w0 > list_n
    static float list[CAP];
    for (uint32_t list_n : {0u, 5u, 127u})
        for (uint32_t w0 : {0u, 3u, 200u, 5000u})
            for (uint32_t e = w0; e < w0 + CAP - list_n; e++)
                if (list_at(list, list_n - w0, e) != list + (list_n + (e - w0)) && bad++ < 20)
                    printf("list %u window %u entry %u: another address\n", list_n, w0, e);
    printf("bad %d\n", bad);
    return bad != 0;
}
