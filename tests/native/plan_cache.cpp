// Host threads that ask a context's plan cache for more shapes than it keeps: every plan handed out must be, from the first
// word to the last, the one its key asks for.
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>

#include "../../paper_2609_02652_b200/csrc/llvq_internal.cuh"

using namespace llvq;

static GemvLaunch fill(GemvPlan &plan, int shape) {
    plan.panel = plan.npanels = plan.xblocks = shape;
    for (CtaShare &c : plan.cta) c.first = shape;
    return {shape, (size_t)shape};
}

static bool whole(const GemvPlan &plan, const GemvLaunch &launch, int shape) {
    bool ok = plan.panel == shape && plan.npanels == shape && plan.xblocks == shape && launch.grid == shape && launch.smem == (size_t)shape;
    for (const CtaShare &c : plan.cta) ok = ok && c.first == shape;
    return ok;
}

int main() {
    PlanCache cache;
    std::atomic<long> wrong{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 4; t++)
        threads.emplace_back([&, t] {
            GemvPlan plan;
            uint32_t pick = 12345u * (uint32_t)(t + 1);
            for (int i = 0; i < 100000; i++) {
                pick = pick * 1664525u + 1013904223u;
                PlanKey key{};
                key.nb = 1 + (int)(pick >> 16) % 12;
                const GemvLaunch launch = cache.get(key, plan, [&](GemvPlan &p) { return fill(p, key.nb); });
                if (!whole(plan, launch, key.nb)) wrong++;
            }
        });
    for (std::thread &t : threads) t.join();
    std::printf("%ld\n", wrong.load());
    return wrong.load() ? 1 : 0;
}
