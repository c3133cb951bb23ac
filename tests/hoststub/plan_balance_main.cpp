// Work lists of batched plans with many short streams beside a long one (test only): prints,
// per mix and launch shape, the largest and the mean over the CTAs of what their items
// take, and the largest number of items of a CTA.  An item takes its samples' multiply-adds,
// and at least 350,000 (1.7 us on an SM, measured on items of 64 to 500 samples).
#include <algorithm>
#include <complex>
#include <cstdio>
#include <vector>

#include "dpd.h"
#include "stub_batched.h"

static std::vector<dpd::BatchItem> g_items;
static std::vector<dpd::BatchStream> g_streams;
static int g_nsub;
namespace dpd {
int record(const BatchArgs &a)
{
    g_items.assign(a.items, a.items + a.nitems);
    g_streams.assign(a.streams, a.streams + a.nstreams);
    g_nsub = a.nsub;
    return 0;
}
}

int main()
{
    struct Mix { int64_t longest; int count; int64_t n; } mixes[] = {{1 << 24, 4000, 500}, {1 << 22, 2000, 64}, {1 << 22, 8000, 300}, {0, 5000, 1500}};
    const int shapes[][5] = {{0}, {6, 16, 2, 0, 4}, {8, 16, 2, 0, 4}};
    std::vector<std::complex<float>> x((1 << 24) + 2), y((1 << 24) + 2), h(97);
    for (const Mix &m : mixes) {
        std::vector<dpd_stream_desc> d;
        if (m.longest) d.push_back({x.data(), y.data(), m.longest, 9, 9, 4, h.data()});
        // the plan refuses overlapping outputs: the short streams' are consecutive
        std::vector<std::complex<float>> ys((size_t)m.count * (m.n + 2));
        for (int i = 0; i < m.count; ++i) d.push_back({x.data(), ys.data() + (size_t)i * (m.n + (m.n & 1)), m.n, 5, 5, 2, h.data()});
        dpd_plan p = nullptr;
        if (dpd_plan_batched(d.data(), (int)d.size(), DPD_HOST, &p) != DPD_OK) return 1;
        for (const int *s : shapes) {
            if (s[0] && dpd_plan_set_launch(p, s[0], s[1], s[2], s[3], s[4]) != DPD_OK) return 2;
            if (dpd_exec_batched(p, nullptr) != DPD_OK) return 3;
            const int G = 152, block = (s[0] ? s[0] * s[1] : 6 * 16) * 32;
            std::vector<double> cost(G, 0.0);
            std::vector<int> number(G, 0);
            for (size_t i = 0; i < g_items.size(); ++i) {
                const dpd::BatchItem w = g_items[i];
                if (w.stream < 0) continue;
                const dpd::BatchStream &st = g_streams[w.stream];
                const int64_t first = (int64_t)(w.tile / 4) * block, len = std::min<int64_t>((w.tile % 4 + 1) * (int64_t)block, st.n - first);
                cost[i % G] += std::max(350000.0, (4.0 * st.B * st.T + 28.0) * len);
                ++number[i % G];
            }
            double sum = 0.0;
            for (double c : cost) sum += c;
            size_t in_order = 0;   // items that follow the one before them in the plan's order
            for (size_t i = 1; i < g_items.size(); ++i)
                in_order += g_items[i].stream == g_items[i - 1].stream ? g_items[i].tile > g_items[i - 1].tile
                                                                       : g_items[i].stream >= 0 && g_items[i - 1].stream >= 0;
            std::printf("dealt out in order: %d\n", in_order == g_items.size() - 1);
            std::printf("mix %lld + %d x %lld shape %d: largest %.3f of the mean, %d items at most\n", (long long)m.longest, m.count,
                        (long long)m.n, s[0], *std::max_element(cost.begin(), cost.end()) / (sum / G),
                        *std::max_element(number.begin(), number.end()));
        }
        dpd_plan_destroy(p);
    }
}
