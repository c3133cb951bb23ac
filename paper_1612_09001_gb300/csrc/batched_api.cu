// libdpd C ABI, batched part: plans of many independent streams executed by
// one persistent launch (see dpd_batched.cuh and include/dpd.h).
#include <algorithm>
#include <cstdint>
#include <new>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/dpd.h"
#include "dpd_model.h"
#include "dpd_batched.cuh"

struct dpd_plan_s {
    int device = 0, sm_count = 0;
    std::vector<dpd::BatchStream> streams;   // host copy (device pointers, sizes, table offsets)
    dpd::BatchStream *d_streams = nullptr;
    dpd::BatchItem *d_items = nullptr;
    float *d_tabs = nullptr;
    float *d_h = nullptr;          // raw coefficients, 2*K floats per stream
    int *d_status = nullptr;
    int nitems = 0;
    int64_t tab_floats = 0;
    int small = 1;            // every stream has B <= 5 and T <= 7
    int V = 0, warps = 0, stages = 0, ctas_per_sm = 0, group = 0;   // launch shape (default_shape, or set explicitly)
    int nsub = 0;             // sub-blocks per thread and item (follows the launch shape)
};

namespace {

constexpr int64_t kMaxBlocks = (int64_t)1 << 29;   // what dpd::batch_tile packs
// What an item of one sub-block costs besides its samples, in multiply-adds: it ends before
// the copies of the item after the next have arrived, where a full item covers them.
constexpr double kShortItem = 250000.0;

// Whether the work list is cut into one run of equal cost per CTA (build_items): for launches
// of one CTA per SM (the ring takes more than half of the shared memory) with 6 samples per
// thread.  With 8 the window loads' bank conflicts and with 4 the loads themselves bound a
// sample more than its multiply-adds, so runs of equal cost are not of equal time: 64
// streams of mixed models, us, dealt out in order / in runs: V = 8, 16 warps, 2 stages 160
// / 198, V = 8, 8 warps, 4 stages 188 / 236, V = 4, 16 warps, 4 stages 155 / 167, V = 6, 16
// warps in groups of 4, 2 stages 126 / 119, V = 6, 8 warps, 4 stages 161 / 148.
bool equal_runs(int V, int warps, int group, int stages, int nsub)
{
    return V == 6 && dpd::batch_smem(warps, group > 0 ? group : warps, stages, V, nsub) > dpd::kBatchSmemMax / 2;
}

int nbranch(int order) { return order > 0 ? (order + 1) / 2 : 0; }
bool aligned(const void *p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }
bool overlap(const void *a, size_t na, const void *b, size_t nb)
{
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return na && nb && x < y + nb && y < x + na;
}

// Launch shape of a new plan.  6 samples per thread (the 16-byte window loads of a
// quarter warp on distinct banks) and 16 warps in groups of 4, one CTA per SM with a
// run of items of up to 12,288 samples.  Batches that leave an SM fewer than 8,192
// samples are bound by latency and take 4 samples per thread, 4 warps and items of 2,048
// samples on as many CTAs as fit an SM.  GB300, us per launch, first shape / second shape
// / 8 samples per thread on 8 warps with items of 8,192 dealt out in order: 64 streams,
// 36.7 M samples 125.9 / 150 / 217.7; 24 streams, 12.2 M 47.7 / 57.7 / 89.3; 33 streams, 3.8 M
// 25.5 / 27.3 / 49.5; 16 streams, 1.3 M 16.9 / 17.1 / 23.1; 8 streams, 0.17 M 12.8 / 11.1 / 15.1.
void default_shape(dpd_plan p)
{
    int64_t units = 0;   // of 1024 samples
    for (const dpd::BatchStream &st : p->streams) units += st.n / 1024;
    const bool large = units >= 8 * (int64_t)p->sm_count;
    p->V = large ? 6 : 4;
    p->warps = large ? 16 : 4;
    p->stages = large ? 2 : 3;
    p->group = large ? 4 : 0;
    p->nsub = dpd::batch_nsub(p->warps, 4, p->stages, p->V);
}

void free_plan(dpd_plan p)
{
    cudaFree(p->d_streams);
    cudaFree(p->d_items);
    cudaFree(p->d_tabs);
    cudaFree(p->d_h);
    cudaFree(p->d_status);
    delete p;
}

// Work list: streams by decreasing per-sample cost (B * T), in items of up to nsub
// sub-blocks of warps * 32 * V samples.  CTA b of a launch of G takes items b, b + G, ...
// With `contiguous` (equal_runs) those are one run of the ordered list of equal cost
// for each CTA, so a CTA stays with one model's code (the kernel holds one unrolled
// body per model, and its instruction fetch was an eighth of the stalls) and the SMs
// with little arithmetic per sample move their bytes while the others compute: 64
// streams of mixed models, 36.7 M samples, 121.4 us against 126.0 with full items
// dealt out in order.  The list goes to a new device buffer that replaces the plan's only
// once it holds the list, so on failure the plan keeps its previous list (and tiling)
// unchanged.
dpd_status build_items(dpd_plan p, int V, int warps, int nsub, bool contiguous)
{
    const int block = warps * 32 * V;
    std::vector<int> order(p->streams.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    // Costliest models first (B T per sample), and streams of the same model
    // next to each other, so that the items a CTA takes one after another
    // mostly run the same (B, T) code path.
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        const int ca = p->streams[a].B * p->streams[a].T, cb = p->streams[b].B * p->streams[b].T;
        if (ca != cb) return ca > cb;
        return p->streams[a].B > p->streams[b].B;
    });
    std::vector<dpd::BatchItem> items;
    auto put = [&](std::vector<dpd::BatchItem> &list, int si, int64_t from, int64_t count) {
        for (int64_t b = from; b < from + count; b += nsub)
            list.push_back({si, dpd::batch_tile(b, (int)std::min<int64_t>(nsub, from + count - b))});
    };
    double total = 0.0;
    auto blocks_of = [&](int si) { return (p->streams[si].n + block - 1) / block; };
    // Cost of a sub-block of a stream, in multiply-adds.  A sample: 4 B T, and what it takes
    // besides them (about the time of 28: one model at a time over 5.6 M samples, us per
    // launch, 60 multiply-adds 18.6, 100 26.7, 140 32.9), a part of a sub-block costing as
    // much as a whole one; and the share in what the stream's last item takes more.
    auto cost = [&](int si) {
        const int64_t blocks = blocks_of(si), missing = (nsub - blocks % nsub) % nsub;
        return (4.0 * p->streams[si].B * p->streams[si].T + 28.0) * block +
               kShortItem * (double)missing / (double)((nsub > 1 ? nsub - 1 : 1) * blocks);
    };
    for (int si : order) {
        if (blocks_of(si) > kMaxBlocks) return DPD_ERR_UNSUPPORTED;
        if (blocks_of(si) > 0) total += cost(si) * (double)blocks_of(si);
    }
    const int G = p->sm_count;
    if (!contiguous || total <= 0.0) {
        for (int si : order) put(items, si, 0, blocks_of(si));
    } else {
        std::vector<std::vector<dpd::BatchItem>> run((size_t)G);
        int k = 0;            // the CTA being filled
        double done = 0.0;    // cost given out
        for (int si : order) {
            const int64_t blocks = blocks_of(si);
            const double c = blocks > 0 ? cost(si) : 0.0;
            for (int64_t b = 0; b < blocks;) {
                const double room = total / G * (k + 1) - done;
                int64_t take = blocks - b;
                if (k < G - 1) take = std::min(take, (int64_t)(room / c + 0.5));
                if (take <= 0) {
                    ++k;
                    continue;
                }
                put(run[(size_t)k], si, b, take);
                b += take;
                done += c * (double)take;
            }
        }
        size_t rounds = 0;
        for (const auto &r : run) rounds = std::max(rounds, r.size());
        items.assign(rounds * (size_t)G, {-1, -1});   // the end of a CTA's list
        for (int b = 0; b < G; ++b)
            for (size_t r = 0; r < run[(size_t)b].size(); ++r) items[r * (size_t)G + b] = run[(size_t)b][r];
    }
    if (items.size() > (size_t)INT32_MAX) return DPD_ERR_UNSUPPORTED;
    dpd::BatchItem *d_new = nullptr;
    const size_t cap = std::max<size_t>(items.size(), 1);
    if (cudaMalloc(&d_new, cap * sizeof(dpd::BatchItem)) != cudaSuccess) return DPD_ERR_ALLOC;
    if (!items.empty() &&
        cudaMemcpy(d_new, items.data(), items.size() * sizeof(dpd::BatchItem), cudaMemcpyHostToDevice) !=
            cudaSuccess) {
        cudaFree(d_new);
        return DPD_ERR_CUDA;
    }
    cudaFree(p->d_items);
    p->d_items = d_new;
    p->nitems = (int)items.size();
    return DPD_OK;
}

}  // namespace

extern "C" {

dpd_status dpd_plan_batched(const dpd_stream_desc *descs, int count, int where, dpd_plan *out)
{
    if (!out || count < 0 || (count > 0 && !descs)) return DPD_ERR_INVALID_ARGUMENT;
    if (where != DPD_HOST && where != DPD_DEVICE) return DPD_ERR_INVALID_ARGUMENT;
    // validate every stream before touching the device
    size_t hfloats = 0, tfloats = 0;
    for (int i = 0; i < count; ++i) {
        const dpd_stream_desc &d = descs[i];
        const dpd_status mst = dpd::model_status(d.P, d.Q, d.M);
        if (mst != DPD_OK) return mst;
        if (d.n < 0 || !d.h) return DPD_ERR_INVALID_ARGUMENT;
        if (d.n > (int64_t)(INT64_MAX / sizeof(float2))) return DPD_ERR_INVALID_ARGUMENT;
        if (d.n > 0 && (!d.x || !d.y || !aligned(d.x, 16) || !aligned(d.y, 8))) return DPD_ERR_INVALID_ARGUMENT;
        if (!aligned(d.h, where == DPD_HOST ? 4 : 8)) return DPD_ERR_INVALID_ARGUMENT;
        const int Bp = nbranch(d.P), Bq = nbranch(d.Q), B = std::max(Bp, Bq), T = d.M + 1;
        hfloats += 2 * (size_t)((Bp + Bq) * T + 1);
        tfloats += (size_t)((dpd::wl_table_floats(B, T) * 4 + 15) / 16) * 4;
    }
    for (int i = 0; i < count; ++i) {   // outputs overlap no input and no other output
        const size_t bi = (size_t)descs[i].n * sizeof(float2);
        for (int j = 0; j < count; ++j) {
            const size_t bj = (size_t)descs[j].n * sizeof(float2);
            if (overlap(descs[i].y, bi, descs[j].x, bj)) return DPD_ERR_INVALID_ARGUMENT;
            if (j != i && overlap(descs[i].y, bi, descs[j].y, bj)) return DPD_ERR_INVALID_ARGUMENT;
        }
    }
    dpd_plan p = new (std::nothrow) dpd_plan_s();
    if (!p) return DPD_ERR_ALLOC;
    if (cudaGetDevice(&p->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, p->device) != cudaSuccess) {
        delete p;
        return DPD_ERR_CUDA;
    }
    if (cudaMalloc(&p->d_status, sizeof(int)) != cudaSuccess ||
        cudaMalloc(&p->d_h, std::max<size_t>(hfloats, 2) * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&p->d_tabs, std::max<size_t>(tfloats, 4) * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&p->d_streams, std::max(count, 1) * sizeof(dpd::BatchStream)) != cudaSuccess) {
        free_plan(p);
        return DPD_ERR_ALLOC;
    }
    if (cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess) {
        free_plan(p);
        return DPD_ERR_CUDA;
    }
    size_t hoff = 0, toff = 0;
    for (int i = 0; i < count; ++i) {
        const dpd_stream_desc &d = descs[i];
        const int Bp = nbranch(d.P), Bq = nbranch(d.Q), B = std::max(Bp, Bq), T = d.M + 1;
        const int K = (Bp + Bq) * T + 1;
        float2 *hdst = reinterpret_cast<float2 *>(p->d_h + hoff);
        const cudaMemcpyKind kind = where == DPD_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice;
        if (cudaMemcpy(hdst, d.h, sizeof(float2) * K, kind) != cudaSuccess ||
            dpd::launch_wl_table(hdst, Bp, Bq, T, p->d_tabs + toff, nullptr, 0) != cudaSuccess) {
            free_plan(p);
            return DPD_ERR_CUDA;
        }
        dpd::BatchStream st;
        st.x = static_cast<const float2 *>(d.x);
        st.y = static_cast<float2 *>(d.y);
        st.n = d.n;
        st.B = B;
        st.T = T;
        st.tab_off = (int)toff;
        st.tab_bytes = ((dpd::wl_table_floats(B, T) * 4 + 15) / 16) * 16;
        p->streams.push_back(st);
        if (B > 5 || T > 7) p->small = 0;
        hoff += 2 * (size_t)K;
        toff += (size_t)st.tab_bytes / 4;
    }
    p->tab_floats = (int64_t)toff;
    if (count > 0 &&
        cudaMemcpy(p->d_streams, p->streams.data(), count * sizeof(dpd::BatchStream), cudaMemcpyHostToDevice) !=
            cudaSuccess) {
        free_plan(p);
        return DPD_ERR_CUDA;
    }
    default_shape(p);
    dpd_status st = build_items(p, p->V, p->warps, p->nsub, equal_runs(p->V, p->warps, p->group, p->stages, p->nsub));
    if (st == DPD_OK && cudaDeviceSynchronize() != cudaSuccess) st = DPD_ERR_CUDA;
    if (st != DPD_OK) {
        free_plan(p);
        return st;
    }
    *out = p;
    return DPD_OK;
}

dpd_status dpd_plan_set_launch(dpd_plan p, int V, int warps, int stages, int ctas_per_sm, int group)
{
    if (!p) return DPD_ERR_INVALID_ARGUMENT;
    if ((V != 4 && V != 6 && V != 8) || warps < 1 || warps > 16 || stages < 2 || stages > 8 || ctas_per_sm < 0 || group < 0 ||
        (group > 0 && warps % group != 0))
        return DPD_ERR_INVALID_ARGUMENT;
    const int gw = group > 0 ? group : warps;
    if (dpd::batch_smem(warps, gw, stages, V) > dpd::kBatchSmemMax) return DPD_ERR_UNSUPPORTED;
    const int nsub = dpd::batch_nsub(warps, gw, stages, V);
    const bool runs = equal_runs(V, warps, group, stages, nsub);
    if (V != p->V || warps != p->warps || nsub != p->nsub ||
        runs != equal_runs(p->V, p->warps, p->group, p->stages, p->nsub)) {
        // Re-tile first: the new shape is kept only once its work list is on
        // the device; on failure the plan runs with its previous shape.
        const dpd_status st = build_items(p, V, warps, nsub, runs);
        if (st != DPD_OK) return st;
    }
    p->V = V;
    p->warps = warps;
    p->nsub = nsub;
    p->stages = stages;
    p->ctas_per_sm = ctas_per_sm;
    p->group = group;
    return DPD_OK;
}

dpd_status dpd_exec_batched(dpd_plan p, void *stream)
{
    if (!p) return DPD_ERR_INVALID_ARGUMENT;
    if (p->nitems == 0) return DPD_OK;
    if (!p->d_items || !p->d_streams || !p->d_tabs || !p->d_status) return DPD_ERR_INVALID_ARGUMENT;
    dpd::BatchArgs a;
    a.streams = p->d_streams;
    a.items = p->d_items;
    a.nitems = p->nitems;
    a.nstreams = (int)p->streams.size();
    a.tabs = p->d_tabs;
    a.tab_floats = p->tab_floats;
    a.status = p->d_status;
    a.gw = p->group;
    a.nsub = p->nsub;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = p->small ? dpd::launch_batched_57(a, p->V, p->warps, p->stages, p->ctas_per_sm, p->sm_count, s)
                             : dpd::launch_batched_68(a, p->V, p->warps, p->stages, p->ctas_per_sm, p->sm_count, s);
    return e == cudaSuccess ? DPD_OK : DPD_ERR_CUDA;
}

dpd_status dpd_plan_sync_status(dpd_plan p, void *stream)
{
    if (!p) return DPD_ERR_INVALID_ARGUMENT;
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return DPD_ERR_CUDA;
    int flags = 0;
    if (cudaMemcpy(&flags, p->d_status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return DPD_ERR_CUDA;
    if (flags && cudaMemset(p->d_status, 0, sizeof(int)) != cudaSuccess) return DPD_ERR_CUDA;
    if (flags & dpd::kFlagTimeout) return DPD_ERR_TIMEOUT;
    if (flags) return DPD_ERR_CUDA;
    return DPD_OK;
}

dpd_status dpd_plan_destroy(dpd_plan p)
{
    if (p) free_plan(p);
    return DPD_OK;
}

}  // extern "C"
