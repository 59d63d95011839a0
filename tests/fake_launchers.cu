// The kernel launchers that csrc/api.cu calls, on a CPU: the batch's record what they were
// given, with the cameras as the launch reads them when it runs; the others do nothing.
#include "fgs_internal.cuh"

#include "fake_cuda.h"

#include <cstring>
#include <vector>

struct Record {
    int what;                      // 0: batch front, 1: batch blend
    int views;
    uint32_t n_pad;
    const void* rgb;
    int null_args;                 // null (or too small) buffers among the launch's
    float t[64][3];                // the cameras' translations
};

static std::vector<Record> g_records;
static long g_nulls = 0;           // null buffers given to the single-view launches

extern "C" {

void fake_clear() { g_records.clear(); }
long fake_nulls() { return g_nulls; }
long fake_records() { return (long)g_records.size(); }
void fake_record(long i, int* head, uint64_t* rgb, float* t)
{
    const Record& r = g_records.at((size_t)i);
    head[0] = r.what, head[1] = r.views, head[2] = (int)r.n_pad, head[3] = r.null_args;
    *rgb = (uint64_t)r.rgb;
    memcpy(t, r.t, sizeof r.t);
}

}  // extern "C"

namespace fgs {

template <class... P>
static int nulls(const P*... p)
{
    return (0 + ... + (p == nullptr));
}

static void record(int what, const DevCamera* cams, int V, uint32_t n_pad, const void* rgb, int null_args,
                   cudaStream_t s)
{
    fake_push(s, [=] {
        Record r{what, V, n_pad, rgb, null_args, {}};
        for (int v = 0; v < V; ++v) memcpy(r.t[v], cams[v].t, sizeof r.t[v]);
        g_records.push_back(r);
    });
}

int occ_filter_pred() { return 1; }
int occ_filter_anc() { return 1; }
int occ_compact() { return 1; }
int occ_scatter() { return 1; }
int occ_segsort() { return 1; }
int occ_tile_scan() { return 1; }
void launch_frame_begin(const FrameBegin&, cudaStream_t) {}
void launch_filter_pred(const DevTree&, const DevCamera&, uint32_t* pbits, FrameState*, const FrameBegin& f, int,
                        cudaStream_t)
{
    g_nulls += nulls(pbits, f.st, f.tile_cnt, f.sel_cnt);
}
void launch_chunk_boxes(const DevTree&, int, cudaStream_t) {}
void launch_filter_anc(const DevTree&, const uint32_t* pbits, uint32_t* selbits, uint32_t* sel_cnt, int, cudaStream_t)
{
    g_nulls += nulls(pbits, selbits, sel_cnt);
}
void launch_wait_probe(const unsigned long long*, FrameState*, cudaStream_t) {}
void launch_compact(const uint32_t*, uint32_t, uint32_t*, uint32_t, unsigned long long*, FrameState*, int, cudaStream_t) {}
void launch_compact_counted(const uint32_t* selbits, uint32_t, uint32_t* sel, uint32_t, const uint32_t* sel_cnt,
                            FrameState* st, cudaStream_t)
{
    g_nulls += nulls(selbits, sel, sel_cnt, st);
}
void launch_project(const DevTree&, const DevCamera&, const uint32_t* sel, float* splat, uint4* foot, uint32_t* tile_cnt,
                    FrameState* st, int, cudaStream_t)
{
    g_nulls += nulls(sel, splat, foot, tile_cnt, st);
}
void launch_tile_scan(uint32_t* tile_cnt, uint2* ranges, uint32_t, uint32_t* large, unsigned long long,
                      unsigned long long* lookback, FrameState* st, int, cudaStream_t)
{
    g_nulls += nulls(tile_cnt, ranges, large, lookback, st);
}
void launch_scatter(const DevCamera&, const uint4* foot, uint32_t* cursor, unsigned long long* items, unsigned long long,
                    FrameState* st, int, cudaStream_t)
{
    g_nulls += nulls(foot, cursor, items, st);
}
void launch_segsort(const uint2* ranges, uint32_t, const uint32_t* large, unsigned long long* items,
                    unsigned long long* keys_out, uint32_t* vals_out, uint32_t* heavy, FrameState* st, int, cudaStream_t)
{
    g_nulls += nulls(ranges, large, items, keys_out, vals_out, heavy, st);
}
void launch_blend(const DevCamera&, const uint2* ranges, const uint32_t* heavy, const uint32_t* vals, const float* splat,
                  float* rgb, float*, uint2*, FrameState* st, bool, cudaStream_t)
{
    g_nulls += nulls(ranges, heavy, vals, splat, rgb, st);
}
void launch_blend_kpc(const DevCamera&, const uint2*, const uint32_t*, const float*, float*, float*, FrameState*,
                      cudaStream_t) {}
void launch_eval_exp(const float*, float*, uint64_t, cudaStream_t) {}
void launch_prep_params(const DevTree&, const float*, const float*, const float*, const float*, const float*, int,
                        cudaStream_t) {}
void launch_backward(const DevTree&, const DevCamera&, const uint2*, const uint32_t*, const uint32_t*, const float*,
                     uint2*, bool, const uint32_t*, const uint32_t*, const float*, float*, const float* const*,
                     float* const*, bool, int, FrameState*, cudaStream_t) {}
void launch_levelwise_step(const DevTree&, const DevCamera&, const uint32_t*, const uint32_t*, const uint32_t*, uint32_t,
                           uint32_t*, uint32_t*, uint32_t*, cudaStream_t) {}
void launch_batch_front(const DevTree& t, const DevCamera* cams, int V, uint32_t, const uint32_t* tile_base, uint32_t* pbits,
                        uint32_t* selbits, uint32_t* sel, uint32_t, float* splat, uint4* foot, uint32_t* tile_cnt,
                        uint32_t* large, uint32_t* heavy, unsigned long long* items, unsigned long long* keys,
                        uint32_t* vals, unsigned long long, uint32_t* sel_cnt, unsigned long long* lb_scan,
                        uint2* ranges, FrameState* st, int, cudaStream_t s)
{
    const size_t words = (size_t)t.n_pad / 32 * V;
    record(0, cams, V, t.n_pad, nullptr,
           nulls(cams, tile_base, pbits, selbits, sel, splat, foot, tile_cnt, large, heavy, items, keys, vals, sel_cnt,
                 lb_scan, ranges, st) +
               (fake_size(pbits) < 4 * words) + (fake_size(selbits) < 4 * words) +
               (fake_size(sel_cnt) < 4 * batch_sel_tiles(words)),
           s);
}
void launch_batch_blend(const DevCamera* cams, int V, uint32_t, const uint32_t* tile_base,
                        const unsigned long long* img_off, const uint2* ranges, const uint32_t* heavy,
                        const uint32_t* vals, const float* splat, float* rgb, float*, FrameState* st, cudaStream_t s)
{
    record(1, cams, V, 0, rgb, nulls(cams, tile_base, img_off, ranges, heavy, vals, splat, rgb, st), s);
}
// a kernel that takes the cameras by value: they are read when it is launched
void launch_batch_cameras(const DevCamera* cams, int V, DevCamera* dst, cudaStream_t s)
{
    std::vector<DevCamera> v(cams, cams + V);
    fake_push(s, [=] { memcpy(dst, v.data(), v.size() * sizeof(DevCamera)); });
}

}  // namespace fgs
