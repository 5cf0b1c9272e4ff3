// batch.cu -- uneven batches: many scalar fields of different truncations
// transformed by one graph launch.
//
// Each distinct (lmax, nlat, nphi) gets one plan; every field keeps its own
// intermediate buffer.  The host builds, once, a tile list per stage covering
// all fields -- synthesis Legendre tiles (field, m, pair block), analysis
// Legendre tiles (field, m), FFT tiles (field, pair group) -- sorted longest
// first (the load-balancing concern of Sec. 3.3, applied to CTAs instead of
// threads).  A transform is then: copy the per-field pointer table, reset the
// work counters, one persistent Legendre kernel and one persistent FFT kernel
// (in the order of Sec. 2.2 / 2.3).  That sequence is captured once into a
// CUDA graph and replayed on every call.  The persistent kernels take tiles
// with atomicAdd on a counter and never wait on each other.
//
// Tensor-core mode: the fields of one shape form a group whose spectra (a
// gather kernel copies them in, or the results out) and intermediates are
// contiguous, so each group's Legendre stage is one batched tcgen05
// contraction against that plan's P panels.  The automatic mode times both and
// keeps the faster.
//
// Up to kMaxGroups shapes, the FFTs are one launch per shape, and each shape's
// copies, contraction and FFT a branch of the graph of their own: one shape's FFT
// fills the SMs that another's contraction leaves.
// (The persistent FFT kernel fetches its tile, the field's plan and pointers one
// after the other before any data, and runs the registers and shared memory of
// the largest length: 99 / 86 us for 96 fields of N = 63 .. 511, against 37 / 38
// us for the four launches on their own.)  More shapes keep the persistent kernel.
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <memory>
#include <new>
#include <string>
#include <tuple>
#include <vector>

#include "sht_internal.h"

namespace {
// Shapes with launches and graph branches of their own.  The bound keeps the graph small;
// it is not where the branches stop paying (round trip, 6 fields per shape, N = 40 ..
// 510, branches against persistent kernels: tensor cores 8 shapes 248 / 417 us, 9 285 /
// 471, 32 950 / 1509; CUDA cores 8 shapes 407 / 465, 9 465 / 540, 32 1484 / 1713).
constexpr size_t kMaxGroups = 8;

// One copy of the gather (synthesis) or scatter (analysis) of the tensor-core mode.
struct BatchCopy {
    const float2 *src;
    float2 *dst;
    long long n;   // complex values
};
}  // namespace

struct sht_batch_plan {
    int nfields = 0;
    int device = 0;
    int mode = SHT_F32;                    // SHT_F32 (persistent CUDA-core kernels) or SHT_TC_BF16X3
    std::vector<std::vector<int>> group_fields;   // tensor cores: the fields of each plan, in order
    float *d_gspec = nullptr;              // ... contiguous spectra of each group
    std::vector<size_t> gspec_off;         // ... per group, floats
    std::vector<size_t> field_gspec;       // ... per field: its slot in d_gspec, floats
    std::vector<size_t> ginter_off;        // ... per group: its contiguous intermediate in d_inter, floats
    std::vector<size_t> inter_tc;          // ... per field: its intermediate in that layout
    // per call: pointer table of the group FFTs and copy list, fields in group order, one
    // upload from the direction's own pinned staging, beside the field table's
    struct Staging {
        unsigned char *up = nullptr;
        sht::BatchField *fields = nullptr;
    };
    Staging stage[2];
    std::vector<Staging> captured;         // of calls that a caller captured into a graph of its own
    unsigned char *d_up = nullptr;
    std::vector<size_t> group_first;       // first entry of each group in that order
    std::vector<int> order;                // groups by falling size
    bool grouped = false;                  // FFTs by group
    std::vector<unsigned long long> fft_plan[2];   // per direction and shape: passes of the persistent FFT kernel's tiles
    sht::BatchPtrs *h_ptrs(const Staging &st) const { return reinterpret_cast<sht::BatchPtrs *>(st.up); }
    BatchCopy *h_copies(const Staging &st) const
    {
        return reinterpret_cast<BatchCopy *>(st.up + sizeof(sht::BatchPtrs) * nfields);
    }
    const sht::BatchPtrs *d_ptrs() const { return reinterpret_cast<const sht::BatchPtrs *>(d_up); }
    const BatchCopy *d_copies() const
    {
        return reinterpret_cast<const BatchCopy *>(d_up + sizeof(sht::BatchPtrs) * nfields);
    }
    size_t up_bytes() const { return (sizeof(sht::BatchPtrs) + sizeof(BatchCopy)) * nfields; }
    cudaError_t alloc(Staging &st) const
    {
        cudaError_t e = cudaMallocHost(&st.fields, sizeof(sht::BatchField) * nfields);
        return e == cudaSuccess ? cudaMallocHost(&st.up, up_bytes()) : e;
    }
    static void release(Staging &st)
    {
        if (st.fields) cudaFreeHost(st.fields);
        if (st.up) cudaFreeHost(st.up);
        st = Staging();
    }
    float tuned_ms[2] = {0.f, 0.f};        // automatic mode: round trip per path (CUDA cores, tensor cores)
    std::vector<std::unique_ptr<sht::Plan>> plans;   // one per distinct shape
    std::vector<int> field_plan;
    std::vector<int> lmax, nlat, nphi;
    sht::BatchField *d_fields = nullptr;
    int4 *d_tiles = nullptr;               // [synth legendre | synth fft | analys fft | analys legendre]
    int ntile[4] = {0, 0, 0, 0};
    size_t tile_off[4] = {0, 0, 0, 0};
    int *d_counters = nullptr;             // 4 counters
    float *d_inter = nullptr;
    std::vector<size_t> inter_off;
    size_t fft_smem = 0;
    int ctas_legendre_syn = 0, ctas_legendre_ana = 0, ctas_fft = 0;
    cudaGraphExec_t graph[2] = {nullptr, nullptr};   // synthesis, analysis
    cudaEvent_t used[2] = {nullptr, nullptr};        // last launch of each direction (guards its staging)
    cudaEvent_t done = nullptr;                      // last launch (guards the device buffers)
};

namespace {

int bfail(int code, const std::string &msg) { return sht::set_error(code, msg); }

void free_batch(sht_batch_plan *b)
{
    if (!b) return;
    for (auto g : b->graph)
        if (g) cudaGraphExecDestroy(g);
    if (b->done) cudaEventDestroy(b->done);
    for (int dir = 0; dir < 2; ++dir) {
        if (b->used[dir]) cudaEventDestroy(b->used[dir]);
        b->release(b->stage[dir]);
    }
    for (auto &st : b->captured) b->release(st);
    cudaFree(b->d_up);
    cudaFree(b->d_gspec);
    cudaFree(b->d_fields);
    cudaFree(b->d_tiles);
    cudaFree(b->d_counters);
    cudaFree(b->d_inter);
    for (auto &p : b->plans)
        if (p) sht::plan_free(*p);
    delete b;
}

// Gather / scatter of the tensor-core mode: blockIdx.y = copy, kCopyPer complex
// values per thread.  16 bytes at a time where source and destination lie alike
// on 16 bytes (a field's spectrum starts on 8), all loads before the stores.
constexpr int kCopyPer = 8;
__global__ void __launch_bounds__(256) k_batch_copy(const BatchCopy *__restrict__ copies)
{
    const BatchCopy c = copies[blockIdx.y];
    const size_t sa = reinterpret_cast<size_t>(c.src) & 15, da = reinterpret_cast<size_t>(c.dst) & 15;
    if (sa == da) {
        const long long lead = sa ? 1 : 0, n4 = (c.n - lead) >> 1;
        const float4 *src = reinterpret_cast<const float4 *>(c.src + lead);
        float4 *dst = reinterpret_cast<float4 *>(c.dst + lead);
        const long long i0 = (long long)blockIdx.x * (256 * kCopyPer / 2) + threadIdx.x;
        float4 v[kCopyPer / 2];
#pragma unroll
        for (int u = 0; u < kCopyPer / 2; ++u)
            if (i0 + 256 * u < n4) v[u] = src[i0 + 256 * u];
#pragma unroll
        for (int u = 0; u < kCopyPer / 2; ++u)
            if (i0 + 256 * u < n4) dst[i0 + 256 * u] = v[u];
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            if (lead) c.dst[0] = c.src[0];
            if (lead + 2 * n4 < c.n) c.dst[c.n - 1] = c.src[c.n - 1];
        }
        return;
    }
    const long long i0 = (long long)blockIdx.x * (256 * kCopyPer) + threadIdx.x;
#pragma unroll
    for (int u = 0; u < kCopyPer; ++u)
        if (i0 + 256 * u < c.n) c.dst[i0 + 256 * u] = c.src[i0 + 256 * u];
}

// Fill the per-call tables.
void fill_fields(sht_batch_plan *b, bool synth, void *const *in, void *const *out, const sht_batch_plan::Staging &st)
{
    const bool tc = b->mode == SHT_TC_BF16X3;
    for (size_t g = 0; g < b->group_fields.size(); ++g)
        for (size_t i = 0; i < b->group_fields[g].size(); ++i) {
            const int f = b->group_fields[g][i];
            const size_t at = b->group_first[g] + i;
            sht::BatchPtrs &q = b->h_ptrs(st)[at];
            q.in = static_cast<const float *>(in[f]);
            q.out = static_cast<float *>(out[f]);
            q.inter = b->d_inter + (tc ? b->inter_tc[f] : b->inter_off[f]);
            if (!tc) continue;
            BatchCopy &c = b->h_copies(st)[at];
            float2 *slot = reinterpret_cast<float2 *>(b->d_gspec + b->field_gspec[f]);
            c.n = b->plans[g]->nlm;
            c.src = synth ? static_cast<const float2 *>(in[f]) : slot;
            c.dst = synth ? slot : static_cast<float2 *>(out[f]);
        }
    if (tc && b->grouped) return;   // only the persistent kernels read the field table
    for (int f = 0; f < b->nfields; ++f) {
        sht::BatchField &bf = st.fields[f];
        const sht::Plan &p = *b->plans[b->field_plan[f]];
        bf.pv = p.view32();
        bf.pv.fftplan = b->fft_plan[synth ? 0 : 1][b->field_plan[f]];
        bf.in = static_cast<const float *>(in[f]);
        bf.out = static_cast<float *>(out[f]);
        bf.inter = b->d_inter + (tc ? b->inter_tc[f] : b->inter_off[f]);
        // row FFT tiles for power-of-two lengths <= 2^10, else the mixed-radix kernel
        const int H = p.nphi / 2;
        int logH = 0;
        while ((1 << logH) < H) ++logH;
        bf.logH = (1 << logH) == H ? logH : 31;
        bf.G = sht::batch_fft_group(H, p.npairs);
    }
}

// Copies of `count` fields from entry `first` of the list, of at most n values each.
cudaError_t copies(sht_batch_plan *b, size_t first, size_t count, int n, cudaStream_t s)
{
    const dim3 grid((unsigned)((n + 256 * kCopyPer - 1) / (256 * kCopyPer)), (unsigned)count);
    k_batch_copy<<<grid, 256, 0, s>>>(b->d_copies() + first);
    return cudaGetLastError();
}

// One group's copies, contraction and FFT.
cudaError_t group_copies(sht_batch_plan *b, int g, cudaStream_t s)
{
    return copies(b, b->group_first[g], b->group_fields[g].size(), b->plans[g]->nlm, s);
}

cudaError_t group_contraction(sht_batch_plan *b, bool synth, int g, cudaStream_t s)
{
    float *spec = b->d_gspec + b->gspec_off[g], *inter = b->d_inter + b->ginter_off[g];
    const int nb = (int)b->group_fields[g].size();
    return synth ? sht::tc_batch_legendre(*b->plans[g], true, spec, inter, nb, s)
                 : sht::tc_batch_legendre(*b->plans[g], false, inter, spec, nb, s);
}

cudaError_t group_fft(sht_batch_plan *b, bool synth, int g, cudaStream_t s)
{
    return sht::launch_group_fft(synth, b->plans[g]->view32(), b->d_ptrs() + b->group_first[g],
                                 (int)b->group_fields[g].size(), s);
}

// A stream per group beside `main` while a graph is captured (empty otherwise:
// every step then runs on `main`).  Fork and join through events.
struct Branches {
    cudaStream_t main = nullptr;
    std::vector<cudaStream_t> streams;
    std::vector<cudaEvent_t> events;
    cudaError_t err = cudaSuccess;

    cudaStream_t of(int g) const { return streams.empty() ? main : streams[g]; }
    // `to` goes on once what `from` holds so far is done
    void after(cudaStream_t to, cudaStream_t from)
    {
        if (to == from || err != cudaSuccess) return;
        cudaEvent_t ev = nullptr;
        err = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (err != cudaSuccess) return;
        events.push_back(ev);
        err = cudaEventRecord(ev, from);
        if (err == cudaSuccess) err = cudaStreamWaitEvent(to, ev, 0);
    }
    void run(cudaError_t e) { if (err == cudaSuccess) err = e; }
    cudaError_t open(cudaStream_t s, int groups, bool fork)
    {
        main = s;
        for (int g = 0; g < groups && fork && err == cudaSuccess; ++g) {
            cudaStream_t t = nullptr;
            err = cudaStreamCreateWithFlags(&t, cudaStreamNonBlocking);
            if (err == cudaSuccess) streams.push_back(t);
        }
        return err;
    }
    ~Branches()
    {
        for (cudaEvent_t e : events) cudaEventDestroy(e);
        for (cudaStream_t t : streams) cudaStreamDestroy(t);
    }
};

// Enqueue the steps of one direction on stream s, those of a group on its branch.
cudaError_t enqueue(sht_batch_plan *b, bool synth, cudaStream_t s, Branches &br, const sht_batch_plan::Staging &st)
{
    const bool tc = b->mode == SHT_TC_BF16X3;
    const int ng = (int)b->plans.size();
    br.run(cudaMemcpyAsync(b->d_up, st.up, b->up_bytes(), cudaMemcpyHostToDevice, s));
    if (!tc || !b->grouped) {
        br.run(cudaMemcpyAsync(b->d_fields, st.fields, sizeof(sht::BatchField) * b->nfields,
                               cudaMemcpyHostToDevice, s));
        br.run(cudaMemsetAsync(b->d_counters, 0, 4 * sizeof(int), s));
    }
    const auto persistent_fft = [&] {
        const int k = synth ? 1 : 2;
        br.run(sht::launch_batch_fft(synth, b->d_fields, b->d_tiles + b->tile_off[k], b->ntile[k], b->d_counters + k,
                                     b->ctas_fft, b->fft_smem, s));
    };
    const auto all_copies = [&] {   // blocks past the end of a shorter field return at once
        int n = 0;
        for (const auto &p : b->plans) n = std::max(n, p->nlm);
        br.run(copies(b, 0, (size_t)b->nfields, n, s));
    };
    const auto legendre = [&] {
        const int k = synth ? 0 : 3;
        br.run(sht::launch_batch_legendre(synth, b->d_fields, b->d_tiles + b->tile_off[k], b->ntile[k],
                                          b->d_counters + k, synth ? b->ctas_legendre_syn : b->ctas_legendre_ana, s));
    };
    // each group's steps follow one another on its branch, the largest group first
    if (synth && !tc) legendre();
    if (!synth && !b->grouped) persistent_fft();
    if (synth && tc && !b->grouped) all_copies();
    for (int i = 0; i < ng && (tc || b->grouped); ++i) {
        const int g = b->order[i];
        cudaStream_t gs = br.of(g);
        br.after(gs, s);
        if (!synth && b->grouped) br.run(group_fft(b, false, g, gs));
        if (tc && synth && b->grouped) br.run(group_copies(b, g, gs));
        if (tc) br.run(group_contraction(b, synth, g, gs));
        if (tc && !synth && b->grouped) br.run(group_copies(b, g, gs));
        if (synth && b->grouped) br.run(group_fft(b, true, g, gs));
    }
    for (int g = 0; g < ng; ++g) br.after(s, br.of(g));
    if (!synth && tc && !b->grouped) all_copies();
    if (synth && !b->grouped) persistent_fft();
    if (!synth && !tc) legendre();
    return br.err;
}

int run(sht_batch_plan *b, bool synth, void *const *in, void *const *out, int use_graph, void *stream)
{
    if (!b) return bfail(SHT_EINVAL, "null batch handle");
    if (!in || !out) return bfail(SHT_EINVAL, "null pointer array");
    for (int f = 0; f < b->nfields; ++f)
        if (!in[f] || !out[f]) return bfail(SHT_EINVAL, "null data pointer for field " + std::to_string(f));
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != b->device)
        return bfail(SHT_EINVAL, "current CUDA device differs from the batch plan's device");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // this direction's previous launch copies its staging when it runs: the host
    // waits for it before overwriting; the other direction's launch may still be
    // running, and the stream waits for it before this one uses the device buffers
    const int dir = synth ? 0 : 1;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) cudaGetLastError();
    if (cap == cudaStreamCaptureStatusActive && use_graph)
        return bfail(SHT_ECUDA, "a batch graph cannot be launched into a stream capture: call with use_graph = 0");
    if (cap == cudaStreamCaptureStatusActive) {
        // into the caller's graph, whose replays read the staging again: one of the call's own, kept
        // with the plan, and no events, which would tie the graph to calls outside of it
        sht_batch_plan::Staging st;
        cudaError_t e = b->alloc(st);
        if (e == cudaSuccess) {
            fill_fields(b, synth, in, out, st);
            Branches br;
            br.open(s, 0, false);
            e = enqueue(b, synth, s, br, st);
        }
        b->captured.push_back(st);
        if (e != cudaSuccess) return bfail(SHT_ECUDA, std::string("batch launch under capture: ") + cudaGetErrorString(e));
        return SHT_OK;
    }
    const sht_batch_plan::Staging &st = b->stage[dir];
    cudaError_t e = cudaEventSynchronize(b->used[dir]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, b->done, 0);
    if (e != cudaSuccess) return bfail(SHT_ECUDA, std::string("waiting for the previous batch call: ") + cudaGetErrorString(e));
    fill_fields(b, synth, in, out, st);
    if (use_graph) {
        if (!b->graph[dir]) {
            cudaStream_t cs;
            e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
            if (e != cudaSuccess) return bfail(SHT_ECUDA, "cudaStreamCreate failed");
            cudaGraph_t g = nullptr;
            e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                Branches br;
                cudaError_t e2 = br.open(cs, (int)b->plans.size(), b->grouped);
                if (e2 == cudaSuccess) e2 = enqueue(b, synth, cs, br, st);
                e = cudaStreamEndCapture(cs, &g);
                if (e == cudaSuccess) e = e2;
            }
            if (e == cudaSuccess) e = cudaGraphInstantiate(&b->graph[dir], g, 0);
            if (g) cudaGraphDestroy(g);
            cudaStreamDestroy(cs);
            if (e != cudaSuccess) {
                b->graph[dir] = nullptr;
                return bfail(SHT_ECUDA, std::string("capturing the batch graph: ") + cudaGetErrorString(e));
            }
        }
        e = cudaGraphLaunch(b->graph[dir], s);
    } else {
        Branches br;
        br.open(s, 0, false);
        e = enqueue(b, synth, s, br, st);
    }
    if (e == cudaSuccess) e = cudaEventRecord(b->used[dir], s);
    if (e == cudaSuccess) e = cudaEventRecord(b->done, s);
    if (e != cudaSuccess) return bfail(SHT_ECUDA, std::string("batch launch: ") + cudaGetErrorString(e));
    return SHT_OK;
}

// The captured graphs run the path they were captured for.
void drop_graphs(sht_batch_plan *b)
{
    for (auto &g : b->graph) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
}

// Automatic mode: time a synthesis + analysis of zero fields on each path and
// keep the faster; as graphs, after a warm-up, since only there the groups' steps
// overlap (96 fields of N = 63 .. 511: 221 us, 281 us by direct launches).
int choose_mode(sht_batch_plan *b)
{
    const int nf = b->nfields;
    std::vector<size_t> so(nf), go(nf);
    size_t bytes = 0;
    for (int f = 0; f < nf; ++f) {
        const sht::Plan &p = *b->plans[b->field_plan[f]];
        so[f] = bytes;
        bytes = (bytes + (size_t)p.nlm * 8 + 255) & ~(size_t)255;
        go[f] = bytes;
        bytes = (bytes + (size_t)p.nlat * p.nphi * 4 + 255) & ~(size_t)255;
    }
    unsigned char *buf = nullptr;
    cudaStream_t s = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaMalloc(&buf, bytes);
    if (e == cudaSuccess) e = cudaMemset(buf, 0, bytes);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    std::vector<void *> spec(nf), grid(nf);
    for (int f = 0; f < nf && buf; ++f) {
        spec[f] = buf + so[f];
        grid[f] = buf + go[f];
    }
    int rc = SHT_OK;
    float best = 0.f;
    int best_mode = SHT_F32;
    const int modes[2] = {SHT_F32, SHT_TC_BF16X3};
    for (int k = 0; k < 2 && e == cudaSuccess && rc == SHT_OK; ++k) {
        b->mode = modes[k];
        for (int it = 0; it < 5 && rc == SHT_OK; ++it) {
            if (it == 2) e = cudaEventRecord(e0, s);
            rc = run(b, true, spec.data(), grid.data(), 1, s);
            if (rc == SHT_OK) rc = run(b, false, grid.data(), spec.data(), 1, s);
        }
        if (rc != SHT_OK) break;
        if (e == cudaSuccess) e = cudaEventRecord(e1, s);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        drop_graphs(b);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        b->tuned_ms[k] = ms / 3.f;
        if (e == cudaSuccess && (k == 0 || ms < best)) {
            best = ms;
            best_mode = modes[k];
        }
    }
    if (s) cudaStreamSynchronize(s);
    drop_graphs(b);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (s) cudaStreamDestroy(s);
    cudaFree(buf);
    b->mode = best_mode;
    if (rc != SHT_OK) return rc;
    if (e != cudaSuccess) return bfail(SHT_ECUDA, std::string("timing the batch paths: ") + cudaGetErrorString(e));
    return SHT_OK;
}

}  // namespace

extern "C" {

int sht_batch_create(int nfields, const int *lmax, const int *nlat, const int *nphi, sht_batch *out)
{
    return sht_batch_create_mode(nfields, lmax, nlat, nphi, SHT_F32, out);
}

int sht_batch_create_mode(int nfields, const int *lmax, const int *nlat, const int *nphi, int mode, sht_batch *out)
{
    if (!out) return bfail(SHT_EINVAL, "out is NULL");
    *out = nullptr;
    if (nfields < 1 || !lmax || !nlat || !nphi) return bfail(SHT_EINVAL, "need nfields >= 1 and size arrays");
    if (mode != SHT_F32 && mode != SHT_TC_BF16X3 && mode != SHT_F32_AUTO)
        return bfail(SHT_EINVAL, "batch mode must be SHT_F32, SHT_TC_BF16X3 or SHT_F32_AUTO");
    for (int f = 0; f < nfields; ++f) {
        if (lmax[f] < 0 || nlat[f] < lmax[f] + 1 || nphi[f] < 2 * lmax[f] + 1)
            return bfail(SHT_EINVAL, "field " + std::to_string(f) + ": need nlat >= lmax+1 and nphi >= 2 lmax + 1");
        if (nphi[f] < 2 || nphi[f] > 4096 || nphi[f] % 2 != 0 || sht::fft_plan_of(nphi[f] / 2) == sht::kFftPlanBad)
            return bfail(SHT_EUNSUPPORTED, "field " + std::to_string(f) + ": nphi must be 2 x 2^a 3^b 5^c in [2, 4096]");
        if ((nlat[f] + 1) / 2 > sht::kBatchMaxPairs)
            return bfail(SHT_EUNSUPPORTED, "field " + std::to_string(f) + ": nlat > 1024 is not supported in a batch");
    }
    sht_batch_plan *b = new (std::nothrow) sht_batch_plan;
    if (!b) return bfail(SHT_ENOMEM, "host allocation failed");
    b->nfields = nfields;
    b->lmax.assign(lmax, lmax + nfields);
    b->nlat.assign(nlat, nlat + nfields);
    b->nphi.assign(nphi, nphi + nfields);
    cudaGetDevice(&b->device);
    std::map<std::tuple<int, int, int>, int> shape_plan;
    for (int f = 0; f < nfields; ++f) {
        auto key = std::make_tuple(lmax[f], nlat[f], nphi[f]);
        auto it = shape_plan.find(key);
        if (it == shape_plan.end()) {
            auto p = std::make_unique<sht::Plan>();
            p->lmax = lmax[f];
            p->mmax = lmax[f];
            p->nlat = nlat[f];
            p->nphi = nphi[f];
            std::string err;
            int rc = sht::plan_build(*p, err);
            if (!rc) rc = sht::plan_seeds32(*p, err);   // the CUDA-core kernels restart from these
            if (rc) {
                sht::plan_free(*p);
                free_batch(b);
                return bfail(rc, err);
            }
            it = shape_plan.emplace(key, (int)b->plans.size()).first;
            b->plans.push_back(std::move(p));
        }
        b->field_plan.push_back(it->second);
    }
    b->group_fields.assign(b->plans.size(), std::vector<int>());
    for (int f = 0; f < nfields; ++f) b->group_fields[b->field_plan[f]].push_back(f);
    b->grouped = b->plans.size() <= kMaxGroups;
    size_t first = 0;
    std::vector<double> work;   // of a group: panel bytes and data
    for (size_t g = 0; g < b->plans.size(); ++g) {
        const sht::Plan &p = *b->plans[g];
        b->group_first.push_back(first);
        first += b->group_fields[g].size();
        b->order.push_back((int)g);
        for (int dir = 0; dir < 2; ++dir) b->fft_plan[dir].push_back(sht::tile_fft_plan32(p.nphi / 2, dir == 0));
        work.push_back((double)p.nlm * p.npairs * 4 + (double)b->group_fields[g].size() * p.nlat * p.nphi * 8);
    }
    std::stable_sort(b->order.begin(), b->order.end(), [&](int x, int y) { return work[x] > work[y]; });
    // intermediates, tile lists (longest first)
    size_t inter = 0;
    std::vector<std::pair<double, int4>> syn, ffts, ana;
    size_t smem = 0;
    for (int f = 0; f < nfields; ++f) {
        const sht::Plan &p = *b->plans[b->field_plan[f]];
        b->inter_off.push_back(inter);
        inter += (size_t)(p.mmax + 1) * p.npairs * 4;  // floats
        inter = (inter + 63) & ~(size_t)63;
        const int npb = (p.npairs + sht::kBatchSynthPairs - 1) / sht::kBatchSynthPairs;
        for (int m = 0; m <= p.mmax; ++m) {
            for (int pb = 0; pb < npb; ++pb) {
                const int np = std::min(sht::kBatchSynthPairs, p.npairs - pb * sht::kBatchSynthPairs);
                syn.push_back({(double)(p.lmax - m + 1) * (np + 32), make_int4(f, m, pb, 0)});
            }
            const int nseg = (p.lmax - m + sht::kSeedSeg) / sht::kSeedSeg;
            for (int seg = 0; seg < nseg; seg += sht::kBatchAnalysSegs)
                ana.push_back({(double)std::min(sht::kBatchAnalysSegs, nseg - seg) * (p.npairs + 32),
                               make_int4(f, m, seg, 0)});
        }
        int logH = 0;
        while ((1 << logH) < p.nphi / 2) ++logH;
        const int G = sht::batch_fft_group(p.nphi / 2, p.npairs);
        smem = std::max(smem, sht::batch_fft_smem(p.nphi / 2, G));
        for (int p0 = 0; p0 < p.npairs; p0 += G)
            ffts.push_back({(double)G * p.nphi * (logH + 2) + p.mmax, make_int4(f, p0, 0, 0)});
    }
    // tensor-core layout: each group's intermediates and spectra contiguous
    bool tc_ok = mode != SHT_F32;
    size_t inter_tc = 0, gspec = 0;
    b->inter_tc.assign(nfields, 0);
    b->field_gspec.assign(nfields, 0);
    for (size_t g = 0; g < b->plans.size() && tc_ok; ++g) {
        const sht::Plan &p = *b->plans[g];
        const size_t stride = (size_t)(p.mmax + 1) * p.npairs * 4;
        b->ginter_off.push_back(inter_tc);
        b->gspec_off.push_back(gspec);
        for (size_t i = 0; i < b->group_fields[g].size(); ++i) {
            b->inter_tc[b->group_fields[g][i]] = inter_tc + i * stride;
            b->field_gspec[b->group_fields[g][i]] = gspec + i * (size_t)p.nlm * 2;
        }
        inter_tc = (inter_tc + b->group_fields[g].size() * stride + 63) & ~(size_t)63;
        gspec = (gspec + b->group_fields[g].size() * (size_t)p.nlm * 2 + 63) & ~(size_t)63;
        const int rc = sht::tc_batch_prepare(*b->plans[g], (int)b->group_fields[g].size());
        if (rc) {
            if (mode == SHT_TC_BF16X3) {
                free_batch(b);
                return rc;   // message set by the preparation
            }
            tc_ok = false;   // automatic mode: keep the CUDA-core path
        }
    }
    if (tc_ok) inter = std::max(inter, inter_tc);
    auto by_cost = [](const std::pair<double, int4> &a, const std::pair<double, int4> &c) { return a.first > c.first; };
    std::stable_sort(syn.begin(), syn.end(), by_cost);
    std::stable_sort(ffts.begin(), ffts.end(), by_cost);
    std::stable_sort(ana.begin(), ana.end(), by_cost);
    std::vector<int4> tiles;
    auto append = [&](int k, const std::vector<std::pair<double, int4>> &v) {
        b->tile_off[k] = tiles.size();
        b->ntile[k] = (int)v.size();
        for (auto &x : v) tiles.push_back(x.second);
    };
    append(0, syn);
    append(1, ffts);
    append(2, ffts);
    append(3, ana);
    b->fft_smem = smem;
    if (sht::batch_fft_prepare(smem) != cudaSuccess) {
        free_batch(b);
        return bfail(SHT_ECUDA, "setting the FFT kernel's shared-memory size failed");
    }
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
    b->ctas_legendre_syn = sms * 8;   // 128-thread CTAs
    b->ctas_legendre_ana = sms * 4;   // 128-thread CTAs of independent warps
    b->ctas_fft = sms * std::max(1, (int)std::min<size_t>(8, (200 * 1024) / std::max<size_t>(smem, 1)));
    cudaError_t e = cudaSuccess;
    for (int dir = 0; dir < 2; ++dir) {
        if (e == cudaSuccess) e = b->alloc(b->stage[dir]);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->used[dir], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) e = cudaMalloc(&b->d_fields, sizeof(sht::BatchField) * nfields);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_tiles, sizeof(int4) * tiles.size());
    if (e == cudaSuccess) e = cudaMalloc(&b->d_counters, 4 * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&b->d_inter, sizeof(float) * std::max<size_t>(inter, 64));
    if (e == cudaSuccess) e = cudaMemcpy(b->d_tiles, tiles.data(), sizeof(int4) * tiles.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_up, b->up_bytes());
    if (e == cudaSuccess && tc_ok) e = cudaMalloc(&b->d_gspec, sizeof(float) * std::max<size_t>(gspec, 64));
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->done, cudaEventDisableTiming);
    if (e != cudaSuccess) {
        free_batch(b);
        return bfail(SHT_ENOMEM, std::string("allocating the batch plan: ") + cudaGetErrorString(e));
    }
    b->mode = mode == SHT_TC_BF16X3 ? SHT_TC_BF16X3 : SHT_F32;
    if (mode == SHT_F32_AUTO && tc_ok) {
        const int rc = choose_mode(b);
        if (rc) {
            sht_batch_destroy(b);
            return rc;
        }
    }
    *out = b;
    return SHT_OK;
}

int sht_batch_mode(sht_batch b, float *ms_f32, float *ms_tc)
{
    if (!b) return bfail(SHT_EINVAL, "null batch handle");
    if (ms_f32) *ms_f32 = b->tuned_ms[0];
    if (ms_tc) *ms_tc = b->tuned_ms[1];
    return b->mode;
}

void sht_batch_destroy(sht_batch b)
{
    if (!b) return;
    cudaEventSynchronize(b->done);
    free_batch(b);
}

int sht_batch_synth(sht_batch b, void *const *spec, void *const *grid, int use_graph, void *stream)
{
    return run(b, true, spec, grid, use_graph, stream);
}

int sht_batch_analys(sht_batch b, void *const *grid, void *const *spec, int use_graph, void *stream)
{
    return run(b, false, grid, spec, use_graph, stream);
}

}  // extern "C"
