// Continuous-batching server (not in the paper): requests of any size, each
// with its own k / itopk / entry, are admitted while others run and share the
// GPU query by query.
//
// Ring of `capacity` query slots (query vector, kmax results) and ring of
// request records in page-locked host memory that the device reads and writes
// directly; learned-entry seeds, the counts of queries taken and available and the
// per-request counts of queries finished in device memory. Host state: the requests in
// flight, in slot order.
//
// submit(): admission checks ring space and request records (ANN_EBUSY when
// either is short: admission by buffer memory). The queries, the record and the
// slot->request map are written into the rings and one serve kernel is launched,
// on one of several compute streams: a launch makes the host's earlier writes
// visible, so no copy, event or second stream is needed. Only the learned
// entry's prediction needs the queries on the device: a copy and the prediction
// on an ingest stream, which the launches then wait for. Kernels of successive
// requests overlap and take queries from the same FIFO; each launch has room for
// every query in flight, its own request's included, and its warps leave early
// only when all that is published has been taken (serve_take.cuh), so every
// published query is served. A request counts as published once its launch was
// accepted. Measured: 200 requests of 1-64 queries at once 19.5 -> 4.5 ms (2.7 of
// which the host spends submitting them), one request of 6,548 queries 5.1 ->
// 2.1, of 608 3.5 -> 0.76.
//
// poll(): a request is done when its flag is set (by the warp that finished its
// last query, after a system-scope fence); its results are copied out of the
// ring and its space is reclaimed in slot order. Latency is submit ->
// poll-observed completion on the host's steady clock.
#include <chrono>
#include <cstring>
#include <deque>
#include <vector>

#include "ann_internal.cuh"

using namespace ann;

namespace {

double now_s()
{
    return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

struct Pending {
    uint64_t req_id;
    uint32_t ri;
    uint64_t start;    // first query counter
    uint32_t nq, k;
    uint32_t *ids_out;
    float *dists_out;
    double t_submit;
    bool done;
};

}  // namespace

struct ann_server {
    ann_index *ix = nullptr;
    ann_mlp *mlp = nullptr;
    uint32_t P = 0;
    float tau = 0.0f;
    uint32_t cap = 0, nreq = 0, kmax = 0, per_warp = 0;
    ann_search_params maxp{};
    void *plan = nullptr;
    float *d_queries = nullptr;                // learned entry: the network's input
    uint32_t *d_seeds = nullptr;
    unsigned long long *d_counters = nullptr;
    uint32_t *d_done = nullptr;
    // page-locked, mapped: one allocation, as the host and the device see it
    uint8_t *h_ring = nullptr, *d_ring = nullptr;
    size_t o_queries = 0, o_ids = 0, o_dists = 0, o_slot_req = 0, o_reqs = 0, o_flags = 0, o_tail = 0;
    cudaStream_t ingest = nullptr;             // learned entry only
    std::vector<cudaStream_t> compute;
    std::vector<cudaEvent_t> ev;
    uint32_t next_stream = 0;
    uint64_t tail = 0, seq = 0;
    std::deque<Pending> inflight;
    std::deque<ann_completion> ready;

    template <typename T> T *host(size_t o) const { return reinterpret_cast<T *>(h_ring + o); }
    template <typename T> T *dev(size_t o) const { return reinterpret_cast<T *>(d_ring + o); }
};

namespace {

void server_release(ann_server *s)
{
    if (s->ingest) cudaStreamSynchronize(s->ingest);
    for (cudaStream_t c : s->compute) cudaStreamSynchronize(c);
    void *dev[] = {s->d_queries, s->d_seeds, s->d_counters, s->d_done};
    for (void *p : dev) if (p) cudaFree(p);
    if (s->h_ring) cudaFreeHost(s->h_ring);
    for (cudaEvent_t e : s->ev) cudaEventDestroy(e);
    for (cudaStream_t c : s->compute) cudaStreamDestroy(c);
    if (s->ingest) cudaStreamDestroy(s->ingest);
    if (s->plan) serve_plan_free(s->plan);
}

// Copy `n` consecutive ring rows starting at counter `start` (wrapping) of
// width `w` elements (pitch kmax) into dst rows of width w.
template <typename T>
void copy_out(T *dst, const T *ring, uint64_t start, uint32_t n, uint32_t w, uint32_t pitch, uint32_t cap)
{
    for (uint32_t i = 0; i < n; ++i)
        memcpy(dst + (size_t)i * w, ring + ((start + i) % cap) * (size_t)pitch, (size_t)w * sizeof(T));
}

}  // namespace

extern "C" {

ann_status ann_server_create(ann_index *ix, const ann_server_config *cfg, ann_mlp *mlp, ann_server **out)
{
    if (!ix || !cfg || !out) { set_error("ann_server_create: NULL argument"); return ANN_EINVAL; }
    *out = nullptr;
    if (cfg->capacity == 0 || cfg->max_requests == 0) {
        set_error("ann_server_create: capacity and max_requests must be positive");
        return ANN_EINVAL;
    }
    const ann_search_params &mp = cfg->max_params;
    if (mp.entry > ANN_ENTRY_GIVEN_GHOST) {
        set_error("ann_server_create: entry %u is not served (given base seeds need ann_search)", mp.entry);
        return ANN_EINVAL;
    }
    if (mp.entry == ANN_ENTRY_GIVEN_GHOST && (!mlp || cfg->seeds_per_query == 0 || cfg->seeds_per_query > 8)) {
        set_error("ann_server_create: the learned entry needs an MLP and 1..8 seeds per query");
        return ANN_EINVAL;
    }
    int prev = -1;
    {
        const ann_status ds = enter_device(ix->device, &prev, "ann_server_create");
        if (ds != ANN_OK) return ds;
    }
    ann_server *s = new ann_server();
    s->ix = ix;
    s->mlp = mlp;
    s->P = mp.entry == ANN_ENTRY_GIVEN_GHOST ? cfg->seeds_per_query : 0;
    s->tau = cfg->tau;
    s->cap = cfg->capacity;
    s->nreq = cfg->max_requests;
    s->kmax = mp.k;
    s->per_warp = cfg->queries_per_warp;
    s->maxp = mp;
    const uint32_t ns = cfg->streams ? cfg->streams : 4;
    ann_status st = serve_plan(ix, &mp, s->P ? s->P : 1, ns, &s->plan);
    cudaError_t e = cudaSuccess;
    auto al = [&](void **p, size_t bytes) { if (e == cudaSuccess) e = cudaMalloc(p, bytes); };
    if (st == ANN_OK) {
        if (s->P) al((void **)&s->d_queries, (size_t)s->cap * ix->dim * 4);
        if (s->P) al((void **)&s->d_seeds, (size_t)s->cap * s->P * 4);
        al((void **)&s->d_counters, 64);
        al((void **)&s->d_done, (size_t)s->nreq * 4);
        if (e == cudaSuccess) e = cudaMemset(s->d_counters, 0, 64);
        if (e == cudaSuccess) e = cudaMemset(s->d_done, 0, (size_t)s->nreq * 4);
        size_t bytes = 0;
        auto take = [&](size_t b) {
            const size_t at = bytes;
            bytes += (b + 255) & ~(size_t)255;
            return at;
        };
        s->o_queries = take((size_t)s->cap * ix->dim * 4);
        s->o_ids = take((size_t)s->cap * s->kmax * 4);
        s->o_dists = take((size_t)s->cap * s->kmax * 4);
        s->o_slot_req = take((size_t)s->cap * 4);
        s->o_reqs = take((size_t)s->nreq * sizeof(ServeReq));
        s->o_flags = take((size_t)s->nreq * 4);
        s->o_tail = take(8);
        if (e == cudaSuccess) e = cudaHostAlloc((void **)&s->h_ring, bytes, cudaHostAllocMapped);
        if (e == cudaSuccess) e = cudaHostGetDevicePointer((void **)&s->d_ring, s->h_ring, 0);
        int lo = 0, hi = 0;
        if (e == cudaSuccess) e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
        if (e == cudaSuccess && s->P) e = cudaStreamCreateWithPriority(&s->ingest, cudaStreamNonBlocking, hi);
        for (uint32_t i = 0; i < ns && e == cudaSuccess; ++i) {
            cudaStream_t c;
            e = cudaStreamCreateWithPriority(&c, cudaStreamNonBlocking, lo);
            if (e == cudaSuccess) s->compute.push_back(c);
        }
        for (uint32_t i = 0; i < (s->P ? s->nreq : 0u) && e == cudaSuccess; ++i) {
            cudaEvent_t ev;
            e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
            if (e == cudaSuccess) s->ev.push_back(ev);
        }
        if (e != cudaSuccess) st = cuda_fail(e, "ann_server_create");
        else {
            memset(s->host<uint32_t>(s->o_flags), 0, (size_t)s->nreq * 4);
            *s->host<uint64_t>(s->o_tail) = 0;
        }
    }
    leave_device(ix->device, prev);
    if (st != ANN_OK) {
        server_release(s);
        delete s;
        return st;
    }
    *out = s;
    return ANN_OK;
}

ann_status ann_server_submit(ann_server *s, uint64_t req_id, const float *queries, uint32_t nq,
                             const ann_search_params *p, uint32_t *ids, float *dists)
{
    if (!s || !p || (nq && (!queries || !ids || !dists))) { set_error("ann_server_submit: NULL argument"); return ANN_EINVAL; }
    if (nq == 0) { set_error("ann_server_submit: empty request"); return ANN_EINVAL; }
    const ann_search_params &mp = s->maxp;
    if (p->k > mp.k || p->itopk > mp.itopk || p->search_width > mp.search_width ||
        (p->ghost_search_width ? p->ghost_search_width : 1) > (mp.ghost_search_width ? mp.ghost_search_width : 1) ||
        ((p->dgs_discard > 0.0f || p->dgs_min_match > 0.0f) &&
         !(mp.dgs_discard > 0.0f || mp.dgs_min_match > 0.0f)) ||
        (p->rerank && !mp.rerank) || p->entry > ANN_ENTRY_GIVEN_GHOST ||
        (p->entry != ANN_ENTRY_RANDOM && mp.entry == ANN_ENTRY_RANDOM) ||
        (p->entry == ANN_ENTRY_GIVEN_GHOST && !s->P) ||
        (p->entry != ANN_ENTRY_RANDOM && (p->ghost_itopk ? p->ghost_itopk : std::min(p->itopk, 64u)) >
                                             (mp.ghost_itopk ? mp.ghost_itopk : std::min(mp.itopk, 64u)))) {
        set_error("ann_server_submit: parameters exceed the server's max_params");
        return ANN_EINVAL;
    }
    if (nq > s->cap) { set_error("ann_server_submit: %u queries exceed the ring capacity %u", nq, s->cap); return ANN_EINVAL; }
    QParams q;
    ann_status st = derive_qparams(s->ix, p, p->entry == ANN_ENTRY_GIVEN_GHOST ? s->P : 0, &q);
    if (st != ANN_OK) return st;
    const uint64_t oldest = s->inflight.empty() ? s->tail : s->inflight.front().start;
    if (s->inflight.size() >= s->nreq || s->tail + nq - oldest > s->cap) {
        set_error("ann_server_submit: no room (ring or request records full)");
        return ANN_EBUSY;
    }
    int prev = -1;
    {
        const ann_status ds = enter_device(s->ix->device, &prev, "ann_server_submit");
        if (ds != ANN_OK) return ds;
    }
    const uint32_t ri = (uint32_t)(s->seq % s->nreq);
    const uint32_t dim = s->ix->dim;
    const uint32_t slot0 = (uint32_t)(s->tail % s->cap);
    const uint32_t first = std::min<uint32_t>(nq, s->cap - slot0);
    s->host<volatile uint32_t>(s->o_flags)[ri] = 0;
    s->host<ServeReq>(s->o_reqs)[ri] = ServeReq{q, nq, slot0, ri};
    float *ring = s->host<float>(s->o_queries);
    memcpy(ring + (size_t)slot0 * dim, queries, (size_t)first * dim * 4);
    if (first < nq) memcpy(ring, queries + (size_t)first * dim, (size_t)(nq - first) * dim * 4);
    uint32_t *map = s->host<uint32_t>(s->o_slot_req);
    for (uint32_t i = 0; i < nq; ++i) map[slot0 + i < s->cap ? slot0 + i : slot0 + i - s->cap] = ri;
    cudaError_t e = cudaSuccess;
    if (p->entry == ANN_ENTRY_GIVEN_GHOST) {
        cudaStream_t in = s->ingest;
        e = cudaMemcpyAsync(s->d_queries + (size_t)slot0 * dim, ring + (size_t)slot0 * dim, (size_t)first * dim * 4,
                            cudaMemcpyHostToDevice, in);
        if (e == cudaSuccess && first < nq)
            e = cudaMemcpyAsync(s->d_queries, ring, (size_t)(nq - first) * dim * 4, cudaMemcpyHostToDevice, in);
        if (e == cudaSuccess)
            st = ann_mlp_predict(s->mlp, s->d_queries + (size_t)slot0 * dim, first, s->P, s->tau,
                                 s->d_seeds + (size_t)slot0 * s->P, nullptr, in);
        if (st == ANN_OK && e == cudaSuccess && first < nq)
            st = ann_mlp_predict(s->mlp, s->d_queries, nq - first, s->P, s->tau, s->d_seeds, nullptr, in);
    }
    // the launch may take queries of any request before it, so it waits for
    // every prediction so far (the ingest stream is in order)
    if (st == ANN_OK && e == cudaSuccess && s->P) e = cudaEventRecord(s->ev[ri], s->ingest);
    if (st == ANN_OK && e == cudaSuccess) {
        const uint32_t si = (uint32_t)(s->next_stream++ % s->compute.size());
        cudaStream_t c = s->compute[si];
        if (s->P) e = cudaStreamWaitEvent(c, s->ev[ri], 0);
        if (e == cudaSuccess) {
            ServeRing r{};
            r.queries = s->dev<float>(s->o_queries);
            r.seeds = s->d_seeds;
            r.P = s->P;
            r.ids = s->dev<uint32_t>(s->o_ids);
            r.dists = s->dev<float>(s->o_dists);
            r.slot_req = s->dev<uint32_t>(s->o_slot_req);
            r.reqs = s->dev<ServeReq>(s->o_reqs);
            r.done = s->d_done;
            r.counters = s->d_counters;
            r.tail = s->tail + nq;
            r.flags = s->dev<uint32_t>(s->o_flags);
            r.cap = s->cap;
            r.kmax = s->kmax;
            r.per_warp = s->per_warp;
            // On an idle stream the launch starts now: a warp for every query
            // not yet known complete, and no later ones. Behind another launch
            // it starts when that ends and takes what was published by then: a
            // warp for as many queries as can be resident. Warps leave as soon
            // as the launch's capacity covers the queries in flight, so a
            // stream is free again after one query's time. (With four queries
            // a warp and launches sized for that, a burst of 200 requests of
            // 1-64 queries went through the streams in five generations of four
            // small kernels: 15 to 19 ms, most of the GPU idle.) A server with
            // a network takes no later queries: their seeds may not be there
            // yet.
            const uint32_t pending = (uint32_t)(s->tail + nq - oldest);   // at most the ring's capacity
            uint32_t warps = pending;
            const cudaError_t busy = cudaStreamQuery(c);
            if (busy == cudaErrorNotReady && !s->P) {
                r.live = s->dev<unsigned long long>(s->o_tail);
                warps = s->cap;
            }
            if (busy == cudaErrorNotReady) cudaGetLastError();
            else e = busy;
            if (e == cudaSuccess) {
                st = serve_launch(s->plan, r, warps, pending, c, si);
                // only now: queued launches publish what they read here, and a
                // request whose launch was refused is not one of the server's
                if (st == ANN_OK) __atomic_store_n(s->host<uint64_t>(s->o_tail), s->tail + nq, __ATOMIC_RELEASE);
            }
        }
    }
    if (st == ANN_OK && e != cudaSuccess) st = cuda_fail(e, "ann_server_submit");
    if (st == ANN_OK) {
        s->inflight.push_back(Pending{req_id, ri, s->tail, nq, p->k, ids, dists, now_s(), false});
        s->tail += nq;
        s->seq++;
    }
    leave_device(s->ix->device, prev);
    return st;
}

ann_status ann_server_poll(ann_server *s, ann_completion *out, uint32_t max, uint32_t *n_out)
{
    if (!s || (max && !out) || !n_out) { set_error("ann_server_poll: NULL argument"); return ANN_EINVAL; }
    int prev = -1;
    {
        const ann_status ds = enter_device(s->ix->device, &prev, "ann_server_poll");
        if (ds != ANN_OK) return ds;
    }
    ann_status st = ANN_OK;
    for (Pending &pd : s->inflight) {
        // the acquire pairs with the device's fence: the results precede the flag
        if (pd.done || !__atomic_load_n(s->host<uint32_t>(s->o_flags) + pd.ri, __ATOMIC_ACQUIRE)) continue;
        copy_out(pd.ids_out, s->host<uint32_t>(s->o_ids), pd.start, pd.nq, pd.k, s->kmax, s->cap);
        copy_out(pd.dists_out, s->host<float>(s->o_dists), pd.start, pd.nq, pd.k, s->kmax, s->cap);
        pd.done = true;
        s->ready.push_back(ann_completion{pd.req_id, 0, pd.nq, now_s() - pd.t_submit});
    }
    while (!s->inflight.empty() && s->inflight.front().done) s->inflight.pop_front();
    uint32_t n = 0;
    while (n < max && !s->ready.empty()) {
        out[n++] = s->ready.front();
        s->ready.pop_front();
    }
    *n_out = n;
    leave_device(s->ix->device, prev);
    return st;
}

uint32_t ann_server_in_flight(const ann_server *s) { return s ? (uint32_t)s->inflight.size() : 0; }

ann_status ann_server_destroy(ann_server *s)
{
    if (!s) return ANN_OK;
    int prev = -1;
    const bool switched = enter_device(s->ix->device, &prev, "ann_server_destroy") == ANN_OK;   // frees best-effort
    server_release(s);
    if (switched) leave_device(s->ix->device, prev);
    delete s;
    return ANN_OK;
}

}  // extern "C"
