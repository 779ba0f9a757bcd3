// Native request executor (include/executor.h): arXiv 2608.07152 Sec. 2.1
// (ranked lists read page by page as a stable, only-extended prefix) over
// the PVS cursors of Sec. 2.3.
//
// A fixed pool of worker threads, each bound to the index's device with its
// own non-blocking stream.  A run publishes one job; the workers take request
// indexes from it.  For a request a worker opens the cursor on its own stream, reads the pages one
// after another through pvs_next straight into the request's rows of the
// caller's buffers, and closes the cursor.  With a group size G >= 2 a
// worker takes G requests at a time: one grouped open (one pass over the
// codes for all G queries, pvs_cursor_open_group), then every page of the G
// cursors in one batched pull.  A run of more requests than two groups, over a
// corpus of some size, takes blocks of requests instead (batch_block):
// their cursors come from one tensor-core pass (cursor_open_serving) and all
// their pages from one deep batched pull.  Requests that the block does not
// serve (a working set past the pass's capacity, a cursor's error) follow in
// groups, on whichever workers have no block.  No lock is held across a device
// wait; the job lock is taken only at the start and end of a run.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <condition_variable>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

#include "../../include/executor.h"
#include "runtime.h"

namespace {

constexpr int32_t kMaxWorkers = 64;

struct Job {
    const pvs_snapshot* snap = nullptr;
    const float* queries = nullptr;
    int32_t nq = 0, ranks = 0, page = 0;
    int32_t on_device = 0;              // queries, ids and scores in device memory
    int64_t* ids = nullptr;
    float* scores = nullptr;
    int32_t* n_out = nullptr;
    int32_t* status = nullptr;
    int32_t block = 0;                  // requests per batched open (0: groups of ex->group)
};

}  // namespace

struct pvs_executor {
    pvs_index* index = nullptr;
    std::vector<std::thread> threads;
    std::vector<cudaStream_t> streams;
    std::mutex m;                       // guards what follows, up to stop
    std::condition_variable work_cv, done_cv;
    Job job;
    int32_t next = 0;                   // next request index to hand out
    int32_t open = 0;                   // requests of the job not yet served
    // a run in blocks: the requests that finished blocks left, served in groups
    // by whichever worker is free
    std::vector<int32_t> left;
    int32_t left_groups = 0;            // groups of them being served
    bool stop = false;
    std::mutex run_mutex;               // one run at a time
    int32_t group = 1;                  // requests per grouped open
    std::atomic<int64_t> requests{0}, failed{0}, pages{0}, ranks{0};
    std::atomic<int64_t> passes{0}, refined{0};
    std::mutex ms_mutex;
    double interval_ms = 0.0;           // device time of the passes over the codes
};

namespace {

// Ranks [from, ranks) of request i's row: -1 / NaN (device rows: all bits
// set, which is -1 as an int64 and a NaN as a float32).
void fill_rest(const Job& j, cudaStream_t st, int32_t i, int32_t from) {
    if (from >= j.ranks) return;
    int64_t* ids = j.ids + (size_t)i * j.ranks;
    float* sc = j.scores + (size_t)i * j.ranks;
    if (j.on_device) {
        cudaMemsetAsync(ids + from, 0xff, (size_t)(j.ranks - from) * sizeof(int64_t), st);
        cudaMemsetAsync(sc + from, 0xff, (size_t)(j.ranks - from) * sizeof(float), st);
        return;
    }
    for (int32_t k = from; k < j.ranks; ++k) {
        ids[k] = -1;
        sc[k] = NAN;
    }
}

void count_request(pvs_executor* ex, pvs_status s, int64_t pages, int32_t total) {
    ex->requests.fetch_add(1, std::memory_order_relaxed);
    if (s < 0) ex->failed.fetch_add(1, std::memory_order_relaxed);
    ex->pages.fetch_add(pages, std::memory_order_relaxed);
    ex->ranks.fetch_add(total, std::memory_order_relaxed);
}

// The pass counters of a closed group: the interval time of its cursors'
// passes (a grouped pass is counted once) and their exact evaluations.
void count_passes(pvs_executor* ex, pvs_cursor* const* cs, int n, bool grouped) {
    double ms = 0.0;
    int64_t passes = 0, refined = 0;
    for (int i = 0; i < n; ++i) {
        pvs_stats st;
        if (pvs_cursor_stats(cs[i], &st) != PVS_OK) continue;
        refined += st.refined;
        if (!grouped || i == 0) {
            ms += st.interval_ms;
            passes += st.interval_passes;
        }
    }
    ex->passes.fetch_add(passes, std::memory_order_relaxed);
    ex->refined.fetch_add(refined, std::memory_order_relaxed);
    std::lock_guard<std::mutex> lk(ex->ms_mutex);
    ex->interval_ms += ms;
}

// One request on its own cursor: open, read the pages, close.  Returns the
// request's status.
pvs_status serve_one(pvs_executor* ex, const Job& j, cudaStream_t st, int32_t i,
                     pvs_cursor* c, int32_t total) {
    int64_t* ids = j.ids + (size_t)i * j.ranks;
    float* sc = j.scores + (size_t)i * j.ranks;
    int64_t pages = 0;
    pvs_status s = PVS_OK;
    const bool own = c == nullptr;   // a cursor handed over was counted with its group
    if (!c) {
        const int32_t dim = ex->index->m;
        s = pvs::cursor_open_on(ex->index, j.snap, j.queries + (size_t)i * dim, j.on_device, st,
                                &c);
    }
    if (s == PVS_OK && c) {
        while (total < j.ranks) {
            int32_t got = 0;
            const int32_t n = std::min(j.page, j.ranks - total);
            s = j.on_device ? pvs_next_device(c, n, ids + total, sc + total, &got)
                            : pvs_next(c, n, ids + total, sc + total, &got);
            ++pages;
            if (s < 0) break;
            total += got;
            if (s == PVS_EXHAUSTED || got < n) break;
        }
        if (s >= 0 && j.on_device) s = pvs_cursor_sync(c);   // device work done, status read
    }
    if (c) {
        if (own) count_passes(ex, &c, 1, false);
        pvs_cursor_close(c);
    }
    fill_rest(j, st, i, total);
    if (j.on_device) cudaStreamSynchronize(st);
    j.n_out[i] = total;
    count_request(ex, s < 0 ? s : PVS_OK, pages, total);
    return s == PVS_EXHAUSTED ? PVS_EXHAUSTED : (s < 0 ? s : PVS_OK);
}

// Requests req[0 .. count) (2 <= count <= PVS_GROUP_MAX) from one
// grouped open; `step` ranks of every cursor in one batched pull.  A failed
// open (a bad query) serves the group's requests one by one instead; a
// failure of the batched pull leaves the failed cursors' requests with
// their error and the others continuing one by one.  A request whose pull of more
// than a page failed is read again page by page: the ranks before its error stand.
void serve_group(pvs_executor* ex, const Job& j, cudaStream_t st, const int32_t* req, int32_t count,
                 int32_t step) {
    const float* queries[PVS_GROUP_MAX];
    for (int32_t i = 0; i < count; ++i) queries[i] = j.queries + (size_t)req[i] * ex->index->m;
    pvs_cursor* cs[PVS_GROUP_MAX] = {nullptr};
    pvs_status s = pvs::cursor_open_group(ex->index, j.snap, queries, count, j.on_device, st,
                                          nullptr, cs);
    if (s != PVS_OK) {   // e.g. one non-finite query: the others go on alone
        for (int32_t i = 0; i < count; ++i)
            j.status[req[i]] = serve_one(ex, j, st, req[i], nullptr, 0);
        return;
    }
    if (step >= j.ranks)   // (nor here)
        for (int32_t i = 0; i < count; ++i) cs[i]->readahead = 1;
    int32_t got[PVS_GROUP_MAX] = {0};
    int32_t n_out[PVS_GROUP_MAX] = {0};
    int64_t* id_rows[PVS_GROUP_MAX];
    float* sc_rows[PVS_GROUP_MAX];
    int64_t pages = 0;
    int32_t total = 0;
    bool batch_ok = true;
    while (total < j.ranks) {
        const int32_t n = std::min(step, j.ranks - total);
        for (int32_t i = 0; i < count; ++i) {
            id_rows[i] = j.ids + (size_t)req[i] * j.ranks + got[i];
            sc_rows[i] = j.scores + (size_t)req[i] * j.ranks + got[i];
        }
        s = pvs::next_batch_rows(cs, count, n, j.on_device, id_rows, sc_rows, n_out);
        pages += (n + j.page - 1) / j.page;
        if (s < 0) {
            batch_ok = false;
            break;
        }
        bool more = false;
        for (int32_t i = 0; i < count; ++i) {
            got[i] += n_out[i];
            more = more || n_out[i] == n;
        }
        total += n;
        if (!more) break;
    }
    const bool again = step > j.page;
    int states[PVS_GROUP_MAX] = {0};
    if (batch_ok && pvs_cursor_sync_batch(cs, count, states) != PVS_OK)
        for (int32_t i = 0; i < count; ++i) states[i] = PVS_ERR_CUDA;
    count_passes(ex, cs, count, true);
    for (int32_t i = 0; i < count; ++i) {
        const int32_t r = req[i];
        if (!batch_ok) {
            pvs_stats st_i;
            const bool failed = pvs_cursor_stats(cs[i], &st_i) != PVS_OK || st_i.state < 0;
            if (failed && again) {
                pvs_cursor_close(cs[i]);
                j.status[r] = serve_one(ex, j, st, r, nullptr, 0);
            } else if (failed) {
                fill_rest(j, st, r, got[i]);
                j.n_out[r] = got[i];
                j.status[r] = st_i.state < 0 ? (pvs_status)st_i.state : s;
                count_request(ex, (pvs_status)j.status[r], pages, got[i]);
                pvs_cursor_close(cs[i]);
            } else {   // continue this request on its own
                j.status[r] = serve_one(ex, j, st, r, cs[i], got[i]);
            }
            continue;
        }
        if (states[i] < 0 && again) {
            pvs_cursor_close(cs[i]);
            j.status[r] = serve_one(ex, j, st, r, nullptr, 0);
            continue;
        }
        fill_rest(j, st, r, got[i]);
        j.n_out[r] = got[i];
        j.status[r] = states[i] < 0 ? (pvs_status)states[i]
                                    : (got[i] < j.ranks ? PVS_EXHAUSTED : PVS_OK);
        count_request(ex, (pvs_status)j.status[r], pages, got[i]);
        pvs_cursor_close(cs[i]);
    }
    if (j.on_device) cudaStreamSynchronize(st);
}

// Requests per batched open for a run, or 0 to serve in groups.  A group of 8
// costs one read of the codes and their bounds written out (8.8M x 768: 1.24
// ms); a batched pass of up to 128 requests reads the codes once and keeps
// only working sets (1.1 ms + 0.2 ms for its thresholds), so it wins from the
// second group on; a run of one or two groups keeps the passes that its group
// size promises (their count is part of the statistics' contract).  Small
// corpora, where a pass takes microseconds, and requests deeper than one
// batched pull stay in groups.
constexpr int64_t kBlockRows = 65536;

// Groups of left-over requests served at once, over all workers: their cursors
// hold some 45 bytes a row each.  All of a block's at once held 100 cursors'
// row state (4.3 GB for 100 requests over 1M near-duplicates of 128 dimensions,
// 46 GB at 8.8M rows).  1, 2, 4 and 8 groups: 223, 159, 124 and 112 ms a run there
// (110 with all at once), first runs 227, 165, 139 and 167; 100 requests for 250
// ranks over 2M x 640 unit normals, half of them left over: 20.7, 17.3, 16.0 and
// 14.3 ms (16.0), first runs 22, 22, 25 and 32 (21: a group's cursors are
// allocated while other groups run).
constexpr int32_t kLeftGroups = 4;

int32_t batch_block(const pvs_executor* ex, const Job& j) {
    const pvs_index* x = ex->index;
    const int64_t rows = j.snap ? j.snap->data->rows : x->size;
    if (ex->group < 2 || j.nq <= 2 * ex->group || j.ranks > pvs::kPullBatchMax || rows < kBlockRows ||
        !pvs::batch_stream_supported(x->m_pad, x->num_sms))
        return 0;
    const int32_t most = pvs::batch_stream_queries(x->m_pad);
    const int32_t blocks = (j.nq + most - 1) / most;
    return (j.nq + blocks - 1) / blocks;   // equal shares
}

// Device rows of a block's host outputs, freed in stream order.
struct BlockOut {
    cudaStream_t st = nullptr;
    int64_t* ids = nullptr;
    float* scores = nullptr;
    cudaError_t get(const pvs_index* x, size_t ranks, cudaStream_t stream) {
        st = stream;
        const cudaError_t e = pvs::pool_alloc(&ids, ranks, x->scratch_pool, st);
        return e == cudaSuccess ? pvs::pool_alloc(&scores, ranks, x->scratch_pool, st) : e;
    }
    ~BlockOut() {
        if (ids) cudaFreeAsync(ids, st);
        if (scores) cudaFreeAsync(scores, st);
    }
};

// Requests first .. first+count-1 from one batched open and one pull of all
// their ranks.  `left` receives the requests that are still to be served (a query
// refused, a working set past the pass's capacity, a cursor's error; all of them
// when the open or the pull failed), each of which then gets its own status.
void serve_block(pvs_executor* ex, const Job& j, cudaStream_t st, int32_t first, int32_t count,
                 std::vector<int32_t>& left) {
    const pvs_index* x = ex->index;
    left.clear();
    std::vector<pvs_cursor*> opened((size_t)count, nullptr), cs;
    std::vector<pvs_status> each((size_t)count, PVS_OK);
    double pass_ms = 0.0;
    if (pvs::cursor_open_serving(ex->index, j.snap, j.queries + (size_t)first * x->m, count,
                                 j.on_device, j.ranks, st, opened.data(), each.data(),
                                 &pass_ms) != PVS_OK) {
        for (int32_t i = 0; i < count; ++i) left.push_back(first + i);
        return;
    }
    std::vector<int32_t> req, refused;   // the requests of cs, and of refused queries
    for (int32_t i = 0; i < count; ++i) {
        if (opened[(size_t)i]) {
            // one pull reads all: no ranks ahead, and no buffers for them (a new
            // index's first block of 128 requests for 20 ranks took 0.4 ms for these)
            opened[(size_t)i]->readahead = 1;
            cs.push_back(opened[(size_t)i]);
            req.push_back(first + i);
        } else if (each[(size_t)i] != PVS_OK) {   // (on its own: not to fail a group's open)
            refused.push_back(first + i);
        } else {
            left.push_back(first + i);
        }
    }
    const int32_t held = (int32_t)cs.size();
    const size_t at = (size_t)first * j.ranks, total = (size_t)count * j.ranks;
    BlockOut buf;
    bool ok = j.on_device || buf.get(x, total, st) == cudaSuccess;
    std::vector<int32_t> n_out((size_t)held, 0);
    if (ok) {
        std::vector<int64_t*> id_rows((size_t)held);
        std::vector<float*> sc_rows((size_t)held);
        for (int32_t i = 0; i < held; ++i) {
            const size_t row = (size_t)(req[(size_t)i] - first) * j.ranks;
            id_rows[(size_t)i] = (j.on_device ? j.ids + at : buf.ids) + row;
            sc_rows[(size_t)i] = (j.on_device ? j.scores + at : buf.scores) + row;
        }
        ok = pvs::next_batch_rows(cs.data(), held, j.ranks, 1, id_rows.data(), sc_rows.data(),
                                  n_out.data()) >= 0;
    }
    if (ok && !j.on_device)   // the block's rows are consecutive on both sides
        ok = pvs::taken(cudaMemcpyAsync(j.ids + at, buf.ids, total * sizeof(int64_t),
                                        cudaMemcpyDeviceToHost, st)) == cudaSuccess &&
             pvs::taken(cudaMemcpyAsync(j.scores + at, buf.scores, total * sizeof(float),
                                        cudaMemcpyDeviceToHost, st)) == cudaSuccess;
    std::vector<pvs_stats> stats((size_t)held);
    if (ok) ok = pvs_cursor_stats_batch(cs.data(), held, stats.data()) == PVS_OK;   // (waits)
    int64_t passes = 1, refined = 0;
    for (int32_t i = 0; i < held; ++i) {
        const int32_t r = req[(size_t)i], got = n_out[(size_t)i];
        if (!ok || stats[(size_t)i].state < 0) {
            left.push_back(r);
            continue;
        }
        const pvs_stats& c = stats[(size_t)i];
        refined += c.refined;
        passes += c.interval_passes;   // (none: the working sets hold every rank)
        pass_ms += c.interval_ms;
        fill_rest(j, st, r, got);
        j.n_out[r] = got;
        j.status[r] = got < j.ranks ? PVS_EXHAUSTED : PVS_OK;
        count_request(ex, PVS_OK, std::max(1, (got + j.page - 1) / j.page), got);
    }
    ex->passes.fetch_add(passes, std::memory_order_relaxed);
    ex->refined.fetch_add(refined, std::memory_order_relaxed);
    {
        std::lock_guard<std::mutex> lk(ex->ms_mutex);
        ex->interval_ms += pass_ms;
    }
    pvs_cursor_close_batch(cs.data(), held);   // (waits for the stream)
    // after the block's copy of all its rows
    for (int32_t r : refused) j.status[r] = serve_one(ex, j, st, r, nullptr, 0);
}

// A worker takes the job's next block or group, or a group of what finished
// blocks left, and serves it.  The run is over with its last request, whether or
// not the workers that found nothing to do have woken up (waiting for them took
// 20 us of a run of one block).
void worker_main(pvs_executor* ex, int w) {
    cudaSetDevice(ex->index->device);
    const cudaStream_t st = ex->streams[(size_t)w];
    std::vector<int32_t> req;   // the requests taken
    std::unique_lock<std::mutex> lk(ex->m);
    for (;;) {
        const auto left_ready = [&] { return !ex->left.empty() && ex->left_groups < kLeftGroups; };
        ex->work_cv.wait(lk, [&] { return ex->stop || ex->next < ex->job.nq || left_ready(); });
        if (ex->stop) return;
        const Job j = ex->job;
        const int32_t G = ex->group;
        const bool left = ex->next >= j.nq;
        const int32_t first = ex->next;
        int32_t count;
        if (left) {
            count = (int32_t)std::min<size_t>((size_t)G, ex->left.size());
            req.assign(ex->left.end() - count, ex->left.end());
            ex->left.resize(ex->left.size() - (size_t)count);
            ++ex->left_groups;
        } else {
            count = std::min(j.block ? j.block : G, j.nq - first);
            ex->next += count;
            req.resize((size_t)count);
            for (int32_t k = 0; k < count; ++k) req[(size_t)k] = first + k;
        }
        lk.unlock();
        if (!left && j.block && count > G) {
            serve_block(ex, j, st, first, count, req);   // req: what it leaves
        } else {
            // (a block's requests are at most one batched pull deep)
            if (count == 1)
                j.status[req[0]] = serve_one(ex, j, st, req[0], nullptr, 0);
            else
                serve_group(ex, j, st, req.data(), count, left ? j.ranks : j.page);
            req.clear();
        }
        lk.lock();
        if (left) --ex->left_groups;
        ex->open -= count - (int32_t)req.size();
        if (!req.empty()) {
            ex->left.insert(ex->left.end(), req.begin(), req.end());
            ex->work_cv.notify_all();
        }
        if (ex->open == 0) ex->done_cv.notify_all();
    }
}

void shutdown(pvs_executor* ex) {
    {
        std::lock_guard<std::mutex> lk(ex->m);
        ex->stop = true;
    }
    ex->work_cv.notify_all();
    for (auto& t : ex->threads)
        if (t.joinable()) t.join();
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(ex->index->device);
    for (cudaStream_t s : ex->streams) cudaStreamDestroy(s);
    if (prev >= 0) cudaSetDevice(prev);
}

}  // namespace

extern "C" {

pvs_status pvs_executor_create(pvs_index* index, int32_t workers, pvs_executor** out) {
    if (!out) return PVS_ERR_INVALID;
    *out = nullptr;
    if (!index || workers < 1 || workers > kMaxWorkers) return PVS_ERR_INVALID;
    pvs_executor* ex = new (std::nothrow) pvs_executor();
    if (!ex) return PVS_ERR_OOM;
    ex->index = index;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaError_t e = cudaSetDevice(index->device);
    for (int32_t w = 0; w < workers && e == cudaSuccess; ++w) {
        cudaStream_t s = nullptr;
        e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
        if (e == cudaSuccess) ex->streams.push_back(s);
    }
    if (prev >= 0) cudaSetDevice(prev);
    if (e != cudaSuccess) {
        cudaGetLastError();
        shutdown(ex);
        delete ex;
        return PVS_ERR_CUDA;
    }
    try {
        for (int32_t w = 0; w < workers; ++w) ex->threads.emplace_back(worker_main, ex, (int)w);
    } catch (...) {
        shutdown(ex);
        delete ex;
        return PVS_ERR_OOM;
    }
    *out = ex;
    return PVS_OK;
}

pvs_status pvs_executor_set_group(pvs_executor* ex, int32_t group) {
    if (!ex || group < 1 || group > PVS_GROUP_MAX) return PVS_ERR_INVALID;
    std::lock_guard<std::mutex> run(ex->run_mutex);   // not during a run
    ex->group = group;
    return PVS_OK;
}

pvs_status pvs_executor_run(pvs_executor* ex, const pvs_snapshot* snap, const float* queries,
                            int32_t nq, int32_t ranks, int32_t page, int64_t* ids, float* scores,
                            int32_t* n_out, int32_t* status) {
    return pvs_executor_run_ex(ex, snap, queries, nq, ranks, page, 0, ids, scores, n_out, status);
}

pvs_status pvs_executor_run_ex(pvs_executor* ex, const pvs_snapshot* snap, const float* queries,
                               int32_t nq, int32_t ranks, int32_t page, int32_t buffers_on_device,
                               int64_t* ids, float* scores, int32_t* n_out, int32_t* status) {
    if (!ex || nq < 0 || ranks < 1 || page < 1 || page > ranks) return PVS_ERR_INVALID;
    if (snap && snap->index != ex->index) return PVS_ERR_INVALID;
    if (nq == 0) return PVS_OK;
    if (!queries || !ids || !scores || !n_out) return PVS_ERR_INVALID;
    std::vector<int32_t> own;
    if (!status) {
        own.assign((size_t)nq, 0);
        status = own.data();
    }
    std::lock_guard<std::mutex> run(ex->run_mutex);
    {
        std::lock_guard<std::mutex> lk(ex->m);
        ex->job = Job{snap, queries, nq, ranks, page, buffers_on_device ? 1 : 0, ids, scores,
                      n_out, status, 0};
        ex->job.block = batch_block(ex, ex->job);
        ex->next = 0;
        ex->open = nq;
    }
    ex->work_cv.notify_all();
    {
        std::unique_lock<std::mutex> lk(ex->m);
        ex->done_cv.wait(lk, [&] { return ex->open == 0; });
    }
    for (int32_t i = 0; i < nq; ++i)
        if (status[i] < 0) return (pvs_status)status[i];
    return PVS_OK;
}

pvs_status pvs_executor_stats_get(pvs_executor* ex, pvs_executor_stats* out) {
    if (!ex || !out) return PVS_ERR_INVALID;
    out->requests = ex->requests.load();
    out->failed = ex->failed.load();
    out->pages = ex->pages.load();
    out->ranks = ex->ranks.load();
    out->workers = (int32_t)ex->threads.size();
    out->group = ex->group;
    out->interval_passes = ex->passes.load();
    out->refined = ex->refined.load();
    {
        std::lock_guard<std::mutex> lk(ex->ms_mutex);
        out->interval_ms = ex->interval_ms;
    }
    return PVS_OK;
}

void pvs_executor_destroy(pvs_executor* ex) {
    if (!ex) return;
    {
        std::lock_guard<std::mutex> run(ex->run_mutex);   // after a run in progress
    }
    shutdown(ex);
    delete ex;
}

}  // extern "C"
