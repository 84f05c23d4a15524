// Serving: a continuous-batching request loop for mining jobs.
//
// Every job is a database in host CSR form plus an absolute minsup.  Jobs are
// admitted in arrival order as soon as a slot is free and their estimated
// device footprint fits the HBM budget left by the jobs in flight; each slot
// runs its job (bitmap build with the minsup as prefilter, sample estimate,
// mine) on its own CUDA stream, so the kernels of concurrent jobs overlap on
// the device.  Bitmaps of a job stay resident until its result is copied out.
// The submitter uploads its database itself while the budget has room for the job (fim_server_submit).
// The persistent DFS of a served job exits as soon as its queue drains (no
// idle polling), so concurrent jobs never hold SMs for one another.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <memory>
#include <mutex>
#include <new>
#include <system_error>
#include <thread>
#include <unordered_map>
#include <vector>

#include "fim_internal.cuh"

namespace {

using Clock = std::chrono::steady_clock;

// Threads that share the host's part of a submission (reading its offsets, copying it) with the submitter, a piece after the
// other.  The caller waits only for the threads that have taken a piece, not for those that are still waking up, and they
// look out for the next call for a moment before they sleep (submissions of a burst follow one another).
class Crew {
 public:
  explicit Crew(uint32_t helpers) {
    threads_.reserve(helpers);
    try {
      for (uint32_t k = 0; k < helpers; ++k) threads_.emplace_back([this] { help(); });
    } catch (const std::system_error&) {  // (fewer than asked for)
    }
  }
  ~Crew() {
    {
      std::lock_guard<std::mutex> lock(mu_);
      stop_ = true;
    }
    cv_open_.notify_all();
    for (auto& t : threads_) t.join();
  }
  // f(0) .. f(n - 1) (one caller at a time; f does not throw)
  template <typename F>
  void run(uint64_t n, const F& f) {
    if (n <= 2 || threads_.empty()) {
      for (uint64_t k = 0; k < n; ++k) f(k);
      return;
    }
    {
      std::lock_guard<std::mutex> lock(mu_);
      ctx_ = &f;
      call_ = [](const void* ctx, uint64_t k) { (*static_cast<const F*>(ctx))(k); };
      n_ = n;
      next_ = 0;
      open_ = true;
      ++turn_;
    }
    cv_open_.notify_all();
    pieces();
    std::unique_lock<std::mutex> lock(mu_);
    open_ = false;
    cv_idle_.wait(lock, [&] { return busy_ == 0; });
  }
  void copy(uint8_t* dst, const uint8_t* src, uint64_t bytes) {
    constexpr uint64_t kPiece = 128 << 10;
    run((bytes + kPiece - 1) / kPiece,
        [=](uint64_t k) { std::memcpy(dst + k * kPiece, src + k * kPiece, std::min(kPiece, bytes - k * kPiece)); });
  }

 private:
  static constexpr std::chrono::microseconds kLookOut{100};
  void pieces() {
    for (uint64_t k; (k = next_.fetch_add(1)) < n_;) call_(ctx_, k);
  }
  void help() {
    uint64_t seen = 0;
    std::unique_lock<std::mutex> lock(mu_);
    for (;;) {
      if (!stop_ && turn_ == seen) {
        lock.unlock();
        const auto until = Clock::now() + kLookOut;
        while (turn_.load() == seen && Clock::now() < until) std::this_thread::yield();
        lock.lock();
      }
      cv_open_.wait(lock, [&] { return stop_ || (open_ && turn_ != seen); });
      if (stop_) return;
      seen = turn_;
      ++busy_;
      lock.unlock();
      pieces();
      lock.lock();
      if (--busy_ == 0) cv_idle_.notify_one();
    }
  }
  std::mutex mu_;
  std::condition_variable cv_open_, cv_idle_;
  const void* ctx_ = nullptr;
  void (*call_)(const void*, uint64_t) = nullptr;
  uint64_t n_ = 0;
  std::atomic<uint64_t> next_{0}, turn_{0};
  uint32_t busy_ = 0;
  bool open_ = false, stop_ = false;
  std::vector<std::thread> threads_;
};

struct Job {
  uint64_t id = 0;
  std::vector<uint32_t> off, items;
  uint32_t D = 0, N = 0, minsup = 1;
  double sample_rate = 0.0;
  uint64_t footprint = 0;
  bool ready = false;      // the server has its copy of the database
  bool reserved = false;   // its footprint is part of in_use (from the submission when the submitter uploads)
  void* d_csr = nullptr;   // the uploaded database: offsets, then items (csr_items bytes further); csr_bytes in all
  uint64_t csr_items = 0, csr_bytes = 0, nnz = 0;
  cudaEvent_t ev_csr = nullptr;  // the upload's end
  Clock::time_point t_submit, t_start, t_end;
  cudaEvent_t ev_start = nullptr, ev_end = nullptr;  // the job's device work on its slot's stream
  fim_status status = FIM_OK;
  std::string error;
  fim_result* result = nullptr;
  bool done = false;
  bool taken = false;
};

}  // namespace

struct fim_server {
  std::mutex mu;
  std::condition_variable cv_work, cv_done;
  std::deque<Job*> queue;
  std::unordered_map<uint64_t, Job*> jobs;
  uint64_t next_id = 1;
  uint64_t budget = 0, in_use = 0;
  uint64_t uploaded = 0;  // bytes of the uploaded databases, at most 1/32 of the device memory
  uint32_t in_flight = 0, peak_in_flight = 0;
  bool stop = false;
  int device = 0;
  uint32_t ctas_per_sm = 1;
  uint64_t max_itemsets = 0;
  uint64_t total_mem = 0;
  std::vector<std::thread> workers;
  std::vector<cudaStream_t> streams;
  std::mutex up_mu;                // one upload at a time
  cudaStream_t up_stream = nullptr;
  std::unique_ptr<Crew> crew;  // (under up_mu)
  uint8_t* stage[2] = {};          // pinned, kStageBytes each: uploads go through them in turn
  cudaEvent_t stage_free[2] = {};  // the buffer's last copy is done
  uint32_t stage_turn = 0;
  cudaEvent_t ev_origin = nullptr;  // recorded at creation: device times of jobs are measured from it
};

namespace {

// Upper bound of the device bytes of one job: CSR copy, bitmaps of the items that
// can reach minsup (at most nnz / minsup of them), pair block, queue, DFS stack,
// output, with the sample of the estimate on top.
uint64_t job_footprint(uint32_t D, uint32_t N, uint64_t nnz, uint32_t max_len, uint32_t minsup, uint32_t grid,
                       uint64_t total_mem, int num_sms) {
  const uint64_t stride = ((uint64_t)(D + 31) / 32 + 31) / 32 * 32;
  const uint64_t rows = std::min<uint64_t>(N, nnz / std::max<uint32_t>(1, minsup) + 1);
  uint64_t b = 4ull * ((uint64_t)D + 1 + nnz);           // CSR
  b += 4ull * rows * stride;                              // bitmaps
  b += 4ull * rows * rows + 12ull * rows * rows / 2;      // pair counts, survivors, queue
  // rows widened to bytes when the engine would take the tensor-core pair kernel
  const uint64_t xb = fim::pair_mma_buffer_bytes((uint32_t)rows, (uint32_t)stride, true);
  if (rows >= 2 && xb <= total_mem / 16 &&
      fim::pair_mma_cost_us((uint32_t)rows, (uint32_t)stride, num_sms, true) <
          fim::pair_cores_cost_us((uint32_t)rows, (uint32_t)stride, num_sms))
    b += xb;
  // DFS stack: the full depth (itemsets are no longer than the longest transaction) when it fits
  // in 1/32 of the device memory, as the engine decides
  const uint64_t depth = std::max<uint32_t>(3, std::min<uint64_t>(max_len, rows)) - 1;
  const uint64_t full = 4ull * (stride + 2 * rows + 8) * depth * grid;
  b += full <= total_mem / 32 ? full : 4ull * (stride + 2 * rows + 8) * (fim::kDfsDepthHint + 1) * grid;
  // the projected DFS of wide rows: class database parts, transactions, the warps' stacks
  if (stride > 2048) b += fim::proj_footprint_bytes((uint32_t)rows, (uint32_t)stride, nnz, (uint32_t)grid);
  b += 64ull << 20;                                       // output, sample, small buffers
  return b;
}

void run_job(fim_server* srv, Job* j, cudaStream_t st) {
  if (j->status != FIM_OK) return;
  cudaSetDevice(srv->device);
  fim_db* db = nullptr;
  fim_status s;
  if (j->d_csr) {
    uint32_t* const d_off = static_cast<uint32_t*>(j->d_csr);
    const cudaError_t e = cudaStreamWaitEvent(st, j->ev_csr, 0);
    s = e != cudaSuccess ? fim::cuda_fail(e, "waiting for the upload")
                         : fim::build_uploaded_db(d_off, d_off + j->csr_items / 4, j->nnz, j->D, j->N, 64, j->minsup, st, &db);
  } else {
    s = fim_build_vertical_db(j->off.data(), j->items.data(), j->D, j->N, 64, j->minsup, st, &db);
  }
  if (s == FIM_OK) db->served = true;
  if (s == FIM_OK && j->sample_rate > 0.0) {
    s = fim_estimate_class_costs(db, j->sample_rate, (double)j->minsup / (double)j->D, 1000 + j->id, nullptr,
                                 nullptr);
  }
  if (s == FIM_OK) {
    fim_mine_opts o;
    fim_mine_opts_init(&o);
    o.ctas_per_sm = srv->ctas_per_sm;
    o.donate = 0;
    o.max_itemsets = srv->max_itemsets;
    s = fim_mine(db, j->minsup, &o, &j->result);
  }
  if (s != FIM_OK) j->error = fim_last_error();
  j->status = s;
  fim_db_free(db);
}

void worker_main(fim_server* srv, size_t slot) {
  cudaSetDevice(srv->device);
  cudaStream_t st = srv->streams[slot];
  for (;;) {
    Job* j = nullptr;
    {
      std::unique_lock<std::mutex> lock(srv->mu);
      std::deque<Job*>::iterator next;
      srv->cv_work.wait(lock, [&] {
        if (srv->stop) return true;
        // the first job whose database has been copied (one whose submitter is still at it holds nobody up).  A job larger
        // than the budget runs alone: with no other in flight, nor one that has its room already
        next = std::find_if(srv->queue.begin(), srv->queue.end(), [](const Job* q) { return q->ready; });
        if (next == srv->queue.end()) return false;
        return (*next)->reserved || srv->in_use == 0 || srv->in_use + (*next)->footprint <= srv->budget;
      });
      if (srv->stop) return;
      j = *next;
      srv->queue.erase(next);
      if (!j->reserved) srv->in_use += j->footprint;
      srv->in_flight += 1;
      srv->peak_in_flight = std::max(srv->peak_in_flight, srv->in_flight);
    }
    j->t_start = Clock::now();
    // (events on the slot's stream bracket the job's device work; timing only, no synchronisation)
    if (cudaEventCreate(&j->ev_start) == cudaSuccess) cudaEventRecord(j->ev_start, st);
    run_job(srv, j, st);
    if (cudaEventCreate(&j->ev_end) == cudaSuccess) cudaEventRecord(j->ev_end, st);
    if (j->d_csr) cudaFreeAsync(j->d_csr, st);
    j->d_csr = nullptr;
    if (j->ev_csr) cudaEventDestroy(j->ev_csr);
    j->ev_csr = nullptr;
    j->t_end = Clock::now();
    {
      std::lock_guard<std::mutex> lock(srv->mu);
      srv->in_use -= j->footprint;
      srv->uploaded -= j->csr_bytes;
      srv->in_flight -= 1;
      j->off.clear();
      j->off.shrink_to_fit();
      j->items.clear();
      j->items.shrink_to_fit();
      j->done = true;
    }
    srv->cv_done.notify_all();
    srv->cv_work.notify_all();
  }
}

constexpr size_t kStageBytes = 8 << 20;

bool upload_create(fim_server* srv) {
  if (cudaStreamCreateWithFlags(&srv->up_stream, cudaStreamNonBlocking) != cudaSuccess) {
    srv->up_stream = nullptr;
    return false;
  }
  for (uint32_t b = 0; b < 2; ++b) {
    if (cudaMallocHost(reinterpret_cast<void**>(&srv->stage[b]), kStageBytes) != cudaSuccess) return false;
    if (cudaEventCreateWithFlags(&srv->stage_free[b], cudaEventDisableTiming) != cudaSuccess) return false;
  }
  try {
    const uint32_t cores = std::thread::hardware_concurrency();
    srv->crew.reset(new Crew(cores > 5 ? 5 : cores > 1 ? cores - 1 : 0));
  } catch (const std::bad_alloc&) {
    return false;
  }
  return true;
}

void upload_release(fim_server* srv) {
  srv->crew.reset();
  if (srv->up_stream) cudaStreamSynchronize(srv->up_stream);
  for (uint32_t b = 0; b < 2; ++b) {
    if (srv->stage[b]) cudaFreeHost(srv->stage[b]);
    if (srv->stage_free[b]) cudaEventDestroy(srv->stage_free[b]);
    srv->stage[b] = nullptr;
    srv->stage_free[b] = nullptr;
  }
  if (srv->up_stream) cudaStreamDestroy(srv->up_stream);
  srv->up_stream = nullptr;
}

// The submitted database copied to the device by the submitting thread through two pinned buffers that it and the crew fill
// in turn.  On return the caller may reuse its arrays; the job's stream waits for the last buffer's copy (ev_csr).
// The copy engine can read pageable memory itself, at 100 to 150 GB/s, but arrays that the device has not read before may
// take it ten times as long, and a service gets new arrays with every request: bursts of 12 jobs (71 MB) took 3 to 15 ms that
// way, through the buffers 2.5 (2.1 and 1.9 when the same arrays come again).  One thread copies 23 GB/s, four 50.
// False, with no error left behind: no memory; the host copy takes its place.
bool upload(fim_server* srv, Job* j, const uint32_t* off, const uint32_t* items) {
  int dev = 0;
  // (a capture that the calling thread has open is not disturbed by calls on another stream)
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) return false;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess && dev != srv->device) e = cudaSetDevice(srv->device);
  if (e == cudaSuccess) {
    std::lock_guard<std::mutex> lock(srv->up_mu);
    void* p = nullptr;
    e = fim::dev_malloc_async(&p, j->csr_bytes, srv->up_stream);
    if (e == cudaSuccess) {
      // the offsets and, csr_items bytes further, the items as one run of bytes
      const uint64_t off_bytes = ((uint64_t)j->D + 1) * 4, end = j->csr_items + j->nnz * 4;
      for (uint64_t at = 0; at < end && e == cudaSuccess;) {
        const uint32_t b = srv->stage_turn++ & 1u;
        const uint64_t n = std::min<uint64_t>(kStageBytes, end - at);
        e = cudaEventSynchronize(srv->stage_free[b]);
        if (e != cudaSuccess) break;
        if (at < off_bytes)
          srv->crew->copy(srv->stage[b], reinterpret_cast<const uint8_t*>(off) + at, std::min(n, off_bytes - at));
        if (at + n > j->csr_items) {
          const uint64_t skip = std::max(at, j->csr_items);
          srv->crew->copy(srv->stage[b] + (skip - at), reinterpret_cast<const uint8_t*>(items) + (skip - j->csr_items),
                          at + n - skip);
        }
        e = cudaMemcpyAsync(static_cast<uint8_t*>(p) + at, srv->stage[b], n, cudaMemcpyHostToDevice, srv->up_stream);
        if (e == cudaSuccess) e = cudaEventRecord(srv->stage_free[b], srv->up_stream);
        at += n;
      }
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&j->ev_csr, cudaEventDisableTiming);
      if (e == cudaSuccess) e = cudaEventRecord(j->ev_csr, srv->up_stream);
      if (e == cudaSuccess) {
        j->d_csr = p;
      } else {
        cudaStreamSynchronize(srv->up_stream);
        cudaFreeAsync(p, srv->up_stream);
      }
    }
  }
  if (dev != srv->device) cudaSetDevice(dev);
  cudaThreadExchangeStreamCaptureMode(&mode);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess;
}

}  // namespace

using namespace fim;

extern "C" {

fim_status fim_server_create(uint64_t hbm_budget_bytes, uint32_t slots, uint32_t ctas_per_sm, uint64_t max_itemsets,
                             fim_server** out) {
  if (!out) return fail(FIM_ERR_INVALID, "out is NULL");
  *out = nullptr;
  if (slots == 0 || slots > 64) return fail(FIM_ERR_INVALID, "slots must be in 1..64");
  fim_server* srv = new (std::nothrow) fim_server();
  if (!srv) return fail(FIM_ERR_OOM, "host allocation");
  {
    size_t free_b = 0, total_b = 0;
    cudaError_t e = cudaGetDevice(&srv->device);
    if (e == cudaSuccess) e = cudaMemGetInfo(&free_b, &total_b);
    if (e != cudaSuccess) {
      delete srv;
      return cuda_fail(e, "server device");
    }
    srv->total_mem = total_b;
    if (hbm_budget_bytes == 0) hbm_budget_bytes = (uint64_t)(free_b * 0.8);
  }
  srv->budget = hbm_budget_bytes;
  srv->ctas_per_sm = ctas_per_sm ? ctas_per_sm : 1;
  srv->max_itemsets = max_itemsets;
  for (uint32_t k = 0; k < slots; ++k) {
    cudaStream_t s;
    cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      for (auto x : srv->streams) cudaStreamDestroy(x);
      delete srv;
      return cuda_fail(e, "server stream");
    }
    srv->streams.push_back(s);
  }
  if (!upload_create(srv)) {  // (every submission is copied on the host)
    upload_release(srv);
    cudaGetLastError();
  }
  if (cudaEventCreate(&srv->ev_origin) == cudaSuccess) cudaEventRecord(srv->ev_origin, srv->streams[0]);
  for (uint32_t k = 0; k < slots; ++k) srv->workers.emplace_back(worker_main, srv, (size_t)k);
  *out = srv;
  return FIM_OK;
}

fim_status fim_server_submit(fim_server* srv, const uint32_t* tx_offsets, const uint32_t* tx_items, uint32_t D,
                             uint32_t N, uint32_t minsup_abs, double sample_rate, uint64_t* job_id) {
  if (!srv || !tx_offsets || !job_id || D == 0 || N == 0 || minsup_abs == 0)
    return fail(FIM_ERR_INVALID, "bad server submission");
  Job* j = new (std::nothrow) Job();
  if (!j) return fail(FIM_ERR_OOM, "host allocation");
  j->t_submit = Clock::now();
  const uint64_t nnz = tx_offsets[D];
  j->nnz = nnz;
  j->D = D;
  j->N = N;
  j->minsup = minsup_abs;
  j->sample_rate = sample_rate;
  int nsm = 152;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, srv->device);
  // the longest transaction, and whether the build will refuse the offsets
  std::atomic<uint32_t> longest{0}, refused{tx_offsets[0] != 0};
  auto scan = [&](uint32_t t0, uint32_t t1) {
    uint32_t m = 0, r = 0;
    for (uint32_t t = t0; t < t1; ++t) {
      const uint32_t a = tx_offsets[t], b = tx_offsets[t + 1], n = b > a ? b - a : 0u;
      m = n > m ? n : m;
      r |= b < a;
    }
    uint32_t seen = longest.load();
    while (m > seen && !longest.compare_exchange_weak(seen, m)) {}
    if (r) refused = 1;
  };
  {
    constexpr uint32_t kPiece = 16384;
    std::unique_lock<std::mutex> lock(srv->up_mu, std::defer_lock);
    if (srv->crew && D > 2 * kPiece && lock.try_lock())
      srv->crew->run((D + kPiece - 1) / kPiece, [&](uint64_t k) {
        scan((uint32_t)k * kPiece, (uint32_t)std::min<uint64_t>(D, (k + 1) * kPiece));
      });
    else
      scan(0, D);
  }
  const uint32_t max_len = longest, bad = refused;
  j->footprint = job_footprint(D, N, nnz, max_len, minsup_abs, (uint32_t)nsm * srv->ctas_per_sm, srv->total_mem, nsm);
  // The submitter uploads the database when the job's footprint fits the budget now and no queued job waits for room (the
  // jobs stay in arrival order).  Else, and for offsets that the build will refuse, it is copied on the host, outside the
  // budget (a burst of 12 jobs with 71 MB: 1.8 ms to submit with uploads, 5.4 with host copies).
  j->csr_items = (((uint64_t)D + 1) * 4 + 255) & ~255ull;
  const uint64_t csr_bytes = j->csr_items + std::max<uint64_t>(1, nnz) * 4;
  bool up = srv->up_stream && !bad && (tx_items || nnz == 0);
  {
    std::lock_guard<std::mutex> lock(srv->mu);
    up = up && srv->in_use + j->footprint <= srv->budget && srv->uploaded + csr_bytes <= srv->total_mem / 32;
    for (const Job* q : srv->queue) up = up && q->reserved;
    if (up) {
      j->reserved = true;
      j->csr_bytes = csr_bytes;
      srv->in_use += j->footprint;
      srv->uploaded += csr_bytes;
    }
    j->id = srv->next_id++;
    *job_id = j->id;
    srv->jobs[j->id] = j;
    srv->queue.push_back(j);
  }
  const bool on_device = up && upload(srv, j, tx_offsets, tx_items);
  bool copied = true;
  if (!on_device) {
    try {
      j->off.assign(tx_offsets, tx_offsets + D + 1);
      if (nnz) j->items.assign(tx_items, tx_items + nnz);
    } catch (const std::bad_alloc&) {
      copied = false;
    }
  }
  {
    std::lock_guard<std::mutex> lock(srv->mu);
    if (up && !on_device) {  // (it keeps its room in the budget)
      srv->uploaded -= j->csr_bytes;
      j->csr_bytes = 0;
    }
    if (!copied) {  // (the job is in the queue: its wait reports it)
      j->status = FIM_ERR_OOM;
      j->error = "host copy of a submitted database";
    }
    j->ready = true;
  }
  srv->cv_work.notify_all();
  return FIM_OK;
}

fim_status fim_server_wait(fim_server* srv, uint64_t job_id, fim_result** out, double* latency_s,
                           double* service_s) {
  return fim_server_wait_ex(srv, job_id, out, latency_s, service_s, nullptr, nullptr);
}

fim_status fim_server_wait_ex(fim_server* srv, uint64_t job_id, fim_result** out, double* latency_s,
                              double* service_s, double* device_start_ms, double* device_end_ms) {
  if (device_start_ms) *device_start_ms = -1.0;
  if (device_end_ms) *device_end_ms = -1.0;
  if (!srv || !out) return fail(FIM_ERR_INVALID, "server or out is NULL");
  *out = nullptr;
  Job* j = nullptr;
  {
    std::unique_lock<std::mutex> lock(srv->mu);
    auto it = srv->jobs.find(job_id);
    if (it == srv->jobs.end() || it->second->taken) return fail(FIM_ERR_INVALID, "unknown job id");
    j = it->second;
    j->taken = true;
    srv->cv_done.wait(lock, [&] { return j->done; });
    srv->jobs.erase(it);
  }
  if (latency_s) *latency_s = std::chrono::duration<double>(j->t_end - j->t_submit).count();
  if (service_s) *service_s = std::chrono::duration<double>(j->t_end - j->t_start).count();
  // the job's device interval from the server's origin event (both events completed: the job's result
  // was synchronised on its stream before the worker marked it done)
  float t0 = -1.f, t1 = -1.f;
  if (srv->ev_origin && j->ev_start && j->ev_end && cudaEventSynchronize(j->ev_end) == cudaSuccess &&
      cudaEventElapsedTime(&t0, srv->ev_origin, j->ev_start) == cudaSuccess &&
      cudaEventElapsedTime(&t1, srv->ev_origin, j->ev_end) == cudaSuccess) {
    if (device_start_ms) *device_start_ms = t0;
    if (device_end_ms) *device_end_ms = t1;
  }
  if (j->ev_start) cudaEventDestroy(j->ev_start);
  if (j->ev_end) cudaEventDestroy(j->ev_end);
  fim_status s = j->status;
  if (s == FIM_OK) *out = j->result;
  else set_error(j->error);
  delete j;
  return s;
}

fim_status fim_server_stats(fim_server* srv, uint64_t* in_use_bytes, uint32_t* in_flight, uint32_t* peak_in_flight,
                            uint64_t* queued) {
  if (!srv) return fail(FIM_ERR_INVALID, "server is NULL");
  std::lock_guard<std::mutex> lock(srv->mu);
  if (in_use_bytes) *in_use_bytes = srv->in_use;
  if (in_flight) *in_flight = srv->in_flight;
  if (peak_in_flight) *peak_in_flight = srv->peak_in_flight;
  if (queued) *queued = srv->queue.size();
  return FIM_OK;
}

void fim_server_free(fim_server* srv) {
  if (!srv) return;
  {
    std::lock_guard<std::mutex> lock(srv->mu);
    srv->stop = true;
  }
  srv->cv_work.notify_all();
  for (auto& t : srv->workers) t.join();
  for (auto& kv : srv->jobs) {  // (the queued jobs are among them)
    if (kv.second->d_csr) cudaFreeAsync(kv.second->d_csr, srv->up_stream);  // (never started)
    if (kv.second->result) fim_result_free(kv.second->result);
    if (kv.second->ev_csr) cudaEventDestroy(kv.second->ev_csr);
    if (kv.second->ev_start) cudaEventDestroy(kv.second->ev_start);
    if (kv.second->ev_end) cudaEventDestroy(kv.second->ev_end);
    delete kv.second;
  }
  for (auto s : srv->streams) cudaStreamDestroy(s);
  upload_release(srv);
  if (srv->ev_origin) cudaEventDestroy(srv->ev_origin);
  delete srv;
}

}  // extern "C"
