// kf_copy.h -- the copy threads of the serving loop (host only).
#pragma once

#include <algorithm>
#include <condition_variable>
#include <cstddef>
#include <cstring>
#include <deque>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

namespace kfi {

// Host threads that share the large copies of kf_submit and kf_poll: an event
// is a few MB in and out, and one thread copies at ~15 GB/s, far below what the
// host memory delivers (13 GB/s into freshly allocated results, whose pages it
// touches first); the calling thread takes chunks too and returns when all of
// its event's chunks are done.  A small event is copied by the caller alone:
// waking the others takes longer.  It never throws.
class CopyPool {
 public:
  struct Piece {
    void* dst;
    const void* src;
    size_t bytes;
  };
  void start(int n_threads) {
    for (int i = 0; i < n_threads; ++i) threads_.emplace_back([this] { worker(); });
  }
  void stop() {
    {
      std::lock_guard<std::mutex> lk(mu_);
      stop_ = true;
    }
    cv_.notify_all();
    for (auto& t : threads_) t.join();
    threads_.clear();
  }
  void copy(const Piece* pieces, int n_pieces) {
    size_t total = 0;
    for (int p = 0; p < n_pieces; ++p) total += pieces[p].bytes;
    if (total <= kAlone) {
      for (int p = 0; p < n_pieces; ++p) std::memcpy(pieces[p].dst, pieces[p].src, pieces[p].bytes);
      return;
    }
    Job job;
    if (threads_.empty() || !queue(pieces, n_pieces, job)) {
      for (int p = 0; p < n_pieces; ++p) std::memcpy(pieces[p].dst, pieces[p].src, pieces[p].bytes);
      return;
    }
    cv_.notify_all();
    while (true) {  // help until the queue is empty, then wait for this job
      Chunk c;
      {
        std::lock_guard<std::mutex> lk(mu_);
        if (q_.empty()) break;
        c = q_.front();
        q_.pop_front();
      }
      run(c);
    }
    std::unique_lock<std::mutex> lk(job.m);
    job.cv.wait(lk, [&] { return job.left == 0; });
  }

 private:
  static constexpr size_t kChunk = size_t(1) << 19, kAlone = size_t(1) << 18;
  struct Job {
    std::mutex m;
    std::condition_variable cv;
    int left = 0;
  };
  struct Chunk {
    char* dst;
    const char* src;
    size_t bytes;
    Job* job;
  };
  // The pieces as chunks of `job` at the end of the queue; false, with nothing
  // queued, for a single chunk and when there is no memory for the queue (the
  // caller then copies alone: an exception would leave a C entry point with a
  // poll's ticket taken and chunks of a dead job queued).
  bool queue(const Piece* pieces, int n_pieces, Job& job) noexcept {
    try {
      std::vector<Chunk> chunks;
      for (int p = 0; p < n_pieces; ++p)
        for (size_t o = 0; o < pieces[p].bytes; o += kChunk)
          chunks.push_back({static_cast<char*>(pieces[p].dst) + o, static_cast<const char*>(pieces[p].src) + o,
                            std::min(kChunk, pieces[p].bytes - o), &job});
      if (chunks.size() <= 1) return false;
      job.left = int(chunks.size());
      std::lock_guard<std::mutex> lk(mu_);
      q_.insert(q_.end(), chunks.begin(), chunks.end());  // all or none
      return true;
    } catch (const std::bad_alloc&) {
      return false;
    }
  }
  static void run(const Chunk& c) {
    std::memcpy(c.dst, c.src, c.bytes);
    std::lock_guard<std::mutex> lk(c.job->m);
    if (--c.job->left == 0) c.job->cv.notify_all();
  }
  void worker() {
    while (true) {
      Chunk c;
      {
        std::unique_lock<std::mutex> lk(mu_);
        cv_.wait(lk, [&] { return stop_ || !q_.empty(); });
        if (q_.empty()) return;  // stopping
        c = q_.front();
        q_.pop_front();
      }
      run(c);
    }
  }
  std::mutex mu_;
  std::condition_variable cv_;
  std::deque<Chunk> q_;
  std::vector<std::thread> threads_;
  bool stop_ = false;
};

}  // namespace kfi
