// Launch-policy autotuner: the first call for a key (kernel, precision,
// shape) times every candidate policy with CUDA events on the caller's
// stream and keeps the fastest, in memory and, when GBMG_TUNE_CACHE names a
// file, on disk ("key value" lines, read on first use).  GBMG_TUNE=0 turns
// tuning off (the first candidate is used).  A stream that is being
// captured into a CUDA graph is never timed: the cached or first candidate
// is used, so tune (make one call) before capturing.
#pragma once

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <fstream>
#include <mutex>
#include <set>
#include <string>
#include <unordered_map>
#include <utility>
#include <vector>

#include "common.cuh"

namespace gbmg {

// The fastest candidate.  run(c, n) makes n launches of policy c one after the
// other and returns the milliseconds they took.  Every candidate is timed on
// three launches; those are tens of microseconds for a small kernel, where one
// delay on the host decides, so the candidates near the best are then timed
// again in turns, kRounds times on launches worth kRoundMs, and each counts by
// its fastest turn (a delay only ever adds).  times: milliseconds per launch.
// (A 14x8x6x6 fine operator on one vector: three launches alone picked one of
// 9.3 or of 11.7 us a call, by the process.)
template <typename Run>
int pick_fastest(const std::vector<int>& cands, Run&& run,
                 std::vector<std::pair<int, float>>& times) {
  constexpr int kRounds = 3;
  constexpr float kRoundMs = 0.15f, kLongMs = 2.f;
  times.clear();
  float best = 1e30f;
  for (int c : cands) {
    run(c, 1);  // warm-up
    times.emplace_back(c, run(c, 3) / 3.f);
    best = std::min(best, times.back().second);
  }
  if (best < kLongMs) {
    const float limit = 1.3f * best + 0.004f;
    std::vector<size_t> near;
    for (size_t i = 0; i < times.size(); ++i)
      if (times[i].second <= limit) near.push_back(i);
    for (int r = 0; near.size() > 1 && r < kRounds; ++r)
      for (size_t i : near) {
        const float t = std::max(times[i].second, 1e-4f);
        const int n = std::min(64, std::max(3, int(kRoundMs / t) + 1));
        times[i].second = std::min(times[i].second, run(times[i].first, n) / float(n));
      }
  }
  size_t pick = 0;
  for (size_t i = 1; i < times.size(); ++i)
    if (times[i].second < times[pick].second) pick = i;
  return times[pick].first;
}

class Tuner {
 public:
  static Tuner& get() {
    static Tuner t;
    return t;
  }

  // Returns the chosen candidate.  launch(c) must enqueue one launch with
  // policy c on stream st; it is called repeatedly while timing.
  template <typename F>
  int choose(const std::string& key, const std::vector<int>& cands, cudaStream_t st, F&& launch) {
    std::lock_guard<std::mutex> lk(mu_);
    load();
    auto it = best_.find(key);
    // a cached or pinned choice is used only if it is a candidate of this call
    if (it != best_.end() &&
        std::find(cands.begin(), cands.end(), it->second) != cands.end())
      return it->second;
    if (!enabled_ || cands.size() == 1) return cands.front();
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone)
      return cands.front();
    cudaEvent_t a, b;
    GB_CHECK(cudaEventCreate(&a));
    GB_CHECK(cudaEventCreate(&b));
    std::vector<std::pair<int, float>> times;
    const int pick = pick_fastest(
        cands,
        [&](int c, int n) {
          GB_CHECK(cudaEventRecord(a, st));
          for (int r = 0; r < n; ++r) launch(c);
          GB_CHECK(cudaEventRecord(b, st));
          GB_CHECK(cudaEventSynchronize(b));
          float ms = 0.f;
          GB_CHECK(cudaEventElapsedTime(&ms, a, b));
          return ms;
        },
        times);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    best_[key] = pick;
    timings_[key] = times;
    if (!path_.empty()) {
      std::ofstream f(path_, std::ios::app);
      if (f) f << key << " " << pick << "\n";
    }
    return pick;
  }

  // number of entries (tests)
  size_t size() {
    std::lock_guard<std::mutex> lk(mu_);
    return best_.size();
  }

  // pin a choice for key (choice < 0 removes the entry, so the next call
  // tunes again); the pin is not written to the cache file
  void set(const std::string& key, int choice) {
    std::lock_guard<std::mutex> lk(mu_);
    load();
    if (choice < 0) {
      best_.erase(key);
      pinned_.erase(key);
    } else {
      best_[key] = choice;
      pinned_.insert(key);
    }
  }
  // the fastest of the candidates first..last when `key` was tuned, if it came
  // within slack_ms of the pick; -1 if none did or the key is pinned or unknown
  int within(const std::string& key, int first, int last, float slack_ms) {
    std::lock_guard<std::mutex> lk(mu_);
    auto it = timings_.find(key);
    if (it == timings_.end() || pinned_.count(key)) return -1;
    int pick = -1;
    float best = 1e30f, ms = 1e30f;
    for (const auto& t : it->second) {
      best = std::min(best, t.second);
      if (t.first >= first && t.first <= last && t.second < ms) {
        ms = t.second;
        pick = t.first;
      }
    }
    return ms <= best + slack_ms ? pick : -1;
  }
  // the candidates timed when `key` was last tuned, with ms per launch
  std::vector<std::pair<int, float>> report(const std::string& key) {
    std::lock_guard<std::mutex> lk(mu_);
    auto it = timings_.find(key);
    return it == timings_.end() ? std::vector<std::pair<int, float>>{} : it->second;
  }
  int get(const std::string& key) {
    std::lock_guard<std::mutex> lk(mu_);
    load();
    auto it = best_.find(key);
    return it == best_.end() ? -1 : it->second;
  }

 private:
  Tuner() {
    const char* e = std::getenv("GBMG_TUNE");
    enabled_ = !(e && std::string(e) == "0");
    const char* p = std::getenv("GBMG_TUNE_CACHE");
    if (p) path_ = p;
  }
  void load() {
    if (loaded_) return;
    loaded_ = true;
    if (path_.empty()) return;
    std::ifstream f(path_);
    std::string k;
    int v;
    while (f >> k >> v) best_[k] = v;
  }
  std::mutex mu_;
  std::unordered_map<std::string, int> best_;
  std::unordered_map<std::string, std::vector<std::pair<int, float>>> timings_;
  std::set<std::string> pinned_;
  bool loaded_ = false;
  bool enabled_ = true;
  std::string path_;
};

}  // namespace gbmg
