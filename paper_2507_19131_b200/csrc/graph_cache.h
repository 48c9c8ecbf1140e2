// Which calls of a context are recorded as CUDA graphs, and which recorded graphs are kept.  Bookkeeping only, no CUDA:
// `Exec` is the graph handle.  Not thread-safe by itself (the context's graph_lock guards it).
//
// Recording a call costs the host several times what issuing its launches does, so a recording has to be earned by
// replays: a caller that rotates through many buffers, keeps every result or sets new ratios on each call would otherwise
// pay it on every call.  A call is identified by its key, every value that shapes its launches.
//   - The first call with a key issues its launches; the key is remembered (the newest `max_keys` keys are).
//   - The second one is recorded, as long as the recordings stay within max_graphs + replays / REPLAYS_PER_RECORDING:
//     the kept set can be filled once for free, every further recording takes the place of a graph that was of use.
//   - Beyond that budget a key is recorded at its PATIENCE-th call: by then its launches have cost more than a recording
//     does, so a program that settles on new arguments gets its graph and one that never does pays a bounded share.
// Kept graphs and remembered keys leave in the order of their last use.
#pragma once
#include <cstddef>
#include <string>
#include <utility>
#include <vector>

namespace mixaq {

template <class Exec>
class GraphCache {
 public:
  struct Graph { std::string key; Exec exec; int launches; };
  static constexpr long REPLAYS_PER_RECORDING = 32;
  static constexpr int PATIENCE = 32;

  GraphCache(size_t max_graphs, size_t max_keys) : max_graphs_(max_graphs), max_keys_(max_keys) {}

  // the graph recorded for the key, NULL: none
  const Graph* replay(const std::string& key) {
    for (size_t i = graphs_.size(); i-- > 0;)
      if (graphs_[i].key == key) {
        ++replays_;
        move_to_back(graphs_, i);
        return &graphs_.back();
      }
    return nullptr;
  }
  // whether the call about to be made should be recorded; a call that is not, and succeeds, is then noted with saw()
  bool worth_recording(const std::string& key) const {
    for (const Seen& s : seen_)
      if (s.key == key)
        return s.calls + 1 >= PATIENCE || recordings_ < (long)max_graphs_ + replays_ / REPLAYS_PER_RECORDING;
    return false;
  }
  void saw(std::string key) {
    for (size_t i = seen_.size(); i-- > 0;)
      if (seen_[i].key == key) {
        ++seen_[i].calls;
        move_to_back(seen_, i);
        return;
      }
    if (seen_.size() >= max_keys_) seen_.erase(seen_.begin());
    seen_.push_back({std::move(key), 1});
  }
  // a recording succeeded; destroy(exec) is called for the graph it displaces
  template <class Destroy>
  void recorded(std::string key, Exec exec, int launches, Destroy destroy) {
    ++recordings_;
    forget(key);
    if (graphs_.size() >= max_graphs_) {
      destroy(graphs_.front().exec);
      graphs_.erase(graphs_.begin());
    }
    graphs_.push_back({std::move(key), exec, launches});
  }
  // a recording failed: the key starts again (and the attempt counts)
  void not_recorded(const std::string& key) {
    ++recordings_;
    forget(key);
  }
  template <class Destroy>
  void clear(Destroy destroy) {
    for (Graph& g : graphs_) destroy(g.exec);
    graphs_.clear();
    seen_.clear();
  }

 private:
  struct Seen { std::string key; int calls; };
  template <class T>
  static void move_to_back(std::vector<T>& v, size_t i) {
    for (; i + 1 < v.size(); ++i) std::swap(v[i], v[i + 1]);
  }
  void forget(const std::string& key) {
    for (size_t i = 0; i < seen_.size(); ++i)
      if (seen_[i].key == key) { seen_.erase(seen_.begin() + i); return; }
  }
  const size_t max_graphs_, max_keys_;
  std::vector<Graph> graphs_;
  std::vector<Seen> seen_;
  long recordings_ = 0, replays_ = 0;
};

}  // namespace mixaq
