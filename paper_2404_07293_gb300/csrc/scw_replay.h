// When a plan's call launches its kernels, captures them into a CUDA graph or replays the graph it has.
// Host code without CUDA, so that the rule can be tested by itself.
#pragma once

namespace scw {

// A plan keeps one graph, for one key (its output). Capturing and instantiating takes about 50 us of host
// time, longer than the kernels of a mid-sized field, so only a key's second call in a row pays it: a program
// that brings a new solution (which drops the graph) or another output with every call never does.
struct ReplayRule {
  enum Step { LAUNCH, CAPTURE, REPLAY };
  const void* graph = nullptr;  // key of the captured graph; null: none
  const void* last = nullptr;   // key of the previous call

  Step next(const void* key) const { return graph == key ? REPLAY : (last == key ? CAPTURE : LAUNCH); }
  void done(Step step, const void* key) {
    last = key;
    if (step == CAPTURE) graph = key;
  }
  void drop() { graph = last = nullptr; }
};

}  // namespace scw
