// first_use.h - a step's first use under CUDA graphs: run as plain launches, then
// captured for the next uses while the GPU is at work (capturing 250 launches before
// the first of them runs would hold a request's first step for a millisecond).
//
// The step's launches commit tokens, so what the caller is told is whether they were
// enqueued.  A capture that fails after them is not the step's failure: the step stays
// uncaptured, and its next use comes here again.
#pragma once

namespace memspec {

// `run` enqueues the step's launches and returns their status (0: enqueued).  Graphs
// makes the CUDA calls (the tests' stand-in makes them fail):
//   bool begin()                         start capturing the step's stream
//   bool end(Graph* g)                   end it; *g is null or to be destroyed
//   bool instantiate(Exec* x, Graph g)
//   void destroy(Graph g)
//   void clear_error()                   forget the error of the call that failed
// Returns run's status; *exec is the executable graph, or null.
template <class Graphs, class Run>
auto run_then_capture(Graphs& cu, Run&& run, typename Graphs::Exec* exec) -> decltype(run()) {
  *exec = nullptr;
  const auto status = run();
  if (status != 0) return status;
  bool ok = cu.begin();
  if (ok) {
    const bool recorded = run() == 0;
    typename Graphs::Graph graph = nullptr;
    ok = cu.end(&graph) && recorded && graph != nullptr;   // ended in any case
    if (ok && !cu.instantiate(exec, graph)) {
      ok = false;
      *exec = nullptr;
    }
    if (graph != nullptr) cu.destroy(graph);
  }
  if (!ok) cu.clear_error();
  return status;
}

}  // namespace memspec
