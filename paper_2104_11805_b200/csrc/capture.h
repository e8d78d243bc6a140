// A chain of launches captured into a graph that can be launched.  The calls are a parameter, so that what happens where one of them fails
// can be looked at without a device.
#pragma once

namespace sdnn_plan {

// Api: begin(), end(&graph), last_error(), instantiate(&exec, graph), destroy(graph); all but the last give 0 where they succeed.
// body: enqueues the launches; gives 0 or its own code, which is then the result.  failed(error, what): what a failing call turns into.
// A graph is kept only if the body, every launch in it (one that failed is missing from the graph), the end of the capture and the
// instantiation all went well; *exec is left alone otherwise.  A capture that was begun is ended, whatever the body gave.
template <class Api, class Exec, class Body, class Failed>
int capture_graph(const Api& api, Exec* exec, const Body& body, const Failed& failed) {
    typename Api::Graph graph{};
    if (const auto e = api.begin()) return failed(e, "cudaStreamBeginCapture");
    int rc = body();
    const auto ended = api.end(&graph);
    const auto launches = api.last_error();
    Exec made{};
    if (!rc && ended) rc = failed(ended, "cudaStreamEndCapture");
    if (!rc && launches) rc = failed(launches, "a launch under capture");
    if (!rc) {
        if (const auto e = api.instantiate(&made, graph)) rc = failed(e, "cudaGraphInstantiate");
        else *exec = made;
    }
    if (graph) api.destroy(graph);
    return rc;
}

}  // namespace sdnn_plan
