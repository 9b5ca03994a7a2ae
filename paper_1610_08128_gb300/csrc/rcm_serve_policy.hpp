// rcm_serve_policy.hpp -- which executor a served request runs on. Plain C++ (no CUDA).
#pragma once

#include <algorithm>

namespace rcm {

// A request runs on one CTA of kServeThreads threads or, from a size on, on a thread-block cluster. One CTA
// with its state in shared memory orders up to a million vertices in half the SM time a cluster needs, so
// under load only the largest requests take clusters; with few requests in the server latency is what
// counts, and idle SMs cost nothing.
//
// GB300, milliseconds for all requests submitted at once: on clusters of 8 from 524,288 vertices; on one CTA
// of 512 threads below 1,048,576; on one of 256 (clusters of 4 from 524,288, the engines of before the
// shared-memory state):
//   one 3D grid of 600,000 vertices        3.8   11.7   15.9  (6.4)
//   one 3D grid of 900,000                 5.1   19.2   25.5  (9.0)
//   one degree-8 random graph of 600,000  10.3   45.4   71.2  (57.5)
//   8 of 525,000 to 1,040,000             23.8   32.2   54.0  (26.8)
//   16 of those                           38.2   26.1   35.2  (47.5)
//   48 of those                           83.4   38.0   60.6  (107)
//   200 of those                          403    102    145   (492)
//   48 of 1,000 to 4M                     98.0   83.6   81.3  (126)
//   128 of 1,000 to 2M                    62.7   64.2   95.6  (77)
//   400 of 1,000 to 1M                    88.2   54.0   82.2  (114)
// At full load (256 in flight, 32 hardware queues), orderings a second on one CTA of 512 / 256 / 128 threads:
// 800 of 1,000 to 4M vertices 2,768 / 2,698 / 2,488; 2,000 up to 300,000: 28,100 / 23,700 / 19,900; 4,000 up to
// 20,000: 34,300 / 34,100 / 34,000.
constexpr int kServeThreads = 512;
constexpr long long kServeClusterMin = 1LL << 20;
constexpr long long kServeClusterMinAlone = 1LL << 19;  // with at most kServeAlone requests in the server
constexpr int kServeAlone = 8;
// CTAs of a cluster: under load, and with at most kServeFew requests in the server (48 requests of 1,000 to 4M
// vertices 75 to 90 ms with 8, 90 to 100 with 4; 800 of them 1,838 orderings/s with 8, 2,702 with 4).
constexpr int kServeClusterBlocks = 4;
constexpr int kServeClusterIdle = 8;
constexpr int kServeFew = 64;

// CTAs of the cluster that takes a request of n vertices admitted with `load` requests in the server (itself
// and those waiting included); 0: one CTA. min_vertices and blocks: the server's options (0 = by load,
// min_vertices -1 = never); most: the largest cluster the device allows (0 = none).
inline int serve_cluster(long long n, int load, long long min_vertices, int blocks, int most) {
    if (min_vertices < 0 || most <= 0) return 0;
    if (n < (min_vertices ? min_vertices : load <= kServeAlone ? kServeClusterMinAlone : kServeClusterMin)) return 0;
    return blocks ? blocks : std::min(load <= kServeFew ? kServeClusterIdle : kServeClusterBlocks, most);
}

}  // namespace rcm
