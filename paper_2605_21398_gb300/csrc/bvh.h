// The bounding-volume tree over an object's triangles, as the host makes it (its
// spheres and slabs are made on the device).
#pragma once
#include <algorithm>
#include <exception>
#include <thread>
#include <vector>

#include "dock_internal.h"

namespace dock {

// The tree over triangles (object frame): median split on the longest centroid
// axis, leaves of <= 4 triangles.  Node spheres and slabs are made on the device
// (launch_node_records); the host decides the splits.  A node's centroids are
// moved with its triangles, so every pass over them is sequential; subtrees of
// many triangles are built by threads of their own, at most as many as the
// machine runs at once (the number of nodes below n triangles depends on n alone,
// so every subtree knows its place and the tree does not depend on the threads).
struct BvhItem {
    double c[3];   // centre of the triangle's box
    int32_t t;
};

struct BvhBuilder {
    std::vector<BvhItem> items;
    std::vector<BvhNode> nodes;
    std::vector<int32_t> order;   // leaf slot -> triangle
    static constexpr int THREAD_MIN = 4096;   // triangles that are worth a thread (about 1 ms)

    // nodes of a tree over n triangles
    static int64_t size(int64_t n)
    {
        // n / 2 and n - n / 2 differ by at most one: two sizes per level
        int64_t a = n, ca = 1, cb = 0, total = 0;   // ca trees of a triangles, cb of a + 1
        while (ca + cb > 0) {
            total += ca + cb;
            // halves of a and a + 1 that are split again
            const int64_t h = a / 2;
            int64_t nh = 0, nh1 = 0;
            if (a > 4) { if (a & 1) { nh += ca; nh1 += ca; } else nh += 2 * ca; }
            if (a + 1 > 4) { if ((a + 1) & 1) { nh += cb; nh1 += cb; } else nh1 += 2 * cb; }
            a = h;
            ca = nh;
            cb = nh1;
        }
        return total;
    }

    // node over items [lo, hi) by `threads` threads (this one among them); its
    // descendants take nodes [next, ...)
    void build(int node, int lo, int hi, int64_t next, int threads)
    {
        const int n = hi - lo;
        BvhNode &nd = nodes[node];
        nd.first = lo;
        nd.count = n;
        nd.pad = 0;
        if (n <= 4) {
            nd.left = -1;
            for (int i = lo; i < hi; ++i) order[i] = items[i].t;
            return;
        }
        double clo[3] = {1e300, 1e300, 1e300}, chi[3] = {-1e300, -1e300, -1e300};
        for (int i = lo; i < hi; ++i)
            for (int a = 0; a < 3; ++a) {
                clo[a] = std::min(clo[a], items[i].c[a]);
                chi[a] = std::max(chi[a], items[i].c[a]);
            }
        int ax = 0;
        double ext = -1;
        for (int a = 0; a < 3; ++a) if (chi[a] - clo[a] > ext) { ext = chi[a] - clo[a]; ax = a; }
        const int mid = (int)(((int64_t)lo + hi) / 2);
        std::nth_element(items.begin() + lo, items.begin() + mid, items.begin() + hi,
                         [ax](const BvhItem &x, const BvhItem &y) {
                             return x.c[ax] < y.c[ax] || (x.c[ax] == y.c[ax] && x.t < y.t);
                         });
        const int l = (int)next;
        nd.left = l;
        const int64_t next_l = next + 2, next_r = next_l + size(mid - lo) - 1;
        std::thread th;
        const int other = n >= 2 * THREAD_MIN ? threads / 2 : 0;
        if (other > 0) {
            try {
                th = std::thread([=] { build(l, lo, mid, next_l, other); });
            } catch (const std::exception &) {
                // no thread to be had: build it here
            }
        }
        const int mine = th.joinable() ? threads - other : threads;
        if (!th.joinable()) build(l, lo, mid, next_l, mine);
        build(l + 1, mid, hi, next_r, mine);
        if (th.joinable()) th.join();
    }
};

inline void build_bvh(const double *V, const int32_t *T, int64_t nt, BvhBuilder &B, int threads)
{
    B.items.resize(nt);
    B.order.resize(nt);
    B.nodes.resize(BvhBuilder::size(nt));
    for (int64_t t = 0; t < nt; ++t) {
        for (int a = 0; a < 3; ++a) {
            const double x0 = V[3 * (int64_t)T[3 * t] + a], x1 = V[3 * (int64_t)T[3 * t + 1] + a], x2 = V[3 * (int64_t)T[3 * t + 2] + a];
            B.items[t].c[a] = 0.5 * (std::min(x0, std::min(x1, x2)) + std::max(x0, std::max(x1, x2)));
        }
        B.items[t].t = (int32_t)t;
    }
    B.build(0, 0, (int)nt, 1, threads);
}

}  // namespace dock
