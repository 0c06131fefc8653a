// Host execution of the FP64 sum of 2D leaf angles (Angle64 of trav2d.cuh), test harness.
#include "../../paper_2605_19200_gb300/csrc/trav2d.cuh"

using namespace gwn;

// GWN of n straight leaves (x0 y0 x1 y1 each) at q, every `stride`-th leaf to one sum as the lanes
// of a warp take them
extern "C" double hx_angle64(const double* leaf, int n, double qx, double qy, int stride) {
    double w = 0;
    for (int s = 0; s < stride; ++s) {
        Angle64 a;
        for (int l = s; l < n; l += stride) {
            const double ax = leaf[4 * l] - qx, ay = leaf[4 * l + 1] - qy, bx = leaf[4 * l + 2] - qx, by = leaf[4 * l + 3] - qy;
            a.add(ax * bx + ay * by, ax * by - ay * bx);
        }
        w += a.value();
    }
    return w;
}
