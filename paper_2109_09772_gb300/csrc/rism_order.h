// rism_order.h -- the atoms' spatial order for the all-space pair sum (host only).
#pragma once

#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <vector>

namespace rism {

inline uint32_t spread10(uint32_t v) {  // the 10 low bits of v to every third bit
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// Spatial order of the atoms for the all-space pair sum: cells of about 32 atoms over the atoms' bounding box,
// the cells in Morton order, the atoms of a cell in index order (a stable counting sort, O(n)).  A warp then
// takes nearby targets and a tile nearby sources, so the costly short-range branch of the pair term is taken by
// whole warps or by none.  perm[k] = original index of the atom at position k.
inline void lra_order(const double* raw, int64_t n, int* perm) {
    double lo[3] = {raw[0], raw[1], raw[2]}, hi[3] = {raw[0], raw[1], raw[2]};
    for (int64_t i = 1; i < n; ++i)
        for (int d = 0; d < 3; ++d) {
            lo[d] = std::min(lo[d], raw[6 * i + d]);
            hi[d] = std::max(hi[d], raw[6 * i + d]);
        }
    double ext[3], vol = 1.0;
    for (int d = 0; d < 3; ++d) {
        ext[d] = std::max(hi[d] - lo[d], 1e-6);
        vol *= ext[d];
    }
    if (!std::isfinite(vol)) {  // atoms 1e100 A apart: no two of them are near, any order serves
        for (int64_t i = 0; i < n; ++i) perm[i] = (int)i;
        return;
    }
    const double side = std::cbrt(vol / (double)std::max<int64_t>(1, n / 32));
    int nc[3];
    double inv[3];  // cells per A: 1 / side, or what 1,024 cells allow over the length of a thin solute
    for (int d = 0; d < 3; ++d) {
        nc[d] = (int)std::max(1.0, std::min(1024.0, std::ceil(ext[d] / side)));
        inv[d] = std::min(1.0 / side, nc[d] / ext[d]);
    }
    const int64_t ncell = (int64_t)nc[0] * nc[1] * nc[2];
    std::vector<uint64_t> key((size_t)ncell);
    for (int z = 0; z < nc[2]; ++z)
        for (int y = 0; y < nc[1]; ++y)
            for (int x = 0; x < nc[0]; ++x) {
                const uint64_t m = spread10((uint32_t)x) | (spread10((uint32_t)y) << 1) | (spread10((uint32_t)z) << 2);
                const int64_t lin = ((int64_t)z * nc[1] + y) * nc[0] + x;
                key[(size_t)lin] = (m << 32) | (uint64_t)lin;
            }
    std::sort(key.begin(), key.end());
    std::vector<int> rank((size_t)ncell), start((size_t)ncell + 1, 0);
    for (int64_t r = 0; r < ncell; ++r) rank[(size_t)(key[(size_t)r] & 0xffffffffu)] = (int)r;
    std::vector<int> cell((size_t)n);
    for (int64_t i = 0; i < n; ++i) {
        int cc[3];
        for (int d = 0; d < 3; ++d)
            cc[d] = std::min(nc[d] - 1, (int)((raw[6 * i + d] - lo[d]) * inv[d]));  // between 0 and nc[d]
        cell[(size_t)i] = rank[(size_t)(((int64_t)cc[2] * nc[1] + cc[1]) * nc[0] + cc[0])];
        ++start[(size_t)cell[(size_t)i] + 1];
    }
    for (int64_t r = 0; r < ncell; ++r) start[(size_t)r + 1] += start[(size_t)r];
    for (int64_t i = 0; i < n; ++i) perm[start[(size_t)cell[(size_t)i]]++] = (int)i;
}

}  // namespace rism
