// What a mask of solid cells is like: how much surface it has, and how many
// separate regions the fluid falls into.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

struct MaskShape {
    long long solid = 0;  // solid cells
    long long faces = 0;  // faces between a fluid and a solid cell
    long long rooms = 0;  // regions of two or more fluid cells joined by faces
};

// n cells along x, y, z; periodic axes wrap.  Linear in the cells: the fluid's
// runs along x are the elements that are joined across rows.
inline MaskShape mask_shape(const int n[3], const bool periodic[3], const uint8_t* solid) {
    MaskShape m;
    const int nx = n[0], ny = n[1], nz = n[2];
    const long long rows = (long long)ny * nz;
    std::vector<int> from, to;               // runs of fluid cells [from, to)
    std::vector<int> first((size_t)rows + 1);  // a row's first run
    std::vector<int> up;                     // a run's parent
    auto root = [&](int r) {
        while (up[r] != r) r = up[r] = up[up[r]];
        return r;
    };
    auto join = [&](int a, int b) {
        a = root(a);
        b = root(b);
        if (a != b) up[std::max(a, b)] = std::min(a, b);
    };
    auto cells = [&](long long row) { return solid + row * nx; };
    for (long long row = 0; row < rows; ++row) {
        first[row] = (int)from.size();
        const uint8_t* s = cells(row);
        for (int i = 0; i < nx;) {
            const int b = i;
            const bool fluid = s[i] == 0;
            while (i < nx && (s[i] == 0) == fluid) ++i;
            if (fluid) {
                from.push_back(b);
                to.push_back(i);
                up.push_back((int)up.size());
            } else {
                m.solid += i - b;
            }
            if (i < nx) ++m.faces;
        }
        if (periodic[0] && (s[0] == 0) != (s[nx - 1] == 0)) ++m.faces;
        if (periodic[0] && s[0] == 0 && s[nx - 1] == 0) join(first[row], (int)from.size() - 1);
    }
    first[rows] = (int)from.size();
    auto rows_meet = [&](long long p, long long q) {
        const uint8_t *s = cells(p), *t = cells(q);
        long long f = 0;
        for (int i = 0; i < nx; ++i) f += (s[i] == 0) != (t[i] == 0);
        m.faces += f;
        int a = first[p], b = first[q];
        while (a < first[p + 1] && b < first[q + 1]) {
            if (from[a] < to[b] && from[b] < to[a]) join(a, b);
            if (to[a] < to[b])
                ++a;
            else
                ++b;
        }
    };
    for (int k = 0; k < nz; ++k)
        for (int j = 0; j < ny; ++j) {
            const long long row = (long long)k * ny + j;
            if (j > 0) rows_meet(row, row - 1);
            else if (periodic[1]) rows_meet(row, row + ny - 1);
            if (k > 0) rows_meet(row, row - ny);
            else if (periodic[2]) rows_meet(row, row + (long long)(nz - 1) * ny);
        }
    std::vector<long long> size(up.size(), 0);
    for (size_t r = 0; r < up.size(); ++r) size[root((int)r)] += to[r] - from[r];
    for (long long c : size) m.rooms += c > 1;
    return m;
}
