// Candidate chunk lengths of the marching scheme step (host).
#pragma once
#include <algorithm>
#include <functional>
#include <vector>

namespace iewpf {

// Lengths of 1, 2, 3, 4, 5, 6, 8, 10, 12, 16, ... equal chunks of ny rows, down
// to 2 rows, or to 8 where that takes more than 32 chunks (the 8 rows around a
// chunk that are computed again cost more than further warps give), and of
// chunks of 16, 32, ... 512 rows: on grids that fill the GPU once or twice it is
// the number of warps that counts, and no rule knows the best.  Longest first.
// 16 scheme steps with 1, 2, 3, 4, 6, 8, 16 and 32 chunks alone -> with these: 60
// x 1000 x 4 particles 560 -> 350 us, 700 x 700 x 2 583 -> 545, 400 x 400 x 3 462
// -> 403 (581 and 422 without the powers of two), 300 x 200 x 10 490 -> 455.
inline std::vector<int> march_rows(int ny)
{
    std::vector<int> th;
    auto chunks = [&](int n) { th.push_back((ny + n - 1) / n); };
    for (int p = 1; p <= ny / 2; p *= 2)
        for (int n : {p, p + p / 4, p + p / 2})
            if (n <= (n <= 32 ? ny / 2 : ny / 8)) chunks(n);
    for (int t = 16; t <= 512 && t <= ny; t *= 2) chunks((ny + t - 1) / t);
    std::sort(th.begin(), th.end(), std::greater<int>());
    th.erase(std::unique(th.begin(), th.end()), th.end());
    return th;
}

}  // namespace iewpf
