// Host-side probe of the planner (tests/test_planner.py): reads lists as "l K bra-pairs ket-pairs flags jk"
// (l < 0: shells of every l; K < 0: of degrees 1 to -K)
// and prints, for each, the number of chunks of the plan at the workspace size, at half of it and at
// the smallest workspace, the return code one byte below the smallest, and whether each chunk's layout
// lies within its workspace.  No device is used.
#include <cstdio>

#include "lx_api.cu"

int main() {
    int l, K, nb, nk, flags, jk;
    while (std::scanf("%d %d %d %d %d %d", &l, &K, &nb, &nk, &flags, &jk) == 6) {
        std::vector<lx_shell> sh(2 * (nb + nk));
        int nprim = 0;
        for (size_t s = 0; s < sh.size(); ++s) {
            sh[s] = lx_shell{};
            sh[s].l = l >= 0 ? l : 3 * (int)s % 8;
            sh[s].nprim = K > 0 ? K : 1 + 5 * (int)s % -K;
            sh[s].prim_offset = nprim;
            nprim += sh[s].nprim;
        }
        const std::vector<double> one(nprim, 1.0);
        std::vector<lx_quartet> q;
        for (int i = 0; i < nb; ++i)
            for (int j = 0; j < nk; ++j) q.push_back({{2 * i, 2 * i + 1, 2 * (nb + j), 2 * (nb + j) + 1}, 0});
        const int32_t n = (int32_t)sh.size();
        const int64_t nq = (int64_t)q.size();
        const int64_t size = workspace_need(sh.data(), n, q.data(), nq, flags, jk ? JK_DIGEST : 0, false);
        const int64_t least = workspace_need(sh.data(), n, q.data(), nq, flags, jk ? JK_DIGEST : 0, true);
        bool fits = true;
        auto chunks = [&](int64_t bytes) {
            PlannedBatch B;
            const int v = plan_batch(sh.data(), n, one.data(), one.data(), (int)one.size(), q.data(), nq,
                                     flags | (jk ? JK_DIGEST : 0), (size_t)bytes, Overrides(), B);
            if (v != LX_OK) return v;
            for (const ChunkPlan& P : B.chunks) fits = fits && B.head + P.total <= (size_t)bytes;
            return (int)B.chunks.size();
        };
        const int a = chunks(size), b = chunks(std::max(least, size / 2)), c = chunks(least), d = chunks(least - 1);
        std::printf("%d %d %d %d %d\n", a, b, c, d, fits ? 1 : 0);
    }
}
