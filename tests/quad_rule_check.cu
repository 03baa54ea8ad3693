// Host check of the rule for four threads per item (quad_sweeps): a mesh alone takes them by its own warps, one of
// several swept side by side by the warps of all.  Counted here from the item counts themselves.
#include <cstdio>
#include "dfgks_bodies.cuh"
using namespace dfk;

static Mesh mesh(int nx, int ny) {
    Mesh m{};
    m.nx = nx; m.ny = ny;
    return m;
}
static long long up32(long long n) { return (n + 31) / 32; }

int main() {
    int bad = 0, both[2] = {0, 0};
    for (int nx = 1; nx <= 160; nx += 3)
        for (int ny = 1; ny <= 160; ny += 7)
            for (int beside = 1; beside <= 8; ++beside) {
                const long long lines = up32((nx + 1LL) * (ny + 4)) + up32((nx + 4LL) * (ny + 1));
                const long long sides = 2 * (up32((nx + 1LL) * ny) + up32(nx * (ny + 1LL)));
                const QuadSweeps q = quad_sweeps(mesh(nx, ny), beside);
                bad += q.lines != (lines * beside <= 304);
                bad += q.faces != (sides * beside <= 456);
                ++both[q.lines];
            }
    const QuadSweeps alone = quad_sweeps(mesh(59, 59), 1), eight = quad_sweeps(mesh(60, 60), 8), large = quad_sweeps(mesh(8192, 8192), 8);
    bad += !(alone.lines && alone.faces) + (eight.lines || eight.faces) + (large.lines || large.faces) + !(both[0] && both[1]);
    std::printf("%d wrong\n", bad);
    return bad ? 1 : 0;
}
