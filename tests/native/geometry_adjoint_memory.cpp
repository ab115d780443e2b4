// Host memory of geometry_adjoint: prints the bytes that one call allocates on a quad mesh of argv[1] x
// argv[1] cells with walls all round ("bytes <n>"), and a checksum of its result ("sum <value>").
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>

#include "fvlbm_internal.h"

using namespace fvlbm;

static std::atomic<size_t> g_bytes{0};
void *operator new(size_t n) {
    g_bytes += n;
    void *p = std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

int main(int argc, char **argv) {
    if (argc < 2) return 2;
    const int n = std::atoi(argv[1]);
    std::vector<double> xy;
    std::vector<int> ptr(1, 0), cn, bn, bt;
    auto node = [&](int i, int j) { return j * (n + 1) + i; };
    for (int j = 0; j <= n; ++j)
        for (int i = 0; i <= n; ++i) {
            xy.push_back(i + 0.1 * ((7 * i + 3 * j) % 5));
            xy.push_back(j + 0.1 * ((3 * i + 5 * j) % 4));
        }
    for (int j = 0; j < n; ++j)
        for (int i = 0; i < n; ++i) {
            for (int a : {node(i, j), node(i + 1, j), node(i + 1, j + 1), node(i, j + 1)}) cn.push_back(a);
            ptr.push_back(static_cast<int>(cn.size()));
        }
    auto edge = [&](int a, int b) {
        bn.push_back(a);
        bn.push_back(b);
        bt.push_back(FVLBM_BC_WALL);
    };
    for (int i = 0; i < n; ++i) {
        edge(node(i, 0), node(i + 1, 0));
        edge(node(n, i), node(n, i + 1));
        edge(node(i + 1, n), node(i, n));
        edge(node(0, i + 1), node(0, i));
    }
    const size_t nc = ptr.size() - 1, nbe = bt.size();
    std::vector<double> bv(5 * nbe, 0.0);
    fvlbm_mesh M{(n + 1) * (n + 1), xy.data(), static_cast<int>(nc), ptr.data(), cn.data()};
    fvlbm_bc B{static_cast<int>(nbe), bn.data(), bt.data(), bv.data(), 0, nullptr, nullptr};
    GeometryAdjoint A;
    auto fill = [](std::vector<double> &v, size_t k) {
        v.resize(k);
        for (size_t q = 0; q < k; ++q) v[q] = 0.25 + static_cast<double>((q * 37) % 101) / 101.0;
    };
    for (auto *v : {&A.sn, &A.lsq, &A.rown, &A.rnbr}) fill(*v, 8 * nc);
    fill(A.dinv, 4 * nc);
    fill(A.wdist, nc);
    fill(A.area, nc);
    fill(A.bnrm, 2 * nbe);
    fill(A.blen, nbe);
    std::vector<double> g(xy.size());
    std::string why;
    const size_t before = g_bytes;
    if (geometry_adjoint(M, B, A, g.data(), &why)) return 5;
    const size_t used = g_bytes - before;
    double sum = 0.0;
    for (size_t k = 0; k < g.size(); ++k) sum += g[k] * (1.0 + 1e-3 * static_cast<double>(k % 17));
    std::printf("bytes %zu\nsum %.17g\n", used, sum);
    return 0;
}
