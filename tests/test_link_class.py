"""The class that decides a link (link_class in csrc/lbm_aux.cuh), against a search written from its rule, over
every node and direction of small random lattices with every boundary kind, cuts and halo classes (CPU: the
function also compiles for the host)."""
import subprocess

from paper_1802_07525_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "lbm_aux.cuh"
using namespace mfc;

// Walls win over inlet and outlet; periodic sources wrap; the outlet's is the last layer; beyond a cut the halo's.
template <int D> int rule(const MaskArgs &m, const int (&p)[3], const int (&c)[3])
{
    const int n[3] = {m.geo.nx, m.geo.ny, m.geo.nz}, fa = D == 2 ? 0 : 2;
    int s[3], beyond = -1;
    for (int a = 0; a < 3; ++a) s[a] = p[a] - c[a];
    if (s[fa] < 0 && m.cut[0]) beyond = 0;
    if (s[fa] >= n[fa] && m.cut[1]) beyond = 1;
    bool inlet = false;
    for (int a = 0; a < D; ++a) {
        if ((s[a] >= 0 && s[a] < n[a]) || (a == fa && beyond >= 0)) continue;
        if (m.bc[a] == BC_WALL || (m.bc[a] == BC_INOUT && a != fa)) return CLS_FLOW | CLS_ADE;
        if (m.bc[a] == BC_PERIODIC) s[a] = (s[a] + n[a]) % n[a];
        else if (s[a] < 0) inlet = true;
        else s[a] = n[a] - 1;
    }
    if (inlet) return 0;
    if (beyond >= 0) return m.halo_cls[beyond] ? m.halo_cls[beyond][D == 2 ? s[1] : s[0] + n[0] * s[1]] : 0;
    return m.cls_new[s[0] + n[0] * (s[1] + n[1] * s[2])];
}

template <int D> long run()
{
    long count = 0;
    for (int t = 0; t < 3000; ++t) {
        MaskArgs m = {};
        const int n[3] = {1 + rand() % 5, 1 + rand() % 5, D == 3 ? 1 + rand() % 5 : 1}, fa = D == 2 ? 0 : 2;
        m.geo.nx = n[0], m.geo.ny = n[1], m.geo.nz = n[2];
        for (int a = 0; a < 3; ++a) m.bc[a] = a == fa ? rand() % 3 : rand() % 2;
        for (int s = 0; s < 2; ++s) m.cut[s] = m.bc[fa] != BC_PERIODIC && rand() % 3 == 0;
        std::vector<uint8_t> cls(n[0] * n[1] * n[2]), halo[2];
        for (auto &v : cls) v = rand() % 8;
        m.cls_new = cls.data();
        for (int s = 0; s < 2; ++s) {
            halo[s].resize(D == 2 ? n[1] : n[0] * n[1]);
            for (auto &v : halo[s]) v = rand() % 8;
            m.halo_cls[s] = rand() % 2 ? halo[s].data() : nullptr;
        }
        for (long long q = 0; q < (long long)cls.size(); ++q) {
            const int p[3] = {(int)(q % n[0]), (int)(q / n[0] % n[1]), (int)(q / (n[0] * n[1]))};
            for (int i = 1; i < FlowSet<D>::Q; ++i) {
                const int c[3] = {FlowSet<D>::c(i, 0), FlowSet<D>::c(i, 1), FlowSet<D>::c(i, 2)};
                const int got = link_class<D>(m, q, p[0], p[1], p[2], c[0], c[1], c[2]), want = rule<D>(m, p, c);
                if ((got ^ want) & (CLS_FLOW | CLS_ADE)) {
                    printf("D%d node %lld direction %d: %d, not %d\n", D, q, i, got, want);
                    exit(1);
                }
                ++count;
            }
        }
    }
    return count;
}

int main()
{
    printf("same %ld\n", run<2>() + run<3>());
    return 0;
}
"""


def test_link_class_follows_its_rule(tmp_path):
    src, exe = tmp_path / "link_class.cu", tmp_path / "link_class"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), "-std=c++17", "-O1", "-I", build.CSRC, *build.ARCH, str(src), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("same"), r.stdout
