"""The lists of the H^2 tensor-core apply by pairs of outputs (h2_group_list,
csrc/h2_build.cpp), on the CPU: the product's own C++ compiled with g++ into a
small driver.  Random lists, with inputs that a list takes twice, an odd number
of outputs and an output without entries, and the apply's own lists: every
entry belongs to exactly one group entry, and every output meets its entries in
the list's order.  For the sphere sizes the GPU test of the pairs uses, the
rules say that the near field (and at 1024 directions the couplings) is taken
by pairs.
"""
import os
import subprocess

import pytest

from test_gpu_h2_pairs import CALLS, rows_for

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, 'paper_2102_09038_gb300', 'csrc')
CUDA_INC = '/usr/local/cuda/include'

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <string>
#include "h2.h"
#include "rte_internal.h"
namespace rte {
int fail(int c, const std::string& m) { std::fprintf(stderr, "%s\n", m.c_str()); return c; }
}
using namespace rte;
static void show(const char* name, const H2List& l, int G) {
    const H2List g = h2_group_list(l, G);
    auto row = [](const char* what, const std::vector<int>& v) {
        std::printf("%s", what);
        for (int x : v) std::printf(" %d", x);
        std::printf("\n");
    };
    std::printf("list %s %d %d\n", name, G, (int)h2_group_pays(l, g));
    row("out", l.out_blk); row("ptr", l.ptr); row("in", l.in_blk); row("mat", l.mat);
    row("gout", g.out_blk); row("gptr", g.ptr); row("gin", g.in_blk); row("gmat", g.mat);
}
int main(int argc, char** argv) {
    if (!std::strcmp(argv[1], "takes")) {
        std::printf("%d\n", (int)h2_takes_groups(std::atoi(argv[2]), std::atoi(argv[3]), std::atoi(argv[4])));
        return 0;
    }
    if (!std::strcmp(argv[1], "random")) {
        std::mt19937 rng(std::atoi(argv[2]));
        for (int nout : {1, 2, 5, 6})
            for (int inputs : {1, 3, 9})
                for (int empty = 0; empty < 2; ++empty) {
                    H2List l;
                    l.ptr.push_back(0);
                    for (int j = 0; j < nout; ++j) {
                        l.out_blk.push_back(100 + j);
                        const int n = empty && j == nout / 2 ? 0 : 1 + (int)(rng() % 7);
                        for (int e = 0; e < n; ++e) {
                            l.in_blk.push_back((int)(rng() % inputs));
                            l.mat.push_back((int)l.mat.size());
                        }
                        l.ptr.push_back((int)l.in_blk.size());
                    }
                    for (int G : {1, 2, 3}) show("random", l, G);
                }
        return 0;
    }
    const int levels = std::atoi(argv[2]), m = std::atoi(argv[3]);
    const SphereMesh S = make_sphere(levels);
    const int qf = 1 << (2 * kRFar);
    std::vector<double> fp((size_t)S.n * qf * 3), fw((size_t)S.n * qf);
    for (int t = 0; t < S.n; ++t) {
        int c = 0;
        quad_one(&S.verts[3 * S.tri[3 * t]], &S.verts[3 * S.tri[3 * t + 1]],
                 &S.verts[3 * S.tri[3 * t + 2]], kRFar, &fp[(size_t)t * qf * 3],
                 &fw[(size_t)t * qf], c);
    }
    H2Plan P;
    if (!h2_plan(levels, 1.4, 4, fp, qf, P)) return 2;
    H2Lists L;
    h2_lists(P, h2_pool(P, m), L);
    // the pool numbers the couplings by entry (the list holds the parts' signs)
    for (size_t e = 0; e < L.couple.mat.size(); ++e) L.couple.mat[e] = (int)e;
    show("near", L.near, 2);
    show("couple", L.couple, 2);
    show("down_leaf", L.down_leaf, 2);
    return 0;
}
"""


@pytest.fixture(scope='module')
def driver(tmp_path_factory):
    if not os.path.isdir(CUDA_INC):
        pytest.skip('CUDA headers not found')
    d = tmp_path_factory.mktemp('h2_groups')
    src = d / 'drv.cpp'
    src.write_text(DRIVER)
    exe = d / 'drv'
    subprocess.run(['g++', '-std=c++17', '-O1', '-ffp-contract=off', '-I', CSRC, '-I', CUDA_INC,
                    os.path.join(CSRC, 'h2_build.cpp'), os.path.join(CSRC, 'setup_host.cpp'),
                    str(src), '-o', str(exe)], check=True, capture_output=True)
    return str(exe)


def run(exe, *args):
    out = subprocess.run([exe] + [str(a) for a in args], check=True, capture_output=True, text=True)
    lists, cur = [], None
    for line in out.stdout.splitlines():
        w = line.split()
        if w[0] == 'list':
            cur = dict(name=w[1], G=int(w[2]), pays=w[3] == '1')
            lists.append(cur)
        elif cur is not None:
            cur[w[0]] = [int(x) for x in w[1:]]
    return lists


def check(l):
    G, nout = l['G'], len(l['out'])
    if any(a == b for a, b in zip(l['ptr'], l['ptr'][1:])):
        assert not l['gout'] and not l['gin'] and not l['pays']   # an output has no entries
        return
    groups = (nout + G - 1) // G
    assert len(l['gptr']) == groups + 1 and l['gptr'][0] == 0 and l['gptr'][-1] == len(l['gin'])
    assert len(l['gout']) == groups * G and len(l['gmat']) == len(l['gin']) * G
    for j in range(groups * G):
        assert l['gout'][j] == (l['out'][j] if j < nout else -1)
        got = [(l['gin'][e], l['gmat'][e * G + j % G])
               for e in range(l['gptr'][j // G], l['gptr'][j // G + 1])
               if l['gmat'][e * G + j % G] >= 0]
        a, b = (l['ptr'][j], l['ptr'][j + 1]) if j < nout else (0, 0)
        assert got == list(zip(l['in'][a:b], l['mat'][a:b]))
    # no group entry that no output takes
    assert all(any(x >= 0 for x in l['gmat'][e * G:(e + 1) * G]) for e in range(len(l['gin'])))


@pytest.mark.parametrize('seed', range(4))
def test_random_lists(driver, seed):
    lists = run(driver, 'random', seed)
    assert len(lists) == 4 * 3 * 2 * 3
    for l in lists:
        check(l)


@pytest.mark.parametrize('levels, parity, groups, paired', CALLS)
def test_lists_of_the_apply(driver, levels, parity, groups, paired):
    lists = {l['name']: l for l in run(driver, 'plan', levels, 1 if parity > 0 else 3)}
    for l in lists.values():
        check(l)
    assert {n for n in lists if lists[n]['pays']} == set(paired)
    # the GPU test's rows reach the pairs of each of these lists, and its
    # short calls do not
    for n in paired:
        g = len(lists[n]['gptr']) - 1
        assert g >= groups
        for sms in (132, 148, 152, 160):
            tiles = -(-rows_for(groups, sms) // 128)
            takes = lambda t: subprocess.run([driver, 'takes', str(g), str(t), str(sms)], check=True,
                                             capture_output=True, text=True).stdout.strip() == '1'
            assert takes(tiles) and not takes(1)
