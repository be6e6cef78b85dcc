"""Host rules that choose the sweep kernel of a launch, from the library's own
header in a small program: which batches run one block per bundle."""
import shutil
import subprocess

import pytest

from conftest import ROOT
from test_gpu_wide import PLANAR

SMS = 152

PROGRAM = r"""
#include <cstdio>
#include "plan.cuh"
using namespace surfmcmc;
// classes, chains per class, syndromes, scan, accepts -> bundles, thread budget
int main() {
    int K, R, scan, acc, at_once;
    long long n;
    while (scanf("%d %d %lld %d %d %d", &K, &R, &n, &scan, &acc, &at_once) == 6) {
        SweepParams sp;
        init_chains(sp, K * R, R, 0);
        sp.scan = scan;
        uint64_t dummy = 0;
        sp.accepts = acc ? &dummy : nullptr;
        sp.n_groups = 1;
        sp.grp[0].n_bundles = bundles_of(sp, n);
        printf("%lld %d\n", sp.grp[0].n_bundles, wide_batch(@SMS@, sp, at_once));
    }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not shutil.which(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cu").write_text(PROGRAM.replace("@SMS@", str(SMS)))
    subprocess.run([nvcc, "-std=c++17", "-I", f"{ROOT}/include", "-I", f"{ROOT}/paper_1302_2669_gb300/csrc", "-o",
                    str(d / "rules"), str(d / "rules.cu")], check=True)

    def ask(rows):
        text = "\n".join(" ".join(map(str, r)) for r in rows) + "\n"
        out = subprocess.run([str(d / "rules")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]

    return ask


def test_small_batch_tests_take_the_small_batch_kernel(rule):
    """The shapes that test_gpu_wide compares with the throughput kernel."""
    rows = [(4, R, n, 0, 0, 1) for _, R, n in PLANAR] + [(16, R, n, 0, 0, 1) for R, n in
                                                         ((1, 5), (4, 3), (1, 33), (2, 3), (4, 2))]
    rows += [(4, R, 5, 0, 0, 1) for R in (1, 4, 8)]
    assert all(threads > 0 for _, threads in rule(rows))


def test_limit_and_thread_budget(rule):
    # 4 x 4 chains: two syndromes to a bundle
    n = [1, 2 * SMS, 2 * SMS + 1, 4 * SMS, 4 * SMS + 1, 6 * SMS, 8 * SMS, 8 * SMS + 1]
    got = rule([(4, 4, k, 0, 0, 1) for k in n])
    assert [t for _, t in got] == [1024, 1024, 512, 512, 341, 341, 256, 0]
    # random scan, accept counts: never; several launches at the same time: all their bundles
    assert [t for _, t in rule([(4, 4, 2, 1, 0, 1), (4, 4, 2, 0, 1, 1), (4, 4, 2, 0, 0, 4 * SMS),
                                (4, 4, 2, 0, 0, 4 * SMS + 1)])] == [0, 0, 256, 0]


def test_full_batch_tests_take_the_throughput_kernel(rule):
    """The shapes of test_gpu_sweep_paths without fixed lanes."""
    assert [t for _, t in rule([(4, 4, 130, 0, 0, 20), (4, 4, 1500, 0, 0, 1), (4, 9, 1500, 0, 0, 1)])] == [0, 0, 0]
