"""Sizes of the message encoder's scratch, compiled for the host alone: what is accepted fits, whatever the shape of the data."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Bounds of the graph network on a hub graph of n nodes (in- and out-degree n - 1 at one of them, 2 (n - 1) edges), as the library infers them.
PROGRAM = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <cstdlib>
#include "wave_sizes.h"
using namespace amp;
int main(int argc, char** argv) {
  for (int a = 1; a < argc; a++) {
    const int n = atoi(argv[a]), edges = 2 * (n - 1), degree = n - 1;
    std::vector<DevNode> nodes;
    auto node = [&](int type, int ppt, int fn_arg, int ui, int ri, int uo, int ro) {
      DevNode h{};
      h.type = type; h.ppt = ppt; h.fn_arg = fn_arg; h.n_pred = h.n_succ = 1; h.U_in = ui; h.rows_in = ri; h.U_out = uo; h.rows_out = ro;
      nodes.push_back(h);
    };
    node(LOOKUP, 0, 0, 1, n, 1, n);
    node(UNGROUP, -1, 0, 1, n, n, 1);
    node(FLATMAP, -1, 0, n, 1, edges, 1);
    node(GROUP, -1, 0, edges, 1, 4, edges);
    node(LINEAR, 1, 0, 4, edges, 4, edges);
    node(GROUP, -1, 0, edges, 1, n, degree);
    node(NPT_SUMROWS, -1, 0, n, degree, n, 1);
    wave::EncModel E{};
    E.n_nodes = (int)nodes.size(); E.n_ppts = 2; E.IT = 5;
    E.ppts[0].node = 0; E.ppts[1].node = 4;
    for (auto& P : {&E.ppts[0], &E.ppts[1]}) for (int k = 0; k < 6; k++) P->cell[k] = -1;
    const bool ok = wave::encoder_sizes(E, nodes, degree);
    unsigned long long keys = 0;                       // references and counters alone, in full width
    const unsigned long long N = n, D = edges, G = degree;
    keys = 5 * (1 * N + N * G + 4 * D + N * G + 1 + N + 4 + N + N);
    printf("%d %d %llu %u %u %u\n", n, (int)ok, keys, E.table_words, E.row_cap, E.scratch_words);
  }
}
"""


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    d = tmp_path_factory.mktemp("sizes")
    (d / "sizes.cpp").write_text(PROGRAM)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "paper_1705_09786_b200", "csrc"),
                           str(d / "sizes.cpp"), "-o", str(d / "sizes")])

    def run(ns):
        out = subprocess.check_output([str(d / "sizes")] + [str(n) for n in ns], text=True)
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    return run


def test_hub_graphs_beyond_the_scratch_limit_are_refused_at_every_size(sizes):
    rows = sizes(list(range(16, 2000, 31)) + list(range(2000, 16001, 7)))
    accepted = [ok for _, ok, *_ in rows]
    assert accepted[0] == 1 and accepted[-1] == 0
    assert accepted == sorted(accepted, reverse=True)               # refused once, refused for every larger graph
    for n, ok, keys, table, row_cap, words in rows:
        if ok:
            assert keys <= table < words <= 1 << 28 and row_cap >= 5 * n * (n - 1), n
        else:
            assert n > 500                                          # (graphs of some hundred nodes stay with the encoder)
