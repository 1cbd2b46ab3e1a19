"""Split of a step's delivery into items where row lengths differ.

The host build of the split: four parts per row unless the average row is
long, whatever the longest one is; item counts beyond 2^31; parts that cover
each row once; hub rows told apart by length, at most 256 of them.  On the GPU
a network of short rows with one or several inputs onto (nearly) every neuron
is compared with the oracle, with and without carried traces staged.
"""
from __future__ import annotations

import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "delivery_split.h"
using namespace eprop;
int main() {
    // (synapses, source rows) and the parts a row may have
    const long long hub1 = 100 * 300000LL + 300000, hub2 = 20 * 1000000LL + 1000000;
    printf("%d %d %d %d %d %d\n", delivery_part_shift(hub1, 300001), delivery_part_shift(hub2, 1000001),
           delivery_part_shift(0, 0), delivery_part_shift(1000LL * 1000000, 1000000),
           delivery_part_shift(10100LL * 128000, 129000), delivery_part_shift(1LL << 43, 1 << 23));
    const int rows = (1 << 24) - 1;
    long long bad = delivery_items(rows, 10) != 17179868160LL;
    const long long lens[] = {0, 1, 5, 1023, 1024, 100003, 16777215};
    for (long long len : lens)
        for (int ps = 2; ps <= 10; ++ps) {
            long long at = 0;
            for (int p = 0; p < 1 << ps; ++p) {
                if (delivery_part_begin(len, p, ps) != at) ++bad;
                at = delivery_part_begin(len, p + 1, ps);
            }
            if (at != len) ++bad;
        }
    // 300 rows of 5000 + i among rows of 10: the longest 256 are hubs; 40 of
    // them: all; rows of 4096 exactly: none
    std::vector<long long> many(1, 0), few(1, 0), edge(1, 0);
    for (int i = 0; i < 1000; ++i) {
        many.push_back(many.back() + (i < 300 ? 5000 + i : 10));
        few.push_back(few.back() + (i < 40 ? 5000 + i : 10));
        edge.push_back(edge.back() + (i < 40 ? 4096 : 10));
    }
    printf("%lld %lld %lld %lld\n", bad, delivery_hub_length(many.data(), 1000, 2),
           delivery_hub_length(few.data(), 1000, 2), delivery_hub_length(edge.data(), 1000, 2));
}
"""


def test_split_follows_the_average_row_and_counts_in_64_bits(tmp_path):
    (tmp_path / "d.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2511_21674_gb300", "csrc"),
                    str(tmp_path / "d.cpp"), "-o", str(tmp_path / "d")], check=True)
    out = subprocess.run([str(tmp_path / "d")], check=True, capture_output=True, text=True).stdout.split()
    assert [int(x) for x in out[:6]] == [2, 2, 2, 2, 4, 10]
    assert [int(x) for x in out[6:]] == [0, 5043, 4096, 4096]


@pytest.mark.gpu
@pytest.mark.parametrize("n_in,trace_kernel", [(1, 1), (1, 3), (40, 1), (40, 3)])
def test_inputs_onto_every_neuron_among_short_rows(n_in, trace_kernel):
    from tests.test_gpu_parity import run_parity
    from workloads import configs as C
    n, T = 5000, 60
    W = C.million_sparse(n_rec=n, k_in=20, n_out=2, T=T, J=0.05, lr=1e-5, update_interval=20)
    W["spec"].n_in = n_in
    size = np.array([n if q == 0 else n - 17 * q for q in range(n_in)])      # hubs of several lengths
    ptr = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    W["ptr"] = np.concatenate([ptr[:-1], W["ptr"] + ptr[-1]])
    W["col"] = np.concatenate([np.arange(m, dtype=np.int32) for m in size] + [W["col"]])
    W["w"] = np.concatenate([np.full(ptr[-1], 0.05, np.float32), W["w"]])
    W["delay"] = np.concatenate([np.full(m, 1 + q % 5, np.uint8) for q, m in enumerate(size)] + [W["delay"]])
    x = (np.arange(T)[:, None] + 3 * np.arange(n_in)) % 7 == 0
    W["x_ptr"] = np.concatenate([[0], np.cumsum(x.sum(1))]).astype(np.int64)
    W["x_ids"] = np.nonzero(x)[1].astype(np.int32)
    rep = run_parity(W, gpu_kw=dict(trace_kernel=trace_kernel))
    assert rep["spikes"] > 100
    assert rep["events"] >= int((x * size).sum())
