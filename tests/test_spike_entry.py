"""Spike entries of the batched single-window gradient at long windows.

The kernel lists a row's spikes as 32-bit entries and decodes each into a row
of the window tables.  The host build of the same functions must give the row
b U + step + d - 1, and tell arrivals past the window, over every sample, word
and bit position a list can hold: windows beyond 2^20 steps, many samples, and
the last word one base serves.  On the GPU a window of more than 2^20 steps is
compared with the eligibility recursion in 64 bits (Eq. eligibility-vector-
substituted, Eq. final-gradient).
"""
from __future__ import annotations

import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "spike_entry.h"
using namespace eprop;
int main(int argc, char **argv) {
    const int B = atoi(argv[1]), T = atoi(argv[2]), U = T, wps = T / 32 + 1;
    const long long words = (long long)B * wps;
    long long checked = 0, bad = 0;
    // lists that begin at the first word, in the middle and near the end
    const long long firsts[4] = {0, words / 3, words / 2 + 1, words - 1};
    for (long long w0 : firsts) {
        const long long base = entry_base((int)(w0 / wps), (int)(w0 % wps), U);
        const long long end = words - w0 < kEntrySpan ? words : w0 + kEntrySpan;
        const long long stride = (end - w0) / 4000 + 1;
        for (long long w = w0; w < end; w = w + stride < end || w == end - 1 ? w + stride : end - 1) {
            const int b = (int)(w / wps), k = (int)(w % wps);
            for (int bit = 0; bit < 32; ++bit) {
                const int step = k * 32 + bit;
                if (step < 1 || step > T) continue;
                const unsigned e = entry_pack(base, b, step, U, T);
                for (int d = 1; d <= 8; ++d) {
                    ++checked;
                    if (entry_arrives(e, d) != (step + d <= T)) ++bad;
                    else if (step + d <= T && entry_row(base, e, d) != (long long)b * U + step + d - 1) ++bad;
                }
            }
        }
    }
    printf("%lld %lld\n", checked, bad);
}
"""


@pytest.fixture(scope="module")
def decoder(tmp_path_factory):
    d = tmp_path_factory.mktemp("entry")
    (d / "e.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2511_21674_gb300", "csrc"),
                    str(d / "e.cpp"), "-o", str(d / "e")], check=True)
    return str(d / "e")


@pytest.mark.parametrize("B,T", [(1, 1), (1, 31), (3, 32), (64, 350), (2047, 1000), (1, (1 << 20) + 37),
                                 (2, 1 << 20), (2047, 1 << 21), (1, (1 << 28) + 100), (7, (1 << 28) - 1)])
def test_entries_decode_to_their_table_rows(decoder, B, T):
    checked, bad = map(int, subprocess.run([decoder, str(B), str(T)], check=True, capture_output=True,
                                           text=True).stdout.split())
    assert checked > 0 or T == 1
    assert bad == 0


@pytest.mark.gpu
@pytest.mark.parametrize("B", [1, 2])
def test_gradient_of_a_window_beyond_2_to_20_steps(B):
    from scipy.signal import lfilter
    import paper_2511_21674_gb300 as ep
    from workloads import configs as C
    T, n, d = (1 << 20) + 37, 3, 5
    rng = np.random.default_rng(B)
    s = C.Spec(name="long", n_in=1, n_rec=n, n_out=1, T=T, batch=B, feedback=1, lr=1e-9, max_delay=d)
    x = rng.random((B, T)) < 0.02
    x[:, -20:] = [True, False] * 10              # arrivals inside and past the end
    x_ptr = np.concatenate([[0], np.cumsum(x.ravel())]).astype(np.int64)
    w = np.array([0.7, 0.3, 0.9], np.float32)
    fb = np.array([[1.0], [-0.5], [0.25]], np.float32)
    tg = rng.standard_normal((B, T, 1)).astype(np.float32)
    net = ep.Network(s, np.array([0, n, n, n, n], np.int64), np.arange(n, dtype=np.int32), w,
                     np.array([1, 2, d], np.uint8), np.full((n, 1), 0.1, np.float32), None, fb,
                     record_grad=1, record_psi=1, launch_mode=0)
    net.set_inputs(x_ptr, np.zeros(int(x.sum()), np.int32), tg, np.ones((B, T), np.uint8),
                   np.full(B, T, np.int32), T)
    net.simulate(T)
    y, _ = net.readout()
    psi = net.surrogate().astype(np.float64)
    w_new, g = net.weights(ep.PROJ_IN, with_grad=True)
    net.close()
    alpha, kappa = np.exp(-s.dt / s.tau_m), np.exp(-s.dt / s.tau_out)
    E = y[..., 0].astype(np.float64) - tg[..., 0]
    for j, dl in enumerate((1, 2, d)):
        G = mag = 0.0
        for b in range(B):
            z = np.concatenate([np.zeros(dl), x[b, :-dl]]).astype(np.float64)
            ebar = lfilter([1.0], [1.0, -kappa], psi[b, :, j] * lfilter([1.0], [1.0, -alpha], z))
            G += float(fb[j, 0]) * (E[b] @ ebar)
            mag += abs(float(fb[j, 0])) * (np.abs(E[b]) @ np.abs(ebar))
        # FP32 terms summed to at least FP32 accuracy per sample and window
        assert abs(g[j] - G / B) <= 1e-5 * mag / B, (j, g[j], G / B, mag / B)
        assert abs(w_new[j] - (w[j] - s.lr * G / B)) <= 1e-5 * s.lr * mag / B + 2 ** -24
