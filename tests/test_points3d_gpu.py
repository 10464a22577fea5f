"""Sampling and injection inside the 3-D sweep against the FP64 oracle:
sources and receivers at the edges of the 64 x 16 columns, of 32-plane words
and of the grid, several at one node (more than 64 entries in one row), ragged
grids, one to many work items a CTA, every time form, the absorbing layer.

Tolerances are those of the parity tests: 1e-5 on traces, 1e-4 on gradients.
"""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2104_00794_gb300 import workloads as wl
from parity_util import host, oracle_dobs, problem, rel_l2, to_dev

pytestmark = pytest.mark.gpu

CASES = [  # nx, ny, nz, shots, order, sponge, form
    (65, 17, 33, 1, 8, 0, "levels"), (64, 16, 32, 2, 4, 0, "levels"), (130, 33, 12, 2, 8, 0, "increment"),
    (3, 5, 70, 1, 8, 0, "levels"), (67, 18, 9, 24, 4, 0, "levels"), (90, 31, 40, 1, 8, 6, "levels"),
    (70, 20, 2, 1, 4, 0, "increment"),
]


def scattered(w, seed):
    rng = np.random.default_rng(seed)
    edge = lambda n, at: [i for i in (0, 1, *at, n - 1) if i < n]
    xs, ys, zs = edge(w.nx, (3, 4, 63, 64, 65)), edge(w.ny, (15, 16, 17)), edge(w.nz, (7, 8, 31, 32))
    def pts(n):
        p = (rng.choice(zs, n) * w.ny + rng.choice(ys, n)) * w.nx + rng.choice(xs, n)
        p[n // 2] = p[0]
        return p
    row = np.tile(np.arange(min(w.nx, 70)), 2)  # two receivers at every node of a row's start
    src = np.stack([pts(6) for _ in range(w.nshots)]).astype(np.int64)
    rec = np.stack([np.concatenate([pts(50), row]) for _ in range(w.nshots)]).astype(np.int64)
    wav = np.ascontiguousarray(np.repeat(w.wavelet, 6, axis=2) * np.array([1, .5, -.7, .3, .9, -.2], np.float32))
    return dataclasses.replace(w, src=src, rec=rec, wavelet=wav)


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_against_oracle(cuda_lib, case):
    nx, ny, nz, shots, order, sponge, form = case
    w = scattered(wl.small_3d(nx=nx, ny=ny, nz=nz, nt=40, order=order, nshots=shots), 5)
    if sponge:
        w = wl.with_sponge(w, sponge)
    g = oracle.grid_of(w)
    p = problem(w, form=form)
    d = host(p.forward(to_dev(w.vel_true), to_dev(w.wavelet)))
    assert rel_l2(d, oracle.batch_forward(w, w.vel_true)) <= 1e-5
    s = wl.synthetic_data(w.nshots, w.nt, w.rec.shape[1], seed=9)
    q = host(p.adjoint(to_dev(w.vel0), to_dev(s)))
    for k in range(w.nshots):
        assert rel_l2(q[k], oracle.adjoint(g, w.src[k], w.rec[k], w.vel0, s[k])) <= 1e-5, k
    if not sponge:
        dobs = oracle_dobs(w)
        gf = host(p.gradient_full(to_dev(w.vel0), to_dev(w.wavelet), to_dev(dobs))[0])
        assert rel_l2(gf, oracle.batch_gradient_full(w, w.vel0, dobs)[0]) <= 1e-4
