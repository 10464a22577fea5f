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


def test_many_points_at_a_node(cuda_lib):
    """Every surface node of a ragged grid several times and one node 300 times,
    in mixed order, two shots with different multiplicities: adjoint against the
    oracle, and a repeated call bit for bit."""
    w = wl.small_3d(nx=70, ny=19, nz=21, nt=30, order=8, nshots=2)
    rng = np.random.default_rng(11)
    surf = np.arange(w.nx * w.ny)
    rec = np.stack([rng.permutation(np.concatenate([surf, surf, surf, np.full(300, 2 * w.nx * w.ny + 67)])),
                    rng.permutation(np.concatenate([np.repeat(surf[:400], 10), surf[:290]]))]).astype(np.int64)
    w = dataclasses.replace(w, rec=rec)
    s = wl.synthetic_data(2, w.nt, rec.shape[1], seed=9)
    p = problem(w)
    q = host(p.adjoint(to_dev(w.vel0), to_dev(s)))
    for k in range(2):
        assert rel_l2(q[k], oracle.adjoint(oracle.grid_of(w), w.src[k], w.rec[k], w.vel0, s[k])) <= 1e-5, k
    assert np.array_equal(q, host(p.adjoint(to_dev(w.vel0), to_dev(s))))


def test_time_of_doubled_receivers(cuda_lib):
    """Two receivers at every surface node take two additions a node, not a scan
    of all shared entries (250 times the call with one receiver a node)."""
    import torch

    def ms(times):
        w = wl.small_3d(nx=64, ny=64, nz=64, nt=40, order=8, nshots=1)
        w = dataclasses.replace(w, rec=np.tile(np.arange(64 * 64, dtype=np.int64), times)[None])
        p, v = problem(w), to_dev(w.vel0)
        s = to_dev(wl.synthetic_data(1, w.nt, w.rec.shape[1], seed=9))
        best = np.inf
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            p.adjoint(v, s)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    assert ms(2) <= 4 * ms(1)
