"""Solid statistics with 8, 4, 2 and 1 CTAs per solid (the count follows the
number of solids) against the oracle, and the det F ones against the field:
every column, with touching pairs whose contact tiles the CTAs share.
"""
import numpy as np
import pytest

import oracle
import scenarios

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_12696_gb300 import build
    build.build()
    oracle.build()


@pytest.mark.parametrize("count", [1, 38, 39, 77, 153])
def test_stats_match_the_oracle(count):
    import paper_2402_12696_gb300 as pkg
    cols = 8
    rows = (count + 2 * cols - 1) // (2 * cols)
    sc = scenarios.fluid_only(56 * cols, 40 * max(rows, 2), 0, 0, 0.8, force_kind=1, force_a=(2e-5, -1e-5))
    sc["solids"] = []
    for k in range(count):  # pairs 0.8 nodes apart
        pair, side = divmod(k, 2)
        sc["solids"].append({"x": 56.0 * (pair % cols) + 20.3 + 14.8 * side, "y": 40.0 * (pair // cols) + 20.1 + 0.2 * side,
                             "r": 7.0, "rho_s": 1.2, "G": 0.01})
    sim = pkg.Simulation(sc, precision="fp64")
    ref = oracle.Oracle(sc)
    sim.step(3)
    ref.step(3)
    st, o = sim.solid_stats(), np.array([ref.solid_stats(s) for s in range(count)])
    umax = float(np.hypot(ref.field("ux"), ref.field("uy")).max())
    scale = np.array([1.0, 1.0, 1.0, 1.0, umax, umax, 0.0, 0.0, 1.0, 1.0]) + np.abs(o)
    scale[:, 8:10] = max(np.abs(o[:, 8:10]).max(), 1e-300)
    rest = [0, 1, 2, 3, 4, 5, 8, 9]
    assert (np.abs(st - o) <= 1e-8 * scale)[:, rest].all(), np.abs(st - o).max(axis=0)
    # det F - 1 against the field of the same state: O(1) products of the same coordinate
    # differences, so a few units of 2^-52 apart
    for s in sorted({0, count // 2, count - 1}):
        phi, dev = sim.field_host("phi", s), np.abs(sim.field_host("detF_dev", s))
        m = np.isfinite(phi) & np.isfinite(dev)
        m[m] = phi[m] < -1e-9
        p = np.minimum(phi[m] / sc["eps"], 1.0)
        lam = np.where(p <= -1, 1.0, 1 - 0.5 * (1 + p + np.sin(np.pi * p) / np.pi))
        assert abs(st[s, 6] - dev[m].max()) <= 1e-13, s
        assert abs(st[s, 7] - (lam * dev[m]).sum() / lam.sum()) <= 1e-13, s
    if count > 1:
        assert np.abs(o[:, 8:10]).max() > 0.0
    ref.close()
    sim.close()
