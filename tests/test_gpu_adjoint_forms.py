"""The reverse kernels on the sizes where their work is split differently,
against central differences in FP64 (directional derivatives of the final
centroids with respect to the body force field and to one solid's density
ratio, which the discrete adjoint reproduces to the differencing error):
windows beyond 5x5 (a disk of a few nodes), a band of 20 layers, disks in
contact, disks across periodic edges, and a disk for each number of CTAs of a cluster from 16 to 1, down
to one CTA whose layers need several rounds.
"""
import numpy as np
import pytest

import scenarios

pytestmark = pytest.mark.gpu

T, K = 8, 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_12696_gb300 import build
    build.build()


def _scenario(n, r, count=1, pitch=0.0, at=(), **more):
    sc = scenarios.adjoint_ldc(n, r=r, G=0.02, rho_ratio=1.3, body=scenarios.smooth_body_field(1, n, amp=2e-5))
    sc.update(more)
    if count > 1:
        one, per = sc["solids"][0], int((n - 8) // pitch)
        # (centres off the nodes: a node on the interface would change sides under the differences)
        sc["solids"] = [{**one, "x": 4.13 + pitch * (k % per + 0.5) + 0.1 * (k % 3), "y": 4.37 + pitch * (k // per + 0.5)}
                        for k in range(count)]
    if at:
        sc["solids"] = [{**sc["solids"][0], "x": x, "y": y} for x, y in at]
    return sc


CASES = {
    "few_nodes": lambda: _scenario(48, 1.7),
    "twenty_layers": lambda: _scenario(96, 9.0, n_layers=20),
    "contact": lambda: _scenario(96, 9.0, count=4, pitch=18.6),
    "across_edges": lambda: _scenario(96, 11.0, at=[(0.43, 95.63), (50.33, 0.71)], wall_x=0, wall_y=0, lid_u=0.0),
    "cluster_16": lambda: _scenario(192, 40.0),
    "cluster_8": lambda: _scenario(192, 20.0, count=9, pitch=61.0),
    "cluster_4": lambda: _scenario(160, 8.0, count=20, pitch=30.0),
    "cluster_2": lambda: _scenario(256, 8.0, count=60, pitch=30.0),
    "cluster_1": lambda: _scenario(288, 9.0, count=80, pitch=30.0),
}


@pytest.mark.parametrize("tile_x", [32, 128])
@pytest.mark.parametrize("case", list(CASES))
def test_adjoint_matches_central_differences(case, tile_x):
    import paper_2402_12696_gb300 as pkg
    sc = CASES[case]()
    n, S = sc["nx"], len(sc["solids"])
    w = np.random.default_rng(3).uniform(-1, 1, (S, 2))
    sim = pkg.Simulation(sc, precision="fp64", tile_x=tile_x)
    body = sc["body_field"]
    sim.forward_checkpointed(T, K)
    _, dr, db = sim.backward(w, body=True)
    db = db.cpu().numpy()
    # differences of the centroids from the unperturbed ones keep the loss small
    c0 = sim.forward_checkpointed(T, K)

    def loss(b, ratio=None):
        sim.set_body_force_field(b)
        sim.set_solid_params(S - 1, (1.3 if ratio is None else ratio) * sc["rho_f"], 0.02)
        return float((w * (sim.forward_checkpointed(T, K) - c0)).sum())

    v = scenarios.smooth_body_field(7, n, amp=1.0)
    fd = (loss(body + 1e-6 * v) - loss(body - 1e-6 * v)) / 2e-6
    # the largest directional derivative there is, as the scale of what may cancel in the sum
    scale = float(np.abs(db * v).sum())
    assert abs((db * v).sum() - fd) <= 1e-5 * scale, ((db * v).sum(), fd, scale)
    h = 1e-4 * 1.3
    fd = (loss(body, 1.3 + h) - loss(body, 1.3 - h)) / (2 * h)
    assert abs(dr[S - 1] - fd) <= 1e-4 * max(abs(fd), np.abs(dr).max()), (dr[S - 1], fd)
    sim.close()
