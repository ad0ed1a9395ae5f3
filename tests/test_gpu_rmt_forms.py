"""The two forms of the reference-map kernel (one CTA per solid; a cluster of
CTAs per solid, strips of rows) on the sizes where they can go wrong.

Both forms form every sum in the same order, so their fields agree bit for bit:
solids of a node or two (windows grown beyond 5x5, strips of two rows), solids at walls
(clipped bands) and across periodic edges, other shapes, many layers, and a disk whose layers
hold more nodes than the narrow form's list.  Tiny
disks are also held to the oracle, whose fits know neither form.
"""
import numpy as np
import pytest

import oracle
import scenarios
from parity_util import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_12696_gb300 import build
    build.build()
    oracle.build()


def _box(nx, ny, wx, wy, solids, **more):
    sc = scenarios.fluid_only(nx, ny, wx, wy, 0.8, force_kind=1, force_a=(2e-5, -1e-5))
    sc.update(more)
    sc["solids"] = [{"rho_s": 1.2, "G": 0.01, **s} for s in solids]
    return sc


def _disk(x, y, r):
    return {"x": x, "y": y, "r": r}


CASES = {
    "tiny": lambda: _box(96, 80, 0, 0, [_disk(30.3, 40.2, 1.0), _disk(70.6, 20.1, 1.4), _disk(60.2, 61.7, 2.3)]),
    "at_walls": lambda: _box(90, 100, 1, 1, [_disk(7.2, 8.1, 5.0), _disk(82.5, 92.4, 5.5), _disk(45.0, 6.3, 4.0)]),
    "across_edges": lambda: _box(131, 118, 0, 0, [_disk(0.4, 117.3, 14.0), _disk(66.0, 58.5, 20.0)]),
    "shapes": lambda: scenarios.shapes_small(1),
    "twenty_layers": lambda: _box(120, 130, 0, 1, [_disk(60.2, 65.3, 9.0)], n_layers=20),
    "wide_margin": lambda: _box(200, 190, 0, 1, [_disk(100.2, 95.3, 8.0)], deform_margin=4.0),
    "one_cta_each": lambda: _box(512, 500, 0, 1, [_disk(25.3 + 51 * (k % 10), 25.2 + 50 * (k // 10), 12.0 + 0.07 * k)
                                                  for k in range(100)]),
    "long_layers": lambda: _box(430, 440, 1, 1, [_disk(214.3, 220.4, 170.0)], deform_margin=0.05),
}


def _run(sc, prec, threads, steps):
    import paper_2402_12696_gb300 as pkg
    sim = pkg.Simulation(sc, precision=prec, rmt_threads=threads)
    sim.step(steps)
    sim.sync()
    out = [sim.field_host(f) for f in ("rho", "ux", "uy", "Fx", "Fy", "drho")]
    for s in range(len(sc["solids"])):
        out += [sim.field_host(f, s) for f in ("xi_x", "xi_y", "phi")]
    out.append(sim.solid_stats())
    sim.close()
    return out


@pytest.mark.parametrize("prec", ["fp32", "fp64", "fp16"])
@pytest.mark.parametrize("case", list(CASES))
def test_forms_bit_identical(case, prec):
    sc = CASES[case]()
    narrow = _run(sc, prec, 256, 7)
    wide = _run(sc, prec, 0, 7)  # few solids: the wide form
    for a, b in zip(narrow, wide):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("threads", [0, 256])
@pytest.mark.parametrize("case", ["tiny", "at_walls", "twenty_layers"])
def test_forms_match_oracle(case, threads):
    import paper_2402_12696_gb300 as pkg
    sc = CASES[case]()
    sim = pkg.Simulation(sc, precision="fp64", rmt_threads=threads)
    ref = oracle.Oracle(sc)
    sim.step(7)
    ref.step(7)
    r = compare(sim, ref, sc)
    for k in ("rho", "u", "xi", "F", "drho"):
        assert r[k] < 1e-8, (k, r)  # the FP64 bound of every parity case
    sim.close()
    ref.close()
