"""The overlapped step with tensor-memory loads (large FP32-arithmetic grids):
the busy regions' tiles go through the staged kernel, the free regions through
the direct-load kernel.  Fields agree bit for bit with the sequential staged
step and with the direct-load overlapped one, on full and on ragged tiles.
"""
import numpy as np
import pytest

import scenarios

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2402_12696_gb300 import build
    build.build()


def _scenario(nx, ny, walls):
    sc = scenarios.fluid_only(nx, ny, walls, walls, 0.8, force_kind=1, force_a=(2e-5, -1e-5))
    rng = np.random.default_rng(5)
    sc["solids"] = [{"rho_s": 1.2, "G": 0.01, "x": 64.0 * i + 40 + rng.uniform(-4, 4),
                     "y": 64.0 * j + 40 + rng.uniform(-4, 4), "r": float(rng.uniform(2, 14))}
                    for i in range(0, nx // 64, 5) for j in range(ny // 64)]
    return sc


@pytest.mark.parametrize("nx,ny,walls", [(2048, 2048, 0), (2056, 2043, 1)])
@pytest.mark.parametrize("prec", ["fp32", "fp16"])
@pytest.mark.parametrize("tile_x", [16, 32])
def test_staged_overlap_bit_identical(nx, ny, walls, prec, tile_x):
    import paper_2402_12696_gb300 as pkg
    sc = _scenario(nx, ny, walls)
    outs = []
    for tma, ov in ((True, True), (True, False), (False, True)):
        sim = pkg.Simulation(sc, precision=prec, use_tma=tma, overlap=ov, tile_x=tile_x)
        sim.step(23)  # one 20-step graph, one 2-step graph, one direct step
        sim.sync()
        assert sim.uses_tma == tma
        assert sim.uses_overlap == (ov and (not tma or nx * ny >= 1 << 22))
        outs.append([sim.field_host(n) for n in ("rho", "ux", "uy", "Fx", "drho")] +
                    [sim.field_host("xi_x", s) for s in (0, len(sc["solids"]) - 1)])
        sim.close()
    for o in outs[1:]:
        for a, b in zip(outs[0], o):
            assert np.array_equal(a, b, equal_nan=True)
