"""The FP64 force kernel takes a tile in four, two or one parts, by how many tiles there are: fields bit for
bit those of the same scenario as a batch member, whose force kernel takes whole tiles.
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


@pytest.mark.parametrize("tile_x", [16, 32, 64, 128])
@pytest.mark.parametrize("count", [2, 9, 64])
def test_parts_match_whole_tiles(count, tile_x):
    import paper_2402_12696_gb300 as pkg
    per = int(np.ceil(np.sqrt(count)))
    sc = scenarios.fluid_only(40 * per + 29, 40 * per + 13, 0, 1, 0.8, force_kind=1, force_a=(2e-5, -1e-5))
    # pairs in contact across the rows of a tile, and ragged edges of the grid
    sc["solids"] = [{"x": 40.0 * (k % per) + 20.3, "y": 40.0 * (k // per) + 12.2 + 5.9 * (k % 2), "r": 8.0 + 0.4 * (k % 5),
                     "rho_s": 1.2, "G": 0.01} for k in range(count)]
    if count > 2:
        sc["solids"][1].update(x=sc["solids"][0]["x"] + 1.0, y=sc["solids"][0]["y"] + 16.9)
    sim, batch = pkg.Simulation(sc, precision="fp64", tile_x=tile_x), pkg.Batch([sc], precision="fp64", tile_x=[tile_x])
    sim.step(11)
    batch.step(11)
    batch.sync()
    for f in ("Fx", "Fy", "drho", "rho", "ux", "uy"):
        assert np.array_equal(sim.field_host(f), batch[0].field_host(f), equal_nan=True), f
    sim.close()
    batch.close()
