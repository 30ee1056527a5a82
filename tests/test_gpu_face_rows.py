"""Rows next to y and z faces: their streaming folds wraps and specular reflections into row shifts.

Every population of every node against the FP64 oracle after one, two and three steps (each layout is read and
written), on boxes of three to nine rows with every pair of y and z faces (edges and corners
included), x faces wrapped or reflected, and rows of less than, exactly and more than one block.

Bounds, in units of the largest population: FP32 storage, a collision of fewer than 64 roundings on
the way to each population, 64 x 2^-24 a step; 16-bit storage, the 2e-3 of its budget
(tests/test_gpu_parity.py).  The fields carry an interface and a velocity of 0.02 that varies from node
to node, so a population taken from a wrong row or direction is off by more than 1e-2.
"""
import numpy as np
import pytest

import lbm_inputs as L
import oracle
import paper_1705_03141_gb300 as pkg

pytestmark = pytest.mark.gpu

SHAPES = [(32, 3, 4), (33, 6, 3), (70, 5, 9)]
XY = [(0, 0), (2, 2), (0, 2), (2, 0), (0, 1), (2, 1)]  # x and y faces: 0 periodic, 1 no-slip, 2 free slip
Z = [(0, 0), (2, 2), (1, 2), (3, 4), (2, 4)]           # z faces; 3 inflow wall, 4 outflow
STORAGES = [("f32", 1), ("f32", 3), ("f16", 1), ("c16", 1)]


@pytest.mark.parametrize("storage,variant", STORAGES)
@pytest.mark.parametrize("shape", SHAPES)
def test_face_rows_match_the_oracle(cuda, shape, storage, variant):
    for bx, by in XY:
        for z in Z:
            p = dict(L.parity_cases()[3 if z[0] == 3 else 1][1]["params"])
            p["bc"] = (bx, bx, by, by) + z
            if z[0] == 3:
                p["inflow"] = dict(p["inflow"], xc=0.5 * (shape[0] - 1), yc=0.5 * (shape[1] - 1), D=2.0)
            w = dict(name="faces", shape=shape, params=p, fields=("random_blobs", dict(seed=3, blobs=2)), steps=3)
            rr, rb, u = L.initial_fields(w, seed=4, u_amp=0.02)
            lat = pkg.Lattice(shape, p, storage=storage, variant=variant)
            lat.init_fields(rr, rb, u)
            orc = oracle.Oracle(shape, p)
            orc.init_fields(rr, rb, u)
            for n in (1, 2, 3):
                lat.step(1)
                orc.step(1)
                g = lat.get_populations()
                tol = (64 * n * 2.0 ** -24 if storage == "f32" else 2e-3) * np.max(orc.f)
                err = np.max(np.abs(g - orc.f))
                assert err < tol, (bx, by, z, n, err, tol)
            lat.close()


# more than two tiles along y and z, a ragged last block and none: the pipelined compact density pass, whose face
# rows read the colour records from global memory (x faces reflect; every pair of y and z faces)
@pytest.mark.parametrize("storage", ["c16", "cbf16"])
@pytest.mark.parametrize("shape", [(32, 9, 6), (45, 14, 7)])
def test_pipelined_compact_face_rows(cuda, shape, storage):
    """Bitwise the one-block pass, and (half) within its budget of the oracle."""
    for by in (0, 1, 2):
        for z in Z + [(1, 1)]:
            p = dict(L.parity_cases()[3 if z[0] == 3 else 1][1]["params"])
            p["bc"] = (2, 2, by, by) + z
            if z[0] == 3:
                p["inflow"] = dict(p["inflow"], xc=0.5 * (shape[0] - 1), yc=0.5 * (shape[1] - 1), D=2.0)
            w = dict(name="faces", shape=shape, params=p, fields=("random_blobs", dict(seed=3, blobs=2)), steps=4)
            rr, rb, u = L.initial_fields(w, seed=4, u_amp=0.02)
            lats = [pkg.Lattice(shape, p, storage=storage, block=b) for b in (1, 4)]
            assert [lat.block for lat in lats] == [1, 4]
            for lat in lats:
                lat.init_fields(rr, rb, u)
            orc = oracle.Oracle(shape, p)
            orc.init_fields(rr, rb, u)
            for n in (1, 2, 3, 4):
                for lat in lats:
                    lat.step(1)
                orc.step(1)
                a, b = (lat.get_populations() for lat in lats)
                assert np.array_equal(a, b), (by, z, n)
                for x, y in zip(*(lat.macro() for lat in lats)):
                    assert np.array_equal(x, y), (by, z, n)
                if storage == "c16":
                    assert np.max(np.abs(b - orc.f)) < 2e-3 * np.max(orc.f), (by, z, n)
            for lat in lats:
                lat.close()
