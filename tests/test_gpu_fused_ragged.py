"""The fused density pass on rows that do not fill whole 32-node blocks, against the two-pass scheme.

Both compute one update; what differs is the rounding of the densities that enter the gradients: the
fused pass sums them in fixed point (2^-25 for densities up to 1), the density pass in FP32 (2^-24 of
each partial sum).  One step therefore changes the fields by a few 2^-24 of the density; 40 steps
of a smooth, stable flow let that grow to at most the bound on FP32 against the oracle
(2e-5 of the density scale, 1e-4 of max|u| + 3e-6, tests/test_gpu_parity.py).
"""
import numpy as np
import pytest

import lbm_inputs as L
import paper_1705_03141_gb300 as pkg

pytestmark = pytest.mark.gpu

# last block with 1, 2 and 31 nodes, less than one block, whole blocks; x faces with fast rows and without
SHAPES = [(33, 8, 9), (34, 9, 8), (63, 7, 10), (21, 12, 9), (64, 8, 8)]
FACES = {"periodic": (0, 0, 0, 0, 0, 0), "jet": (2, 2, 2, 2, 3, 4), "walls": (2, 2, 1, 1, 1, 1),
         "no-slip x": (1, 1, 0, 0, 0, 0), "one no-slip x": (1, 2, 2, 2, 2, 2)}


def _work(shape, faces):
    p = dict(L.parity_cases()[3][1]["params"])
    p.update(bc=FACES[faces])
    p["inflow"] = dict(p["inflow"], xc=0.5 * (shape[0] - 1), yc=0.5 * (shape[1] - 1), D=4.0) if faces == "jet" else None
    return dict(name=faces, shape=shape, params=p, fields=("random_blobs", dict(seed=9, blobs=3)), steps=40)


def _run(w, variant, block=0):
    rr, rb, u = L.initial_fields(w, seed=2, u_amp=0.02)
    lat = pkg.Lattice(w["shape"], w["params"], storage="f32", variant=variant, block=block)
    lat.init_fields(rr, rb, u)
    for n in (1, 23, 16):
        lat.step(n)
    out = lat.macro()
    lat.synchronize()
    lat.close()
    return out


@pytest.mark.parametrize("faces", list(FACES))
@pytest.mark.parametrize("shape", SHAPES)
def test_fused_ragged_rows(cuda, shape, faces):
    w = _work(shape, faces)
    ar, ab, au = _run(w, 1)
    scale = max(np.max(ar), np.max(ab))
    for block in (1, 2, 3):
        r, b, u = _run(w, 3, block)
        assert np.max(np.abs(r - ar)) < 2e-5 * scale and np.max(np.abs(b - ab)) < 2e-5 * scale
        assert np.max(np.abs(u - au)) < 1e-4 * np.max(np.abs(au)) + 3e-6
    again = _run(w, 3, 2)
    for x, y in zip(again, _run(w, 3, 2)):
        assert np.array_equal(x, y)  # bitwise reproducible


# densities far from the phase densities, which set the scale of the fixed-point sums: beyond the fine
# scale's range from the start (times 200), and growing past the density at which the scale changes
# on the way (phase densities 0.05: 2^-28 up to 0.5, range 8; the fields reach 0.36 at first, 0.58 later)
@pytest.mark.parametrize("faces", ["periodic", "walls", "jet"])
@pytest.mark.parametrize("ref,amp", [(1.0, 200.0), (0.05, 0.3)])
def test_fused_density_range(cuda, faces, ref, amp):
    shape = (34, 20, 18)
    w = _work(shape, faces)
    p = w["params"]
    p.update(rho_r0=ref, rho_b0=ref, A=0.0, beta=0.0)
    if faces == "jet":
        p["inflow"].update(D=1.0, u_j0=0.0, noise_frac=0.0)  # one inlet node
    x = np.arange(shape[0])[None, None, :] + 0.5
    z = np.arange(shape[2])[:, None, None] + 0.5
    one = np.ones((shape[2], shape[1], shape[0]))
    rho = amp * (1.0 + 0.2 * np.cos(2 * np.pi * x / shape[0])) * one
    q = 0.5 + 0.3 * np.cos(2 * np.pi * z / shape[2])
    u = np.zeros((3,) + rho.shape)
    u[0] = 0.3 * np.sin(2 * np.pi * x / shape[0]) * one  # towards the middle of the box
    peak = []

    def run(variant, chunks):
        lat = pkg.Lattice(shape, p, storage="f32", variant=variant)
        lat.init_fields(q * rho, (1 - q) * rho, u)
        for n in chunks:
            lat.step(n)
            peak.append(max(np.max(np.add(*lat.macro()[:2])), 0))
        f, m = lat.get_populations(), lat.macro()
        lat.close()
        return f, m

    f1, (r1, b1, u1) = run(1, (8, 16, 16))
    print(faces, ref, "largest density", peak)
    for chunks in ((8, 16, 16), (1,) * 8 + (32,)):
        f3, (r, b, v) = run(3, chunks)
        scale = np.max(np.abs(r1) + np.abs(b1))
        assert np.max(np.abs(r - r1)) < 2e-5 * scale and np.max(np.abs(b - b1)) < 2e-5 * scale
        assert np.max(np.abs(v - u1)) < 1e-4 * np.max(np.abs(u1)) + 3e-6


def test_library_choice_by_size(cuda):
    for shape, faces, variant in (((64, 20, 40), "periodic", 3), ((66, 20, 40), "periodic", 1),
                                  ((126, 104, 41), "periodic", 3), ((66, 20, 40), "jet", 3),
                                  ((126, 104, 41), "jet", 1), ((126, 104, 121), "jet", 3),
                                  ((64, 20, 40), "no-slip x", 1), ((126, 104, 41), "no-slip x", 1),
                                  ((96, 9, 8), "one no-slip x", 1)):
        lat = pkg.Lattice(shape, _work(shape, faces)["params"], storage="f32")
        assert lat.variant == variant
        lat.close()
    # a light phase with fewer than 23 bits above the fixed-point step: two passes on ragged rows
    for rho, shape, variant in (((4.0, 1.0), (126, 104, 41), 3), ((8.0, 1.0), (126, 104, 41), 1),
                                ((1.0, 0.1), (126, 104, 41), 1), ((0.1, 0.1), (126, 104, 41), 3),
                                ((1e-3, 1e-3), (126, 104, 41), 1), ((8.0, 1.0), (64, 20, 40), 3)):
        p = dict(_work(shape, "periodic")["params"], rho_r0=rho[0], rho_b0=rho[1])
        lat = pkg.Lattice(shape, p, storage="f32")
        assert lat.variant == variant, rho
        lat.close()
