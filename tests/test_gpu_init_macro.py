"""Initial populations and macroscopic fields: FP32-arithmetic storages take FP64 fields in through head + tail
FP32 pairs and out through lossless sums of FP32 values.

Bounds.  A pair holds 48 bits and each operation on pairs errs by a few units of 2^-47 of its
operands, so an initial FP32 population is the FP64 value (a sum of terms at most 8 times its size
for |u| <= 0.15) rounded once: 2^-24 of it, plus 2^-40.  A macroscopic density is the sum of 27 stored
values rounded to FP64 in two additions, 2^-52 of it; the velocity, of a speed below 1, carries the roundings of
its momentum (2), of rho (3 in the quotient and the force), of the force and of the quotient: 8 units of 2^-53.
FP64 storage sums in FP64, at most 27 roundings of a partial sum: 2^-48 for all.
"""
import numpy as np
import pytest

import lbm_inputs as L
import oracle
import paper_1705_03141_gb300 as pkg

pytestmark = pytest.mark.gpu

# one node deep, odd, one row of a whole block plus one node, several blocks of threads
SHAPES = [(3, 3, 3), (33, 5, 4), (32, 9, 7), (65, 8, 6)]


def _work(shape):
    p = dict(L.parity_cases()[3][1]["params"])  # the jet's densities and force
    p.update(bc=(0,) * 6, inflow=None)
    return dict(name="box", shape=shape, params=p, fields=("random_blobs", dict(seed=3, blobs=2)), steps=0)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("storage,eps_f,eps_m", [("f64", 2.0 ** -48, 2.0 ** -48), ("f32", 2.0 ** -24 + 2.0 ** -40, 2.0 ** -52),
                                                 ("f16", None, 2.0 ** -52), ("bf16", None, 2.0 ** -52)])
def test_initial_populations_and_macroscopic_sums(shape, storage, eps_f, eps_m):
    w = _work(shape)
    rr, rb, u = L.initial_fields(w, seed=5, u_amp=0.1)
    lat = pkg.Lattice(shape, w["params"], storage=storage)
    lat.init_fields(rr, rb, u)
    f = lat.get_populations()
    orc = oracle.Oracle(shape, w["params"])
    orc.init_fields(rr, rb, u)
    ref = orc.f.reshape(f.shape)
    if eps_f is not None:
        assert np.all(np.abs(f - ref) <= eps_f * np.abs(ref) + 1e-45)
    r, b, v = lat.macro()
    lat.close()
    # the same sums of the stored populations in extended precision
    g = f.astype(np.longdouble)
    sr, sb = g[0].sum(0), g[1].sum(0)
    assert np.all(np.abs(r - sr) <= eps_m * sr + 1e-45) and np.all(np.abs(b - sb) <= eps_m * sb + 1e-45)
    c = oracle.tables()[0]
    c = np.asarray(c).reshape(27, 3)
    p = w["params"]
    rho = sr + sb
    # the force's constants are held in the storage's compute type
    real = np.float64 if storage == "f64" else np.float32
    for a in range(3):
        mom = sum(int(c[i][a]) * (g[0, i] + g[1, i]) for i in range(27))
        F = (rho - np.longdouble(real(p["rho_b0"]))) * np.longdouble(real(p["g"][a]))
        assert np.all(np.abs(v[a] - (mom + F / 2) / rho) <= 4 * eps_m)


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_initial_fields_out_of_the_pairs_range(storage):
    """Infinities, densities that FP32 cannot hold or whose tails it loses, and large velocities: the populations are
    the FP64 equilibria, rounded once to the storage."""
    shape = (33, 5, 4)
    w = _work(shape)
    rr, rb, u = L.initial_fields(w, seed=5, u_amp=0.1)
    n = [(0, 0, 0), (0, 1, 5), (1, 2, 32), (2, 3, 31), (3, 4, 7), (2, 0, 0), (1, 1, 1), (3, 0, 20), (1, 3, 3)]
    rr[n[0]], rr[n[1]], rb[n[2]], rr[n[3]] = np.inf, 1e39, 4e38, 1e-36
    rb[n[4]], rr[n[4]], u[(1,) + n[5]], u[(2,) + n[6]] = 2e-38, 1e-44, 1e20, np.inf
    rr[n[7]], rb[n[7]], rb[n[8]] = 0.0, 1e-42, np.nan
    u[(slice(None),) + n[0]] = 0.0
    lat = pkg.Lattice(shape, w["params"], storage=storage)
    lat.init_fields(rr, rb, u)
    orc = oracle.Oracle(shape, w["params"])
    orc.init_fields(rr, rb, u)
    with np.errstate(all="ignore"):
        ref = orc.f.reshape((2, 27) + shape[::-1])
        ref = ref if storage == "f64" else ref.astype(np.float32).astype(np.float64)
        f = lat.get_populations().reshape(ref.shape)
        for at in n:
            a, b = f[(slice(None), slice(None)) + at], ref[(slice(None), slice(None)) + at]
            assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b)), at
            ok = np.isfinite(b)
            # FP64 operations in another order, and for FP32 storage the unit by which they may round differently
            eps = 2.0 ** -48 if storage == "f64" else 2.0 ** -23
            assert np.all(np.abs(a[ok] - b[ok]) <= eps * np.abs(b[ok]) + (storage == "f32") * 2.0 ** -149), at
    lat.close()


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_macroscopic_fields_of_infinite_populations(storage):
    """A node with an infinite, an overflowing, a NaN population: as the sums in FP64 have it, other nodes untouched."""
    shape = (33, 5, 4)
    w = _work(shape)
    rr, rb, u = L.initial_fields(w, seed=5, u_amp=0.1)
    lat = pkg.Lattice(shape, w["params"], storage=storage)
    lat.init_fields(rr, rb, u)
    f = lat.get_populations().reshape((2, 27) + shape[::-1])
    clean = lat.macro()
    f[0, 3, 1, 2, 4] = np.inf
    f[:, 5:7, 2, 3, 32] = 3e38  # the density of each colour is beyond FP32
    f[1, 9, 3, 0, 7] = np.nan
    lat.set_populations(f)
    r, b, v = lat.macro()
    lat.close()
    assert r[1, 2, 4] == np.inf and b[1, 2, 4] == clean[1][1, 2, 4]
    assert np.isnan(b[3, 0, 7]) and r[3, 0, 7] == clean[0][3, 0, 7] and np.all(np.isnan(v[:, 3, 0, 7]))
    for a, k in ((r, 0), (b, 1)):
        want = f[k, :, 2, 3, 32].astype(np.float32).astype(np.longdouble).sum() if storage == "f32" else f[k, :, 2, 3, 32].sum()
        assert abs(a[2, 3, 32] - want) <= 2.0 ** -48 * want
    hit = np.zeros(r.shape, bool)
    hit[1, 2, 4] = hit[2, 3, 32] = hit[3, 0, 7] = True
    for a, c in zip((r, b, *v), (clean[0], clean[1], *clean[2])):
        assert np.array_equal(a[~hit], c[~hit])
