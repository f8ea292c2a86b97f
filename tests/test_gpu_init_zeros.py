"""Initial states with zeros in them: the reduced formats store zero exactly where every order of
evaluation gives zero, and the rounded FP64 values elsewhere."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FIELDS = {
    "rest": lambda U: 0.0 * U,
    "pulse": lambda U: np.where((np.arange(U.shape[-1]) < 9) & (np.arange(U.shape[-2]) < 7)[:, None], U, 0.0),
    "plane wave": lambda U: U * np.array([1, 0, 1, 1, 0])[:, None, None] * np.array([1, 1, 0])[:, None, None, None],
    "velocity": lambda U: U * np.array([1, 1, 0, 0, 0])[:, None, None],
    "one component": lambda U: U * np.array([0, 0, 0, 1, 0])[:, None, None],
    "gradient only": lambda U: U * np.array([0, 0, 1])[:, None, None, None],
}


@pytest.mark.parametrize("load", [False, True])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("name", FIELDS)
def test_zeros_of_the_initial_state(lbm, name, storage, load):
    nx, ny = 37, 22
    rng = np.random.default_rng(4)
    U = FIELDS[name](rng.standard_normal((3, 5, ny, nx)) * 1e-3)
    B = FIELDS[name](rng.standard_normal((3, 5, ny, nx)))[0, :2] if load else None
    f = {}
    for s in ("f64", storage):
        lat = lbm.Lattice(nx, ny, 0.1, 0.1 / 3.2, 1.0, 0.6, storage=s, track_displacement=False)
        if load:
            lat.set_forcing(np.ones((1, nx)), np.ones((1, ny)), np.zeros((2, 2, 1)))
        lat.init(np.ascontiguousarray(U[0]), np.ascontiguousarray(U[1]), np.ascontiguousarray(U[2]), B, None)
        es, pitch = {"f64": 8, "f32": 4, "bf16": 2}[s], 64              # the stored words
        raw = np.zeros(20 * ny * pitch * es, np.uint8)
        lbm.lbm_save_state(lat.ctx, raw)
        v = raw.view({8: np.float64, 4: np.float32, 2: np.uint16}[es])
        v = (v.astype(np.uint32) << 16).view(np.float32) if es == 2 else v
        f[s] = v.astype(np.float64).reshape(4, 5, ny, pitch)[..., :nx]
        lat.close()
    zero = f["f64"] == 0.0
    assert zero.all() if name == "rest" else zero.any() == (name in ("pulse", "plane wave"))
    assert np.all(f[storage][zero] == 0.0)
    # one rounding to the format, and the FP64 orders' difference
    unit = {"f32": 2.0 ** -24, "bf16": 2.0 ** -8}[storage]
    big = np.abs(f["f64"]).max(axis=(0, 1), keepdims=True)
    assert np.all(np.abs(f[storage] - f["f64"]) <= unit * np.abs(f["f64"]) + 64 * 2.0 ** -52 * big)
