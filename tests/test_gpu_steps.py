"""Step kernels chosen by size, against the same steps taken one kernel at a time: several FP32
steps per pass (default grouping), several FP64 steps in one launch on small lattices, and the FP64
step with a body load on staged rows against the register kernel.  All bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _lattice(lbm, nx, ny, dirichlet, storage, load, nt=40, seed=0):
    rng = np.random.default_rng(seed + nx + 1000 * ny)
    lat = lbm.Lattice(nx, ny, 0.1, 0.1 / 3.2, 1.0, 0.6, dirichlet=dirichlet, storage=storage,
                      track_displacement=load)
    if load:
        R = 3
        lat.set_forcing(rng.standard_normal((R, nx)), rng.standard_normal((R, ny)),
                        rng.standard_normal((nt, 2, R)) * 1e-3)
        if dirichlet:
            lat.set_dirichlet(rng.standard_normal((nt, 2, 2 * (nx + ny))) * 1e-3)
    lat.set_populations(rng.standard_normal((4, 5, ny, nx)) * 1e-3, rng.standard_normal((2, ny, nx)) * 1e-3)
    return lat


def _state(lat):
    lat.synchronize()
    f, us = lat.populations()
    lat.close()
    return f, us


# tiles of 168 columns (56 per warp, 4 halo columns), copies of the wrapped columns for lattices
# wider than a tile; row blocks from 2 to 96 rows
@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("nx,ny,steps", [(2, 2, 4), (3, 5, 9), (55, 3, 5), (57, 9, 6), (112, 2, 7), (167, 11, 13),
                                         (168, 8, 8), (169, 4, 4), (171, 33, 11), (173, 200, 10), (335, 7, 21),
                                         (337, 40, 4), (1000, 3, 6), (61, 1500, 8)])
def test_fp32_default_passes_equal_single_steps(lbm, nx, ny, steps, dirichlet):
    one = _lattice(lbm, nx, ny, dirichlet, "f32", False)
    one.set_step_fusion(1)
    one.step(steps)
    many = _lattice(lbm, nx, ny, dirichlet, "f32", False)
    many.step(steps)
    np.testing.assert_array_equal(_state(one)[0], _state(many)[0])


@pytest.mark.parametrize("storage", ["bf16", "ms_bf16", "ms_f16", "ms_bfp"])
@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("nx,ny", [(55, 3), (119, 11), (121, 130), (167, 4), (168, 9), (173, 5), (239, 5), (240, 64), (241, 9), (243, 4),
                                   (481, 70)])
def test_16_bit_passes_do_not_depend_on_the_row_blocks(lbm, nx, ny, dirichlet, storage):
    states = []
    for rows in (0, 2, 5, 64):
        lat = _lattice(lbm, nx, ny, dirichlet, storage, False)
        if rows:
            lat.set_step_fusion(3, rows)
        lat.step(8)
        states.append(_state(lat)[0])
    for s in states[1:]:
        np.testing.assert_array_equal(states[0], s)


# one segment of 32 columns per warp, four per block; the largest still takes one launch
@pytest.mark.parametrize("load", [False, True])
@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 7), (31, 4), (32, 3), (33, 65), (64, 64), (100, 300), (700, 40),
                                   (2049, 2), (9000, 3)])
def test_fp64_steps_in_one_launch_equal_single_launches(lbm, nx, ny, dirichlet, load):
    many = _lattice(lbm, nx, ny, dirichlet, "f64", load)
    many.step(2)
    many.step(17)
    one = _lattice(lbm, nx, ny, dirichlet, "f64", load)
    for _ in range(19):
        one.step(1)
    a, b = _state(many), _state(one)
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])


@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("nx,ny,rows", [(2, 2, 1), (127, 5, 0), (129, 6, 4), (130, 9, 3), (1031, 7, 2), (260, 1300, 0)])
def test_fp64_body_load_staged_equals_register_kernel(lbm, nx, ny, rows, dirichlet):
    states = []
    for staging in (1, 0):
        lat = _lattice(lbm, nx, ny, dirichlet, "f64", True)
        lat.set_staging(staging)
        lat.set_step_fusion(1, rows)
        lat.step(9)
        states.append(_state(lat))
    np.testing.assert_array_equal(states[0][0], states[1][0])
    np.testing.assert_array_equal(states[0][1], states[1][1])


# two nodes per thread, blocks of 64 threads: 128 columns per block
@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 5), (127, 4), (128, 3), (129, 7), (257, 2), (1021, 9)])
def test_fp32_arithmetic_with_body_load(lbm, nx, ny, dirichlet, storage):
    """Steps launched one behind the other against a host wait after each (same words), and in FP32
    against FP64: 12 steps of some ten roundings of 2^-24 of the largest population each."""
    many = _lattice(lbm, nx, ny, dirichlet, storage, True)
    many.step(12)
    one = _lattice(lbm, nx, ny, dirichlet, storage, True)
    for _ in range(12):
        one.step(1)
        one.synchronize()
    a, b = _state(many), _state(one)
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])
    if storage == "f32":
        ref = _lattice(lbm, nx, ny, dirichlet, "f64", True)
        ref.step(12)
        f, us = _state(ref)
        assert np.max(np.abs(a[0] - f)) < 120 * 2.0 ** -24 * np.max(np.abs(f))
        assert np.max(np.abs(a[1] - us)) < 120 * 2.0 ** -24 * np.max(np.abs(us))
