"""Which step kernels a call launches, and the bounded wait of the launch that takes all its steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _lattice(lbm, nx, ny, storage="f64", dirichlet=False, load=False):
    lat = lbm.Lattice(nx, ny, 0.1, 0.1 / 3.2, 1.0, 0.6, dirichlet=dirichlet, storage=storage, track_displacement=load)
    rng = np.random.default_rng(nx + ny)
    if load:
        lat.set_forcing(rng.standard_normal((2, nx)), rng.standard_normal((2, ny)), rng.standard_normal((60, 2, 2)) * 1e-3)
    lat.set_populations(rng.standard_normal((4, 5, ny, nx)) * 1e-3, None)
    return lat


# the sizes of test_fp64_steps_in_one_launch_equal_single_launches
@pytest.mark.parametrize("load", [False, True])
@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 7), (31, 4), (32, 3), (33, 65), (64, 64), (100, 300), (700, 40),
                                   (2049, 2), (9000, 3)])
def test_small_fp64_lattices_take_one_launch(lbm, nx, ny, dirichlet, load):
    lat = _lattice(lbm, nx, ny, dirichlet=dirichlet, load=load)
    assert lat.step_launches() == (0, 0, 0)
    lat.step(2)
    lat.step(17)
    assert lat.step_launches() == (0, 0, 2)
    lat.step(1)                                  # a single step is one launch as it is
    lat.set_step_fusion(1)
    lat.step(4)
    assert lat.step_launches() == (5, 0, 2)
    lat.synchronize()
    lat.close()


def test_larger_lattices_take_a_launch_per_step_or_pass(lbm):
    # FP64: one launch where two such lattices fit on the chip together, 4 x 152 / 2 blocks of 4 segments
    for nx, ny, storage, want in ((32, 1216, "f64", (0, 0, 1)), (32, 1217, "f64", (9, 0, 0)), (208, 208, "f64", (9, 0, 0)),
                                  (512, 256, "f64", (9, 0, 0)), (64, 64, "f32", (0, 3, 0)), (64, 64, "bf16", (0, 3, 0)),
                                  (64, 64, "ms_bfp", (0, 3, 0))):
        lat = _lattice(lbm, nx, ny, storage)
        lat.step(9)
        assert lat.step_launches() == want, (nx, ny, storage)
        lat.synchronize()
        lat.close()


@pytest.mark.parametrize("nx,ny", [(20, 3), (64, 64)])
def test_one_launch_reports_a_wait_that_runs_out(lbm, nx, ny):
    """Test hook: one block never reports its steps, so its neighbours' bounded waits run out (about
    2 s), theirs with them; lbm_synchronize reports it once and the context stays usable."""
    lat = _lattice(lbm, nx, ny)
    lat.set_staging(2)
    lat.step(5)
    with pytest.raises(lbm.LbmError) as e:
        lat.synchronize()
    assert e.value.status == lbm.LBM_ERR_TIMEOUT
    lat.synchronize()                            # the flag was cleared
    lat.set_staging(1)
    f = np.random.default_rng(1).standard_normal((4, 5, ny, nx)) * 1e-3
    got = []
    for one in (False, True):
        if one:
            lat.set_step_fusion(1)
        lat.set_populations(f, None)
        lat.step(6)
        lat.synchronize()
        got.append(lat.populations()[0])
    assert lat.step_launches() == (6, 0, 2)
    np.testing.assert_array_equal(got[0], got[1])
    lat.close()


@pytest.mark.parametrize("storage,nx,ny,default", [("f32", 300, 40, (0, 3, 0)), ("bf16", 300, 40, (0, 4, 0)),
                                                   ("f64", 64, 64, (0, 0, 1)), ("f64", 512, 256, (12, 0, 0))])
def test_zero_steps_per_pass_restores_the_default(lbm, storage, nx, ny, default):
    lat = _lattice(lbm, nx, ny, storage)
    lat.step(12)
    assert lat.step_launches() == default
    lat.set_step_fusion(1, 7)
    lat.step(12)
    before = lat.step_launches()
    assert before == (default[0] + 12, default[1], default[2])
    lat.set_step_fusion(0)
    lat.step(12)
    assert tuple(b - a for a, b in zip(before, lat.step_launches())) == default
    for bad in (-1, 4):
        with pytest.raises(lbm.LbmError):
            lat.set_step_fusion(bad)
    lat.synchronize()
    lat.close()


@pytest.mark.parametrize("rows", [2, 5, 64])
@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_default_passes_with_rows_given(lbm, storage, dirichlet, rows):
    """FP32's four steps per pass (FP16's three) with the rows of a block given."""
    got = []
    for r in (0, rows):
        lat = _lattice(lbm, 173, 131, storage, dirichlet)
        lat.set_step_fusion(0, r)
        lat.step(12)
        assert lat.step_launches() == (0, {"f32": 3, "f16": 4}[storage], 0)
        lat.synchronize()
        got.append(lat.populations()[0])
        lat.close()
    np.testing.assert_array_equal(got[0], got[1])
