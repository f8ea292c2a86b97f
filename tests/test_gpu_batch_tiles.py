"""Tiles of the batch mode with several steps per pass: one launch holds periodic and Dirichlet
lattices, widths around the warp's 56 and the tile's 168 columns."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("kinds", ["mixed", "periodic", "dirichlet"])
def test_tiles_equal_single_lattices(lbm, storage, kinds):
    """Same passes (three steps each), so the same words as the single-lattice kernel."""
    import torch
    widths = [2, 55, 56, 57, 63, 112, 167, 168, 169, 240, 241, 337]
    bc = {"mixed": (0, 1), "periodic": (0, 0), "dirichlet": (1, 1)}[kinds]
    descs = [(w, 3 + 7 * i, bc[i % 2], 0.1, 0.1 / 3.2, 1.0, 0.6) for i, w in enumerate(widths)]
    gen = torch.Generator(device="cuda").manual_seed(1)
    fields = [torch.randn((3, 5, d[1], d[0]), dtype=torch.float64, device="cuda", generator=gen) * 1e-3 for d in descs]
    b = lbm.lbm_batch_create(descs, storage=lbm.STORAGE[storage])
    lbm.lbm_batch_set_mode(b, 2)
    for i, U in enumerate(fields):
        lbm.lbm_batch_init(b, i, U[0], U[1], U[2])
    lbm.lbm_batch_step(b, 9)
    for i, (d, U) in enumerate(zip(descs, fields)):
        got, want = (torch.empty((10, d[1], d[0]), dtype=torch.float64, device="cuda") for _ in range(2))
        lbm.lbm_batch_moments(b, i, got)
        lat = lbm.Lattice(d[0], d[1], *d[3:], dirichlet=bool(d[2]), storage=storage, track_displacement=False)
        lat.init(U[0], U[1], U[2], None, None)
        lat.step(9)
        lat.moments(want)
        lat.synchronize()
        lbm.lbm_batch_synchronize(b)
        assert torch.equal(got, want), d
        lat.close()
    lbm.lbm_batch_destroy(b)
