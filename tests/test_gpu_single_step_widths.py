"""Single step of the 16-bit formats: four nodes per thread from 2^19 nodes on, two below."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["bf16", "f16"])
@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("nx,ny", [(1024, 512), (1021, 515), (1023, 515), (2050, 300), (131073, 4), (9, 60000)])
def test_four_nodes_per_thread_store_the_same_words(lbm, nx, ny, dirichlet, storage):
    """Against the step with displacement tracking, which has two nodes per thread and the same
    node update."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(nx)
    f = torch.randn((4, 5, ny, nx), dtype=torch.float64, device="cuda", generator=gen).mul_(1e-3).cpu().numpy()
    out = []
    for track in (False, True):
        lat = lbm.Lattice(nx, ny, 0.1, 0.1 / 3.2, 1.0, 0.6, dirichlet=dirichlet, storage=storage, track_displacement=track)
        lat.set_populations(f, None)
        for _ in range(2):
            lat.step(1)
        pitch = (nx + 63) // 64 * 64
        raw = torch.empty(20 * ny * pitch + (2 * ny * pitch * 4 if track else 0), dtype=torch.int16, device="cuda")
        lbm.lbm_save_state(lat.ctx, raw)
        out.append(raw[:20 * ny * pitch].view(20, ny, pitch)[..., :nx].clone())
        lat.close()
    assert torch.equal(out[0], out[1])
