"""The largest particle number that a context takes, 2^31 - 1."""
import pytest

from test_parity_gpu import pm  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

NP = 2 ** 31 - 1
M = 1 << 20     # distinct records; particle i has the record i mod M


@pytest.mark.parametrize("newtonian", [False, True])
def test_two_steps_at_the_largest_particle_number(pm, newtonian):  # noqa: F811
    """Particles with the same record feel the same force, so they keep equal records; every one is moved."""
    import torch
    torch.cuda.empty_cache()
    need = NP * (2 * 32 + 28) + (16 << 30)
    if torch.cuda.mem_get_info()[0] < need:
        pytest.skip("needs %d GB of device memory" % (need >> 30))
    n = 128
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    rec = torch.empty((M, 7), dtype=torch.float32, device="cuda")
    rec[:, 0] = torch.randint(0, n ** 3, (M,), generator=g, device="cuda", dtype=torch.int32).view(torch.float32)
    rec[:, 1:4] = torch.rand((M, 3), generator=g, device="cuda")
    rec[:, 4:] = 1e-3 * torch.randn((M, 3), generator=g, device="cuda")
    io = torch.empty((NP, 7), dtype=torch.float32, device="cuda")
    for i in range(0, NP, M):
        io[i:i + M] = rec[:min(M, NP - i)]
    torch.cuda.synchronize()
    s = pm.PM(n, NP, 400.0, 0.31, 20.0, 0.0, 100, pm.PM_MIXED, pm.PM_NEWTONIAN if newtonian else 0)
    pm.pm_set_particles_packed(s.ctx, NP, io)
    for _ in range(2):
        s.step()
    io.zero_()
    torch.cuda.synchronize()
    pm.pm_get_particles_packed(s.ctx, NP, io)
    torch.cuda.synchronize()
    s.close()
    bits = io.view(torch.int32)
    first = bits[:M].clone()
    cell = first[:, 0].long()
    assert int(cell.min()) >= 0 and int(cell.max()) < n ** 3 and bool(torch.isfinite(io[:M, 1:]).all())
    assert bool((io[:M, 4:] != rec[:, 4:]).any(1).all())       # every particle was kicked
    for i in range(0, NP, M):
        assert torch.equal(bits[i:i + M], first[:min(M, NP - i)])
    del io, bits
    torch.cuda.empty_cache()
