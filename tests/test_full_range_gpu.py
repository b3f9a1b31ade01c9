"""The largest particle number that a context takes, 2^31 - 1."""
import pytest

from test_parity_gpu import pm  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

NP = 2 ** 31 - 1
M = 1 << 20     # distinct records; particle i has the record i mod M


def mass_source(n, rec, box, om, a):
    """R = 4 pi G / a (rho - mean) of the records, each as often as it is there, and the largest 4 pi G / a rho."""
    import torch
    cell, f = rec[:, 0].view(torch.int32).long(), rec[:, 1:4].double()
    count = torch.full((M,), float(-(-NP // M)), dtype=torch.float64, device="cuda")
    count[NP % M:] -= 1
    s = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    c = [cell % n, cell // n % n, cell // n ** 2]
    for i in range(8):
        d = [i & 1, i >> 1 & 1, i >> 2]
        w = count
        for k in range(3):
            w = w * (f[:, k] if d[k] else 1 - f[:, k])
        x, y, z = [(c[k] + d[k]) % n for k in range(3)]
        s.index_add_(0, (z * n + y) * n + x, w)
    g = 1.5 * (box / 2997.92458) ** 2 / a * n ** 3
    return g * (s * om / NP - om / n ** 3), g * om / NP * float(s.max())


@pytest.mark.parametrize("newtonian", [False, True])
def test_two_steps_at_the_largest_particle_number(pm, newtonian):  # noqa: F811
    """Particles with the same record feel the same force, so they keep equal records; every one is moved.

    R of the mass deposit: a weight times the mass has four FP32 roundings, 2^-22 of a sum even where all lean one way
    (a vertex sees few records, 2048 times each), the mass one more.  The 8192 terms' roundings in the high word are at
    most 2^-12 of the sum, and come together in a word whose own roundings are then 2^-24 of the sum: 3.6e-7 in all."""
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
    s.project()
    if newtonian:   # the mass deposit, whose tiles count in 64 bits here
        r = torch.empty(n ** 3, dtype=torch.float64, device="cuda")
        pm.pm_get_field(s.ctx, "R", r)
        want, top = mass_source(n, rec, 400.0, 0.31, 1 / 21.0)
        assert float((r - want).abs().max()) < 1e-6 * top
    s.solve()
    s.update()
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

