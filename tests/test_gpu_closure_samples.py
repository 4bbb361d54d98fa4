"""Box-filtered fields and strain rates of the closure-training samples (two fine cells per load in
the natural layout) against the exported populations: rows that end inside a warp, solid
cells, wall and free-slip faces, every layout and storage precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHANNEL = ("periodic", "periodic", "wall", "wall", "periodic", "periodic")
DUCT = ("periodic", "periodic", "freeslip", "freeslip", "wall", "wall")


@pytest.mark.parametrize("q,precision,streaming", [(19, "f32", "aa"), (27, "f16", "aa"), (19, "bf16", "aa"),
                                                   (27, "f32", "pull"), (19, "f16", "pull")])
@pytest.mark.parametrize("nx,faces", [(2, CHANNEL), (64, CHANNEL), (66, CHANNEL), (98, DUCT)])
def test_samples_match_populations(nx, faces, q, precision, streaming):
    import torch

    from paper_2305_09910_gb300 import lbm

    ny, nz, tau = 10, 6, 0.6
    rng = np.random.default_rng(nx * q)
    lat = lbm.Lattice(nx, ny, nz, stencil=q, tau=tau, faces=faces, streaming=streaming,
                      precision=precision, closure="none")
    flags = (rng.random((nz, ny, nx)) < 0.02).astype(np.uint8)
    lat.set_flags(flags)
    lat.init_equilibrium(rng.uniform(0.98, 1.02, (nz, ny, nx)).astype(np.float32),
                         rng.uniform(-0.05, 0.05, (3, nz, ny, nx)).astype(np.float32))
    n = nx // 2, ny // 2, nz // 2
    nc = n[0] * n[1] * n[2]
    c, _ = lbm.lbm_stencil(q)
    c = np.asarray(c, np.float64)

    def blocks(a):  # (..., nz, ny, nx) -> (..., nc, 8)
        a = a[..., :2 * n[2], :2 * n[1], :2 * n[0]].reshape(a.shape[:-3] + (n[2], 2, n[1], 2, n[0], 2))
        k = a.ndim - 6
        return a.transpose(tuple(range(k)) + (k, k + 2, k + 4, k + 1, k + 3, k + 5)).reshape(a.shape[:k] + (nc, 8))

    fluid = blocks((flags == 0).astype(np.float64))
    whole = fluid.min(-1) == 1
    eps = 2.0 ** -24
    for _ in range(4):
        df = lat.get_populations().astype(np.float64)
        drho, j = df.sum(0), np.einsum("qa,qzyx->azyx", c, df)
        pi = np.einsum("qa,qb,qzyx->abzyx", c, c, df) - np.eye(3)[:, :, None, None, None] * drho / 3
        pi -= j[:, None] * j[None] / (1 + drho)
        rho, j = blocks(1 + drho) * fluid, blocks(j) * fluid
        x, rest = torch.zeros((nc, 7), device="cuda"), [torch.zeros(nc, device="cuda") for _ in range(3)]
        rb, ub = torch.full((nc,), 7.0, device="cuda"), torch.full((3, nc), 7.0, device="cuda")
        lbm.lbm_closure_samples(lat.h, tau, 0.1, (1.0, 1.0), x, *rest)
        lbm.lbm_filter2(lat.h, rb, ub)
        x, rb, ub, smag = x.cpu().numpy(), rb.cpu().numpy(), ub.cpu().numpy(), rest[1].cpu().numpy()
        total = rho.sum(-1)
        # q + 8 float32 additions of values whose magnitudes sum to less than 1 per cell, then a division
        assert np.abs(rb - total / 8).max() <= (q + 10) * eps
        assert np.abs(ub - j.sum(-1) / np.where(total > 0, total, 1)).max() <= 2 * (q + 12) * eps
        # a stress is q + 8 operations on magnitudes below 1, a strain 3 / tau of it, |S| sqrt(18) of a strain
        S = 2 * (-3 / (2 * blocks(1 + drho) * tau) * blocks(pi)).mean(-1)
        ref = np.sqrt(2 * (S * S).sum((0, 1)))
        assert whole.sum() > nc // 2
        assert np.abs(smag - ref)[whole].max() <= 4.3 * (3.1 / tau) * (q + 8) * eps
        assert np.abs(x[:, 6] - (total / 8 - 1))[whole].max() <= (q + 10) * eps
        assert np.all(smag[~whole] == 0) and np.all(x[~whole] == 0)
        lat.step(1)
    assert ref[whole].max() > 1e-3
    lat.close()
