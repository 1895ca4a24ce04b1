"""The full-order models' one-launch kernels (all steps of a call on the chip) at the
sizes where their tiling, clusters and kernel choice change, against the FP64 oracle.
Every FP32 step rounds a value of the field's size a few times (2^-24 each), so after
`steps` steps the relative L2 error stays below 4 steps 2^-24 (the schemes damp errors)."""
import numpy as np
import pytest

from oracle import crom_oracle as O

from helpers import dev, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def c():
    from paper_2206_02607_gb300 import build
    build()
    from paper_2206_02607_gb300 import crom
    return crom


# side, fields: one CTA per field (4, 12, 64), ragged tile rows over eight CTAs (100, 200,
# 252), the clusters and the wide kernels of 128 and 256 on both sides of their border,
# sides that are not multiples of 4 within and beyond the one-CTA kernel
CASES = [(4, 3), (12, 2), (64, 5), (64, 200), (100, 2), (128, 1), (128, 5), (128, 41), (200, 3), (252, 2), (256, 1),
         (256, 9), (256, 12), (3, 2), (5, 1), (97, 3), (101, 2), (127, 2), (129, 1)]


@pytest.mark.parametrize("model", ["heat", "heat_field", "upwind", "central"])
@pytest.mark.parametrize("n,nb", CASES)
def test_2d_one_launch(c, model, n, nb):
    import torch
    rng = np.random.default_rng(n + nb)
    u0 = rng.uniform(0.5, 1.5, size=(nb, n, n)).astype(np.float32)
    ax = ay = None
    if model.startswith("heat"):
        h = 1 / (n - 1)
        dt = h * h / 8
        coef = rng.uniform(0.2, 1.0, size=(nb, n, n) if model == "heat_field" else nb).astype(np.float32)
        kind = c.CROM_FOM_HEAT2D_NEUMANN_FIELD if model == "heat_field" else c.CROM_FOM_HEAT2D_NEUMANN
    else:
        ax, ay = (rng.uniform(-1, 1, size=(nb, n, n)).astype(np.float32) for _ in range(2))
        coef = rng.uniform(0.5, 1.0, size=nb).astype(np.float32)
        dt = 0.1 / n ** 2
        kind = c.CROM_FOM_ADVDIFF2D_PERIODIC if model == "upwind" else c.CROM_FOM_ADVDIFF2D_PERIODIC_CENTRAL
    for steps in (1, 2, 5):
        u = dev(u0, torch.float32)
        c.crom_fom_step(kind, u, torch.empty_like(u), dev(coef, torch.float32), dt=dt, n_steps=steps,
                        ax=None if ax is None else dev(ax, torch.float32), ay=None if ay is None else dev(ay, torch.float32))
        got = u.cpu().numpy()
        for b in sorted({0, nb // 2, nb - 1}):
            ref = u0[b].astype(np.float64)
            for _ in range(steps):
                if ax is None:
                    ref = O.fom_heat2d_neumann_step(ref, dt, coef[b].astype(np.float64))
                else:
                    ref = O.fom_advdiff2d_step(ref, ax[b].astype(np.float64), ay[b].astype(np.float64), float(coef[b]),
                                               dt, scheme="upwind" if model == "upwind" else "central")
            assert rel_l2(got[b], ref) < 4 * steps * 2.0 ** -24, (steps, b)
            # no node is left behind: the largest deviation is of rounding size too
            assert np.abs(got[b] - ref).max() < 16 * steps * 2.0 ** -24 * np.abs(ref).max(), (steps, b)


@pytest.mark.parametrize("P", [3, 33, 1024, 1500, 8192, 8193])
def test_1d_one_launch(c, P):
    import torch
    rng = np.random.default_rng(P)
    u0 = rng.uniform(0.5, 1.5, size=(3, P)).astype(np.float32)
    nu = rng.uniform(0.2, 1.0, size=(3, P)).astype(np.float32)
    dt, steps = 0.25 / (P - 1) ** 2, 5
    for kind, coef in ((c.CROM_FOM_HEAT1D_DIRICHLET, nu[:, 0].copy()), (c.CROM_FOM_HEAT1D_DIRICHLET_FIELD, nu)):
        u = dev(u0, torch.float32)
        c.crom_fom_step(kind, u, torch.empty_like(u), dev(coef, torch.float32), dt=dt, n_steps=steps)
        got = u.cpu().numpy()
        for b in range(3):
            ref = u0[b].astype(np.float64)
            for _ in range(steps):
                ref = O.fom_heat1d_step(ref, dt, coef[b].astype(np.float64))
            assert rel_l2(got[b], ref) < 4 * steps * 2.0 ** -24


# more fields than the GPU holds at once, of sides without a wide kernel: clusters of two
# to eight CTAs, and one CTA per field with two of them on an SM
@pytest.mark.parametrize("model", ["heat", "heat_field", "upwind", "central"])
@pytest.mark.parametrize("n,nb", [(57, 400), (96, 700), (164, 400), (200, 300), (252, 310)])
def test_2d_one_launch_of_many_fields(c, model, n, nb):
    test_2d_one_launch(c, model, n, nb)
