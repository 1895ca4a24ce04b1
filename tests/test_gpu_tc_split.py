"""The tensor-core step with the tiles of few (or uneven) instances dealt to all groups,
one launch per Gauss-Newton iteration, against the form whose groups own whole
instances.  Both add an instance's tiles in the same order, and an instance's result does
not depend on the others in the call, so stepping an instance within a batch of more
instances than groups (whole form) and alone or with a few others (dealt form) gives the
same bits."""
import numpy as np
import pytest

from workloads import gen

from helpers import dev

pytestmark = pytest.mark.gpu

N_FILL = 1100                  # more than one and a quarter instances per group


@pytest.fixture(scope="module")
def c():
    from paper_2206_02607_gb300 import build
    build()
    from paper_2206_02607_gb300 import crom
    return crom


def _step(c, ctx, m, q, alpha, sizes, x, vel, prec, gn, steps=1, rollout=False, per_sample=False):
    import torch
    off = gen.ragged_offsets(sizes)
    qd, st = dev(q, torch.float64), torch.full((len(sizes),), -1, dtype=torch.int32, device="cuda")
    args = (dev(alpha, torch.float32), dev(off, torch.int32), dev(x, torch.float32), st)
    kw = dict(dt=1e-5, gn_iters=gn, max_samples=int(max(sizes)), precision=prec, coef_per_sample=per_sample,
              pde=c.CROM_PDE_HEAT if vel is None else c.CROM_PDE_ADVDIFF,
              vel=None if vel is None else dev(vel, torch.float32))
    if rollout:
        c.crom_rollout(ctx, qd, *args, n_steps=steps, **kw)
    else:
        for _ in range(steps):
            c.crom_step(ctx, qd, *args, **kw)
    assert c.crom_device_flags(ctx) == 0
    return qd.cpu().numpy(), st.cpu().numpy()


# (m, r, hidden, gn iterations, advection, per-sample coefficient)
@pytest.mark.parametrize("prec_name", ["CROM_PREC_F16X2", "CROM_PREC_F16"])
@pytest.mark.parametrize("m,r,hidden,gn,adv,per_sample", [(2, 8, 5, 2, False, False), (2, 15, 3, 1, True, False),
                                                          (1, 3, 2, 3, False, True), (2, 5, 4, 2, True, True)])
def test_dealt_tiles_give_the_same_bits(c, prec_name, m, r, hidden, gn, adv, per_sample):
    prec = getattr(c, prec_name)
    spec = gen.DecoderSpec(m, r, 128, hidden)
    ctx = c.crom_create(m, r, 128, hidden)
    c.crom_set_weights(ctx, gen.pack_params(gen.xavier_decoder(spec, seed=3, bias_std=0.1)))
    rng = np.random.default_rng(17)
    # sizes around the tiles (16 and 32 samples), one large, two the step refuses (r - 1, 0)
    probe = [32, 33, 31, 16, 17, 64, 1000, r - 1, 0, 200, max(r, 8)]
    sizes = np.array(probe + [40] * (N_FILL - len(probe)))
    off = gen.ragged_offsets(sizes)
    x = rng.uniform(0, 1, size=(off[-1], m)).astype(np.float32)
    vel = rng.uniform(-1, 1, size=(off[-1], m)).astype(np.float32) if adv else None
    alpha = rng.uniform(0.5, 2.0, size=off[-1] if per_sample else N_FILL).astype(np.float32)
    q = rng.standard_normal((N_FILL, r))
    whole, st_whole = _step(c, ctx, m, q, alpha, sizes, x, vel, prec, gn, per_sample=per_sample)

    def part(idx, **kw):
        cut = [np.arange(off[i], off[i + 1]) for i in idx]
        rows = np.concatenate(cut) if cut else np.zeros(0, int)
        return _step(c, ctx, m, q[idx], alpha[rows] if per_sample else alpha[idx], sizes[idx], x[rows],
                     None if vel is None else vel[rows], prec, gn, per_sample=per_sample, **kw)

    n = len(probe)
    for idx in (list(range(n)), [6], [9], list(range(n))[::-1], [8, 7, 6]):
        got, st = part(idx)
        assert np.array_equal(st, st_whole[idx]), idx
        assert np.array_equal(got, whole[idx]), idx
    assert st_whole[7] == c.CROM_ERR_INVALID_ARG and np.array_equal(whole[7], q[7])
    # a rollout graph of the dealt form repeats the steps, and a second one finds clean counters
    idx = [6, 9, 5]
    a, _ = part(idx, steps=3)
    b, _ = part(idx, steps=3, rollout=True)
    assert np.array_equal(a, b)
    assert np.array_equal(part(idx, steps=3, rollout=True)[0], b)
    ctx.close()


def test_singular_instance_among_dealt_ones(c):
    """An instance whose Jacobian has no full rank ends as SINGULAR after its first
    iteration and keeps its code; the others are stepped."""
    spec = gen.DecoderSpec(2, 4, 128, 3)
    params = gen.xavier_decoder(spec, seed=5)
    ctx = c.crom_create(2, 4, 128, 3)
    c.crom_set_weights(ctx, gen.pack_params(params))
    rng = np.random.default_rng(1)
    x = rng.uniform(0, 1, size=(600, 2)).astype(np.float32)
    x[:200] = x[0]                                  # 200 equal samples: rank 1
    q = rng.standard_normal((3, 4))
    got, st = _step(c, ctx, 2, q, np.ones(3, np.float32), np.array([200, 200, 200]), x, None, c.CROM_PREC_F16X2, 2)
    assert st[0] == c.CROM_ERR_SINGULAR and np.array_equal(got[0], q[0]), st
    assert st[1] == 0 and st[2] == 0 and not np.array_equal(got[1], q[1])
    ctx.close()
