"""The tensor-core step's dealt form (few or uneven instances, one launch per Gauss-Newton
iteration) where an instance fails in its second iteration: that launch writes its status
while CTAs that were kept waiting for an SM have yet to lay out their tiles.  Every
instance must end with the bits and the status of the whole-instance form."""
import numpy as np
import pytest

from workloads import gen

from helpers import dev

pytestmark = pytest.mark.gpu

N_FILL = 1100                  # more than one and a quarter instances per group: whole form


@pytest.fixture(scope="module")
def c():
    from paper_2206_02607_gb300 import build
    build()
    from paper_2206_02607_gb300 import crom
    return crom


class Batch:
    def __init__(self, sizes, x, q, alpha):
        import torch
        self.q0, self.n = q, len(sizes)
        self.q = dev(q, torch.float64)
        self.status = torch.full((self.n,), -1, dtype=torch.int32, device="cuda")
        self.args = (dev(alpha, torch.float32), dev(gen.ragged_offsets(sizes), torch.int32), dev(x, torch.float32),
                     self.status)
        self.max = int(max(sizes))

    def reset(self):
        import torch
        self.q.copy_(dev(self.q0, torch.float64))

    def step(self, c, ctx, prec, gn):
        c.crom_step(ctx, self.q, *self.args, dt=1e-5, gn_iters=gn, max_samples=self.max, precision=prec)

    def result(self):
        return self.q.cpu().numpy(), self.status.cpu().numpy()


def _ctx(c, params, hidden):
    ctx = c.crom_create(2, 8, 128, hidden)
    c.crom_set_weights(ctx, gen.pack_params(params))
    return ctx


@pytest.mark.parametrize("gn", [2, 3])
@pytest.mark.parametrize("prec_name", ["CROM_PREC_F16X2", "CROM_PREC_F16"])
def test_failure_after_the_first_iteration(c, prec_name, gn):
    import torch
    prec, hidden = getattr(c, prec_name), 4
    params = gen.xavier_decoder(gen.DecoderSpec(2, 8, 128, hidden), seed=3, bias_std=0.1)
    rng = np.random.default_rng(7)
    probe = [300, 200, 64, 1000, 333, 17, 500, 40]
    failing = [1, 4, 6]            # a coefficient so large that the first update leaves the f16 range
    sizes = np.array(probe + [40] * (N_FILL - len(probe)))
    off = gen.ragged_offsets(sizes)
    x = rng.uniform(0, 1, size=(off[-1], 2)).astype(np.float32)
    q = rng.standard_normal((N_FILL, 8))
    alpha = rng.uniform(0.5, 2.0, size=N_FILL).astype(np.float32)
    alpha[failing] = 1e30
    n = len(probe)
    ctx, other = _ctx(c, params, hidden), _ctx(c, params, hidden)
    big = Batch(sizes, x, q, alpha)
    big.step(c, ctx, prec, gn)
    whole, st_whole = (a[:n] for a in big.result())
    assert all(st_whole[i] in (c.CROM_ERR_SINGULAR, c.CROM_ERR_NONFINITE) for i in failing), st_whole
    assert all(st_whole[i] == c.CROM_OK for i in range(n) if i not in failing), st_whole
    assert not np.any(np.all(whole == q[:n], axis=1))          # the failing ones made one update

    few = Batch(sizes[:n], x[:off[n]], q[:n], alpha[:n])
    busy = Batch(sizes, x, q, np.ones(N_FILL, np.float32))
    busy.step(c, other, prec, gn)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for _ in range(4):
        few.reset()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):                           # holds the SMs meanwhile
            for _ in range(2):
                busy.step(c, other, prec, gn)
        few.step(c, ctx, prec, gn)
        torch.cuda.synchronize()
        got, st = few.result()
        assert c.crom_device_flags(ctx) == 0
        assert np.array_equal(st, st_whole), (st, st_whole)
        assert np.array_equal(got, whole)
    # later steps of the same context find its tickets clean, whichever kernels they use
    for p in (prec, c.CROM_PREC_FP32):
        clean = Batch(sizes[:n], x[:off[n]], q[:n], np.ones(n, np.float32))
        clean.step(c, ctx, p, gn)
        got, st = clean.result()
        fresh_ctx, fresh = _ctx(c, params, hidden), Batch(sizes[:n], x[:off[n]], q[:n], np.ones(n, np.float32))
        fresh.step(c, fresh_ctx, p, gn)
        want, st_want = fresh.result()
        assert np.all(st == c.CROM_OK) and np.array_equal(st, st_want) and np.array_equal(got, want)
        fresh_ctx.close()
    ctx.close()
    other.close()


@pytest.mark.parametrize("prec_name", ["CROM_PREC_F16X2", "CROM_PREC_F16"])
def test_overlapping_sample_ranges(c, prec_name):
    """Offsets that decrease between instances whose ranges overlap: the instances in
    between are refused, the others give the bits they give on their own, though their
    tiles are more than the samples make.  One Gauss-Newton iteration: later ones keep
    Delta f per sample, which overlapping instances share in every form of the step."""
    import torch
    prec, n = getattr(c, prec_name), 400
    params = gen.xavier_decoder(gen.DecoderSpec(2, 8, 128, 4), seed=3, bias_std=0.1)
    ctx = _ctx(c, params, 4)
    rng = np.random.default_rng(11)
    x = rng.uniform(0, 1, size=(n, 2)).astype(np.float32)
    off = np.array([0, 300, 100, 400, 0, 400, 0, 17, 1, 400])
    k = len(off) - 1
    q, alpha = rng.standard_normal((k, 8)), rng.uniform(0.5, 2.0, size=k).astype(np.float32)
    qd, st = dev(q, torch.float64), torch.full((k,), -1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        c.crom_step(ctx, qd, dev(alpha, torch.float32), dev(off, torch.int32), dev(x, torch.float32), st, dt=1e-5,
                    gn_iters=1, max_samples=n, precision=prec)
    got, st = qd.cpu().numpy(), st.cpu().numpy()
    for i in range(k):
        lo, hi = off[i], off[i + 1]
        if hi < lo:
            assert st[i] == c.CROM_ERR_INVALID_ARG and np.array_equal(got[i], q[i]), i
            continue
        one = Batch(np.array([hi - lo]), x[lo:hi], q[i:i + 1], alpha[i:i + 1])
        for _ in range(2):
            one.step(c, ctx, prec, 1)
        want, st_want = one.result()
        assert st[i] == st_want[0] == c.CROM_OK and np.array_equal(got[i], want[0]), i
    ctx.close()
