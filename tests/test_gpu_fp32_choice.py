"""The FP32 kernels where the size chooses them: ranges of points large enough for the tile
kernel at every width and channel set, medium ones (general kernel) and small ones (latency
kernel).  All form the same sums in the same order, so a point's channels are the same bits
from each, and reconstruction gives the decode's values."""
import numpy as np
import pytest

from oracle import crom_oracle as O
from workloads import gen

from helpers import dev, rel_l2
from test_gpu_fp32_tiles import SHAPES, c  # noqa: F401 (the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,r,width,hidden,act", SHAPES)
def test_points_give_the_same_bits_from_every_kernel(c, m, r, width, hidden, act):  # noqa: F811
    import torch
    spec = gen.DecoderSpec(m, r, width, hidden)
    siren = act == "siren"
    params = gen.siren_decoder(spec, seed=5) if siren else gen.xavier_decoder(spec, seed=5, bias_std=0.2)
    ctx = c.crom_create(m, r, width, hidden, 0, activation=int(siren))
    c.crom_set_weights(ctx, gen.pack_params(params))
    rng = np.random.default_rng(6)
    n = 61_003                                           # 4 warps per SM at width 32, one channel; a ragged end
    cuts = np.array([0, 1, 30_001, 30_001, n])
    X = dev(rng.uniform(-1 if siren else 0, 1, size=(n, m)), torch.float32)
    Q = rng.standard_normal((4, r)) * 0.5

    def decode(a, b, want, rows):
        off = np.clip(cuts, a, b) - a
        out = torch.empty((rows, b - a), dtype=torch.float32, device="cuda")
        c.crom_decode(ctx, dev(Q, torch.float64), dev(off.astype(np.int32), torch.int32), X[a:b].contiguous(), want, out)
        return out.cpu().numpy()

    sets = [(c.CROM_WANT_VAL, 1), (c.CROM_WANT_DXX, m), (c.CROM_WANT_VAL | c.CROM_WANT_DQ, 1 + r), (31, 2 + 2 * m + r)]
    for want, rows in sets:
        full = decode(0, n, want, rows)
        assert np.all(np.isfinite(full))
        for a, b in ((0, 2), (29_990, 30_020), (n - 301, n), (29_000, 30_400), (n - 5_001, n)):
            assert np.array_equal(decode(a, b, want, rows), full[:, a:b]), (want, a, b)
        if want == c.CROM_WANT_VAL:
            value = full[0]
    for a, b in ((30_001, n), (30_001, 31_000), (n - 97, n)):
        out = torch.empty((1, b - a), dtype=torch.float32, device="cuda")
        c.crom_reconstruct(ctx, dev(Q[3:], torch.float64), X[a:b].contiguous(), out)
        assert np.array_equal(out.cpu().numpy()[0], value[a:b]), (a, b)
    ctx.close()


@pytest.mark.parametrize("r,width,hidden", [(3, 32, 2), (8, 64, 3), (5, 96, 2), (6, 256, 2)])
def test_steps_of_one_a_dozen_and_many_instances(c, r, width, hidden):  # noqa: F811
    """The same instance alone (latency kernel), twelve times (general) and 700 times (tile):
    every copy the same bits, q_{n+1} against the oracle to 1e-5 as in test_gpu_fp32.py."""
    import torch
    spec = gen.DecoderSpec(2, r, width, hidden)
    params = gen.xavier_decoder(spec, seed=9, bias_std=0.2)
    ctx = c.crom_create(2, r, width, hidden, 0)
    c.crom_set_weights(ctx, gen.pack_params(params))
    rng = np.random.default_rng(10)
    M, dt, alpha = 61, 1e-5, 0.75
    X = rng.uniform(0.1, 0.9, size=(M, 2)).astype(np.float32)
    q0 = rng.standard_normal(r) * 0.5
    ref, rst = O.crom_step(O.MLPDecoder(params, 2), q0, X, dt, 2, alpha)
    assert rst == 0
    for n in (1, 12, 700):
        q = dev(np.tile(q0, (n, 1)), torch.float64)
        status = torch.full((n,), 7, dtype=torch.int32, device="cuda")
        c.crom_step(ctx, q, dev(np.full(n, alpha), torch.float32), dev((np.arange(n + 1) * M), torch.int32),
                    dev(np.tile(X, (n, 1)), torch.float32), status, dt=dt, gn_iters=2, max_samples=M)
        q1 = q.cpu().numpy()
        assert not status.any() and np.all(q1 == q1[0]), n
        assert rel_l2(q1[0], ref) < 1e-5, n
    ctx.close()
