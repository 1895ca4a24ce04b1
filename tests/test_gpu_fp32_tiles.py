"""The FP32 forward kernels chosen by problem size: the tile kernel (many points), the
latency kernel (few) and the general one (many channels at the largest widths).  They
form the same sums in the same order, so a point's channels do not depend on which one
runs: decoding points together or a few at a time gives the same bits.  Values are also
held to the FP64 oracle with the tolerances of test_gpu_fp32.py / test_gpu_siren.py."""
import numpy as np
import pytest

from oracle import crom_oracle as O
from workloads import gen

from helpers import dev, rel_l2

pytestmark = pytest.mark.gpu

# (m, r, width, hidden, activation): widths whose quarter of K is 8, 16, 24, 32, 40, 56
# and 64; one hidden layer; three coordinates; few and many channels
SHAPES = [(2, 8, 128, 5, "elu"), (1, 3, 32, 2, "elu"), (2, 5, 64, 1, "elu"), (3, 4, 96, 3, "siren"),
          (2, 6, 160, 2, "elu"), (1, 2, 224, 3, "siren"), (2, 16, 256, 2, "elu"), (3, 32, 256, 2, "elu")]


@pytest.fixture(scope="module")
def c():
    from paper_2206_02607_gb300 import build
    build()
    from paper_2206_02607_gb300 import crom
    return crom


@pytest.mark.parametrize("m,r,width,hidden,act", SHAPES)
def test_decode_does_not_depend_on_the_batch(c, m, r, width, hidden, act):
    import torch
    spec = gen.DecoderSpec(m, r, width, hidden)
    siren = act == "siren"
    params = gen.siren_decoder(spec, seed=7) if siren else gen.xavier_decoder(spec, seed=7, bias_std=0.2)
    ctx = c.crom_create(m, r, width, hidden, 0, activation=int(siren))
    c.crom_set_weights(ctx, gen.pack_params(params))
    rng = np.random.default_rng(8)
    n = 1237                                             # the last tile is ragged
    cuts = [0, 3, 3, 610, n]                             # instance borders inside tiles, one empty
    X = rng.uniform(-1 if siren else 0, 1, size=(n, m)).astype(np.float32)
    Q = rng.standard_normal((len(cuts) - 1, r)) * 0.5
    rows = 1 + m + m + 1 + r

    def decode(a, b, want=31, nrows=rows):
        off = np.clip(np.array(cuts), a, b) - a
        out = torch.empty((nrows, b - a), dtype=torch.float32, device="cuda")
        c.crom_decode(ctx, dev(Q, torch.float64), dev(off.astype(np.int32), torch.int32), dev(X[a:b], torch.float32),
                      want, out)
        return out.cpu().numpy()

    full = decode(0, n)
    # few points: one and two samples per CTA, an odd count, a range across two instances
    for a, b in ((0, 1), (1, 8), (600, 651), (n - 153, n), (0, 303)):
        assert np.array_equal(decode(a, b), full[:, a:b]), (a, b)
    # the value alone (the tile kernel's one-channel form) and without dg/dq
    assert np.array_equal(decode(0, n, c.CROM_WANT_VAL, 1)[0], full[0])
    assert np.array_equal(decode(0, n, c.CROM_WANT_DXX, m), full[1 + m:1 + 2 * m])
    dec = O.MLPDecoder(params, m, activation=act)
    for i in (0, 2, 3):
        s = slice(cuts[i], cuts[i + 1])
        ev = dec(X[s], Q[i])
        tol, tol2 = (1e-4, 1e-3) if siren else (1e-5, 1e-4)
        assert rel_l2(full[0, s], ev.g) < tol
        assert rel_l2(full[1:1 + m, s].T, ev.gx) < tol
        assert rel_l2(full[1 + m:1 + 2 * m, s].T, ev.gxx) < tol2
        assert rel_l2(full[2 + 2 * m:, s].T, ev.gq) < tol
    # reconstruction of the same points
    out = torch.empty((1, 500), dtype=torch.float32, device="cuda")
    c.crom_reconstruct(ctx, dev(Q[3:4], torch.float64), dev(X[610:1110], torch.float32), out)
    assert np.array_equal(out.cpu().numpy()[0], full[0, 610:1110])
    ctx.close()


@pytest.mark.parametrize("n_inst,M", [(1, 8), (1, 17), (1, 152), (1, 153), (1, 607), (1, 608), (3, 203), (40, 61)])
def test_step_at_the_borders_of_the_kernel_choice(c, n_inst, M):
    """One 2D step of the sizes around which the kernel, the samples per CTA, the
    partial rows and the groups of their chains change, against the oracle (q_{n+1} to
    1e-5 and the increment's field-space error as in test_gpu_fp32.py)."""
    from helpers import increment_errors, run_steps
    w = gen.heat2d_batched(n_inst=n_inst, m_lo=M, m_hi=M, first=4000)
    ctx = c.crom_create(2, 8, 128, 5, 0)
    c.crom_set_weights(ctx, gen.pack_params(w.params))
    q1, st = run_steps(ctx, w, 1, c.CROM_PREC_FP32)
    dec = O.MLPDecoder(w.params, 2)
    for i in sorted({0, n_inst - 1}):
        Y = w.samples[w.s_off[i]:w.s_off[i + 1]]
        ref, rst = O.crom_step(dec, w.q0[i], Y, w.dt, w.gn_iters, w.alpha[i])
        assert st[i] == 0 and rst == 0
        assert rel_l2(q1[i], ref) < 1e-5
        _, res, _, margin = increment_errors(w.params, 2, w.q0[i], Y, q1[i], ref, w.dt, w.alpha[i])
        assert res < (2e-4 if margin > 1e-6 else 5e-2), (res, margin)
    # the same batch again: every ticket and group counter is back at zero
    q2, st2 = run_steps(ctx, w, 1, c.CROM_PREC_FP32)
    assert np.array_equal(q1, q2) and np.array_equal(st, st2)
    ctx.close()
