"""FP32 training step at the shapes where its matrix products change tile, load width or
kernel: widths that are not multiples of 4 or of the tiles, one hidden layer, one latent
code, few and many rows; encoders without a convolution, with all of them in the
per-snapshot kernels and with long ones before those, and more snapshots than the bias
sums' chunks.  Loss and every gradient group against the FP64 oracle with the
tolerances of test_gpu_train.py (loss 1e-5, gradients 1e-4 relative L2)."""
import numpy as np
import pytest

from oracle import train_oracle as T

from helpers import dev, rel_l2
from test_gpu_train import groups, make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def c():
    from paper_2206_02607_gb300 import build
    build()
    from paper_2206_02607_gb300 import crom
    return crom


@pytest.mark.parametrize("n,r,width,hidden,B,S", [
    (7, 1, 1, 1, 1, 1), (8, 2, 5, 2, 2, 33), (16, 3, 33, 3, 3, 37), (16, 1, 64, 1, 2, 65), (48, 6, 100, 2, 7, 311),
    (48, 8, 128, 2, 20, 1000), (40, 5, 130, 3, 40, 700), (64, 16, 200, 2, 33, 129), (136, 4, 36, 2, 3, 50),
    (20, 3, 12, 1, 140, 2), (272, 3, 12, 1, 2, 9)])
def test_loss_and_gradients(c, n, r, width, hidden, B, S):
    import torch
    enc, dec, snaps, pt_idx, coords = make_problem(2, n, r, width, hidden, B, S)
    tr = c.CromTrainer(2, r, width, hidden, n * n, B, S)
    tr.set_params(T.flatten(enc, dec).astype(np.float32))
    loss_dev = torch.zeros(1, dtype=torch.float64, device="cuda")
    c.crom_train_step(tr, dev(snaps, torch.float32), dev(pt_idx, torch.int32), dev(coords, torch.float32), 1e-3, loss_dev)
    loss, eg, dg = T.loss_and_grads(enc, dec, snaps.astype(np.float64), pt_idx, coords.astype(np.float64), 2)
    assert abs(loss_dev.item() - loss) < 1e-5 * loss
    g_ref, g_gpu = T.flatten(eg, dg), tr.get_grads().astype(np.float64)
    for sl in groups(enc, dec):
        assert rel_l2(g_gpu[sl], g_ref[sl]) < 1e-4, sl
    # fewer snapshots than the trainer's batch through the encoder alone
    q = torch.empty((max(1, B - 1), r), dtype=torch.float32, device="cuda")
    c.crom_encode(tr, dev(snaps[:q.shape[0]], torch.float32), q)
    tr.close()
