"""The training kernel's slots against the oracle's loss and gradient: one example, fewer and more examples than
CTAs, and more than the slots of all CTAs take in one round."""
import numpy as np
import pytest

import paper_2511_20911_gb300 as crbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    crbm.load_library()


@pytest.mark.parametrize("n,L", [(1, 10), (2, 12), (151, 10), (153, 18), (1217, 10)])
def test_loss_grad_counts_every_example(orc, n, L):
    """fp32 sums against the oracle's double.  An fp32 sum within its rounding error (1e-6) of a bfloat16 tie may
    round an activation the other way, by 2^-8: a few such flips per ten examples, each worth at most 2e-2 of one
    example's gradient and 2e-3 of its loss, independent between examples, so their mean shrinks with sqrt(n)."""
    rng = np.random.default_rng(n)
    spins = rng.choice(np.array([-1, 1], np.int8), (n, L, L))
    origins = rng.integers(0, L, (n, 2)).astype(np.int32)
    bh = np.stack([rng.choice([0.5, 1.5, 3.0], n), rng.choice([-1.0, 2.5, 3.25], n)], 1).astype(np.float32)  # bfloat16 values
    w = orc.random_net(n + 3, scale=0.2)
    p = crbm.Proposal(seed=2)
    p.weights = w
    loss, grad = p.loss_grad(spins, origins, bh)
    inputs = np.array([orc.patch_input(spins[e], int(origins[e, 0]), int(origins[e, 1]), 4, float(bh[e, 0]),
                                       float(bh[e, 1])) for e in range(n)])
    targets = np.array([[spins[e, (origins[e, 0] + a // 4) % L, (origins[e, 1] + a % 4) % L] for a in range(16)]
                        for e in range(n)], np.int8)
    wb = np.vectorize(orc.bf16)(w.astype(np.float32).astype(np.float64))
    l_ref, g_ref = orc.net_loss_grad(4, wb, inputs, targets, use_bf16=True)
    assert abs(loss - l_ref) <= 2e-3 / np.sqrt(n) * abs(l_ref)
    assert np.linalg.norm(grad - g_ref) <= 2e-2 / np.sqrt(n) * np.linalg.norm(g_ref)
