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


def check_against_oracle(orc, p, w, spins, origins, bh, distinct):
    """As above, for examples of which the first `distinct` are repeated in turn."""
    n, L = len(origins), spins.shape[-1]
    loss, grad = p.loss_grad(spins, origins, bh)
    inputs = np.array([orc.patch_input(spins[e], int(origins[e, 0]) % L, int(origins[e, 1]) % L, 4, float(bh[e, 0]),
                                       float(bh[e, 1])) for e in range(distinct)])
    targets = np.array([[spins[e, (origins[e, 0] + a // 4) % L, (origins[e, 1] + a % 4) % L] for a in range(16)]
                        for e in range(distinct)], np.int8)
    wb = np.vectorize(orc.bf16)(w.astype(np.float32).astype(np.float64))
    l_ref, g_ref = orc.net_loss_grad(4, wb, inputs, targets, use_bf16=True)
    assert n % distinct == 0
    assert abs(loss - l_ref) <= 2e-3 / np.sqrt(distinct) * abs(l_ref)
    assert np.linalg.norm(grad - g_ref) <= 2e-2 / np.sqrt(distinct) * np.linalg.norm(g_ref)


# whole configurations in one copy (4, 8, 30), in two (112) and in two slices (32 x 32), patches cut on the host (114, 130);
# blocks at every edge, origins outside the lattice
@pytest.mark.parametrize("L,distinct,repeat", [(4, 7, 1), (8, 40, 1), (30, 60, 1), (112, 40, 1), (32, 40, 1700), (114, 40, 1),
                                               (130, 40, 110)])
def test_loss_grad_slices_and_cut_patches(orc, L, distinct, repeat):
    rng = np.random.default_rng(L + repeat)
    spins = rng.choice(np.array([-1, 1], np.int8), (distinct, L, L))
    edge = np.array([0, 1, 2, 3, L - 1, L - 2, L - 3, L - 4])
    origins = np.stack([rng.permutation(np.resize(edge, distinct)), rng.permutation(np.resize(edge, distinct))], 1).astype(np.int32)
    origins[0] -= L
    origins[-1] += 2 * L
    bh = np.stack([rng.choice([0.5, 1.5, 3.0], distinct), rng.choice([-1.0, 2.5, 3.25], distinct)], 1).astype(np.float32)
    w = orc.random_net(L + 3, scale=0.2)
    p = crbm.Proposal(seed=2)
    p.weights = w
    check_against_oracle(orc, p, w, np.tile(spins, (repeat, 1, 1)), np.tile(origins, (repeat, 1)), np.tile(bh, (repeat, 1)), distinct)


def test_loss_grad_memory_does_not_grow_with_the_lattice():
    """The net reads 100 sites of a configuration: 200 of 1024 x 1024 leave no 210 MB behind on the device."""
    torch = pytest.importorskip("torch")
    p = crbm.Proposal(seed=2)
    p.loss_grad(np.ones((1, 10, 10), np.int8), np.zeros((1, 2), np.int32), np.ones((1, 2), np.float32))
    spins = np.ones((200, 1024, 1024), np.int8)
    free = torch.cuda.mem_get_info()[0]
    p.loss_grad(spins, np.zeros((200, 2), np.int32), np.ones((200, 2), np.float32))
    assert free - torch.cuda.mem_get_info()[0] <= 32 << 20


def test_losses_of_the_steps_before_a_failing_one():
    """A training step whose sweeps fail (here the 32-bit sweep counter) leaves the finished steps' losses written."""
    import ctypes
    n = 64
    s = crbm.Sampler(10, dict(J=[1.0], Jp=[1.0], h=[0.5], beta=[1.0]), n, seed=3, measure_every=0)
    ck = s.save()
    ck[:128].view(np.int64)[6] = 2 ** 32 - 1 - 5   # sweeps so far: two steps of two sweeps still fit
    s.load(ck)
    p = crbm.Proposal(seed=2)
    losses = np.full(4, np.nan, np.float32)
    lib = crbm.load_library()
    rc = lib.crbm_proposal_train(p._p, s._ctx, 4, 32, ctypes.c_float(1e-2), 2,
                                 losses.ctypes.data_as(ctypes.POINTER(ctypes.c_float)))
    assert rc == crbm.CRBM_EINVAL
    assert np.isfinite(losses[:2]).all() and (losses[:2] > 0).all() and np.isnan(losses[2:]).all()
