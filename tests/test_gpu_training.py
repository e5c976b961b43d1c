"""The training pass of the per-site network at the row counts where its tiling changes: partial
tiles of 4 and of 8 rows, one and several row splits, more rows than activations are kept for at
once, and minibatches that do not divide the rows.

Bounds.  Every gradient entry is a sum over the rows of products of FP32 values, each of which comes
from at most three chained dot products of up to 128 FP32 terms; with unit roundoff u = 6e-8 and
random rounding errors that is 3 sqrt(128) u = 2e-6 of the gradient's norm, plus the fast exponential
of the activations (2 ulp), so 2e-5 leaves a factor of about ten.  An AdamW step divides the gradient
by its own running size, so a parameter's update carries the gradient's relative error; over the few
steps here the updates stay below 1e-2 of the parameters' norm, and 2e-5 bounds the difference again."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2509_24742_gb300 import srbe

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b)


def rows(n, seed):
    rng = np.random.default_rng(seed)
    D = np.abs(rng.normal(0.3, 0.2, (n, srbe.N_DESC))).astype(np.float32)
    T = (0.03 * np.tanh(D @ rng.normal(size=srbe.N_DESC) / 4)).astype(np.float32)
    return D, T


@pytest.fixture(scope="module")
def ctx():
    with srbe.Context((2.0, 2.0, 12.0), 3.5, 0.05, 1.2, 10, 2) as c:
        yield c


@pytest.mark.parametrize("n", [1, 3, 4, 5, 511, 608, 609, 1024, 1025, 2051, 65539])
def test_gradients_match_oracle(ctx, n):
    D, T = rows(n, n)
    ctx.mlp_init(seed=3)
    P = ctx.mlp_params()
    g, loss = ctx.mlp_gradients(D, T)
    ref_loss, ref = omlp.loss_and_grad(P, D, T)
    assert rel(g, ref) < 2e-5
    assert abs(loss - ref_loss) < 2e-5 * ref_loss


@pytest.mark.parametrize("n,batch", [(700, 256), (2500, 1030), (37, 64), (1200, 1200)])
def test_training_matches_oracle_steps(ctx, n, batch):
    D, T = rows(n, 7 * n + batch)
    ctx.mlp_init(seed=5)
    P = ctx.mlp_params().astype(np.float64)
    loss = ctx.mlp_train(D, T, epochs=2, batch=batch, lr=1e-4, weight_decay=1e-4, seed=9)
    got = ctx.mlp_params()
    k = omlp.N_TRAIN
    P[k:] = got[k:]                       # the data's standardisation, as the library stored it
    perms = shuffles(n, 2, 9)
    m1, m2, t, ref_loss = np.zeros(k), np.zeros(k), 0, 0.0
    for perm in perms:
        tot = 0.0
        for b0 in range(0, n, batch):
            r = perm[b0:b0 + batch]
            l, g = omlp.loss_and_grad(P, D[r], T[r])
            tot += l * len(r)
            t += 1
            m1 = 0.9 * m1 + 0.1 * g
            m2 = 0.999 * m2 + 0.001 * g * g
            P[:k] -= 1e-4 * ((m1 / (1 - 0.9 ** t)) / (np.sqrt(m2 / (1 - 0.999 ** t)) + 1e-8) + 1e-4 * P[:k])
        ref_loss = tot / n
    assert rel(got, P) < 2e-5
    assert abs(loss - ref_loss) < 1e-4 * ref_loss


def test_prediction_at_tile_edges(ctx):
    """A row's prediction does not depend on the call it is in: one row, partial tiles, one tile per SM, the
    first tile of the second group of warps and several tiles per group give the same bits; new parameters
    are seen at once.  (The values against the oracle: test_gpu_learned.)"""
    D, _ = rows(128 * 456 + 5, 3)
    last = None
    for seed in (3, 4):
        ctx.mlp_init(seed=seed)
        y = ctx.mlp_predict(D)
        assert last is None or not np.array_equal(y, last)
        for n in (1, 127, 128, 129, 300, 128 * 152, 128 * 152 + 1):
            assert np.array_equal(ctx.mlp_predict(D[:n]), y[:n])
        # rows 300 at a time (at most three tiles, all of first groups), against the long call
        for r0 in (128 * 152 - 10, 128 * 304 + 7, 128 * 456 - 295):
            assert np.array_equal(ctx.mlp_predict(D[r0:r0 + 300]), y[r0:r0 + 300])
        last = y


@pytest.mark.parametrize("n", [65535, 65536, 66560, 131072, 132098])
def test_gradients_at_the_chunk_edges(ctx, n):
    """One chunk of activations less a row, a whole one, one split more, two, and a part of the third."""
    D, T = rows(n, n)
    ctx.mlp_init(seed=3)
    P = ctx.mlp_params()
    g, loss = ctx.mlp_gradients(D, T)
    ref_loss, ref = omlp.loss_and_grad(P, D, T)
    assert rel(g, ref) < 2e-5
    assert abs(loss - ref_loss) < 2e-5 * ref_loss


def test_training_scratch_is_bounded():
    """Beside the rows themselves a training or gradient call holds at most 172 MB on the device, whatever their
    number and the minibatch (activations 156 MB, split gradients 7 MB, their sums, the device's 2 MB pages)."""
    import torch
    D, T = rows(300000, 1)
    with srbe.Context((2.0, 2.0, 12.0), 3.5, 0.05, 1.2, 10, 2) as c:
        c.mlp_init(seed=3)
        c.mlp_gradients(D[:100], T[:100])
        c.mlp_predict(D)                       # the rows' own buffer
        free = torch.cuda.mem_get_info()[0]
        c.mlp_gradients(D, T)
        c.mlp_train(D, T, epochs=1, batch=300000, lr=1e-4, seed=2)
        assert free - torch.cuda.mem_get_info()[0] <= 172 * 10 ** 6


def shuffles(n, epochs, seed):
    """Fisher-Yates rows of every epoch, one Philox4x64-10 word per exchange."""
    out, ctr = [], 0
    for e in range(epochs):
        perm = np.arange(n)
        for i in range(n - 1, 0, -1):
            # numpy's generator advances its 256-bit counter before the first block
            c = ctr + (e << 64) + (0x53485546 << 192) - 1
            counter = np.array([(c >> (64 * k)) & (2 ** 64 - 1) for k in range(4)], np.uint64)
            w = int(np.random.Philox(key=np.array([seed, 0x5352424500000004], np.uint64),
                                     counter=counter).random_raw())
            ctr += 1
            j = w % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        out.append(perm)
    return out
