"""The training pass of the surrogate MLP (rows, weight gradients, update) at
the batch sizes where its launches change shape (needs a GB300)."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2311_15088_gb300 import sph

pytestmark = pytest.mark.gpu


def _bf16(a):
    return torch.as_tensor(a, dtype=torch.float32).to(torch.bfloat16)


def _network(seed):
    p = omlp.init_params(seed)
    rng = np.random.default_rng(seed + 1)
    for w, b, n_out, _ in omlp.LAYERS:
        p[w] = _bf16(p[w]).double().numpy()
        p[b] = rng.uniform(-0.1, 0.1, size=n_out)
    return p, np.concatenate([np.concatenate([p[w].ravel(), p[b]]) for w, b, _, _ in omlp.LAYERS]).astype(np.float32)


# 128: one slice per 64 rows; 320 -> 384: uneven slices; 1152: all eight
# slices; 16, 32, 64 rows per CTA up to 16 and 32 x the multiprocessors and
# beyond; a handle
# made for more rows than the batch (longer transposed rows)
@pytest.mark.parametrize("B,max_batch", [(128, 128), (384, 384), (384, 2048), (1152, 1152), (2432, 2432), (2560, 2560), (4864, 4992),
                                         (4992, 4992), (9984, 9984)])
def test_gradients_at_batch_edges(B, max_batch):
    p, packed = _network(61)
    rng = np.random.default_rng(B)
    x = _bf16(rng.normal(size=(B, omlp.D_IN))).double().numpy()
    dy = (rng.normal(size=(B, omlp.D_OUT)) / B).astype(np.float32)
    m = sph.Mlp(max_batch)
    m.set_params(torch.from_numpy(packed))
    g = m.gradients(_bf16(x).cuda(), torch.from_numpy(dy).cuda()).double().cpu().numpy()
    assert m.status() == 0
    ref = omlp.backward(p, omlp.forward(p, x), dy.astype(np.float64))
    o = 0
    for w, b, n_out, n_in in omlp.LAYERS:
        for name, n in ((w, n_out * n_in), (b, n_out)):
            a, r = g[o:o + n], ref[name].ravel()
            o += n
            # every activation and gradient entering a product is rounded to
            # BF16 (2^-9 relative); at most seven such roundings in a chain
            assert np.linalg.norm(a - r) <= 7 * 2.0 ** -9 * np.linalg.norm(r), (name, np.linalg.norm(a - r) / np.linalg.norm(r))


@pytest.mark.parametrize("B", [128, 640, 3072, 5120])
def test_loss_and_phases_at_batch_edges(B):
    """The loss of both phases against the oracle's, and what each phase
    leaves alone; the same step from the same state gives the same bits."""
    p, packed = _network(71)
    rng = np.random.default_rng(B + 1)
    x = _bf16(rng.normal(size=(B, omlp.D_IN))).double().numpy()
    t = rng.normal(size=(B, 4)).astype(np.float32)
    xb, tt = _bf16(x).cuda(), torch.from_numpy(t).cuda()
    y = omlp.forward(p, x)["y"]
    want = (0.5 * np.sum((y[:, :3] - t[:, :3]) ** 2) / B, 0.5 * np.sum((y[:, 3] - t[:, 3]) ** 2) / B)
    for phase in (0, 1):
        out = []
        for _ in range(2):
            m = sph.Mlp(B)
            m.set_params(torch.from_numpy(packed))
            loss = float(m.train_step(xb, tt, 1e-3, phase).item())
            assert m.status() == 0
            out.append((loss, m.get_params().cpu().numpy()))
        assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])
        # a loss of squares of outputs that carry the forward's BF16 error (2e-2)
        assert abs(out[0][0] - want[phase]) <= 4e-2 * want[phase]
        w4 = sum(n_out * n_in + n_out for _, _, n_out, n_in in omlp.LAYERS[:3])
        head = np.zeros(len(packed), bool)
        head[w4 + 3 * 256:w4 + 4 * 256] = True
        head[w4 + 16 * 256 + 3] = True
        same = out[0][1] == packed
        assert np.all(same[~head]) if phase == 1 else np.all(same[head])
        assert not np.any(same[head]) if phase == 1 else not np.all(same[~head])
