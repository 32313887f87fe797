"""Every element of the weight and bias gradients of a batch cut into uneven
slices (14 blocks of 64 rows: 3, 3, 3, 3, 2) against the FP64 oracle (needs a
GB300).

A gradient element is a sum over the batch of an output's delta times an
input's activation.  Each carries at most seven BF16 roundings (2^-9 relative),
so by Cauchy and Schwarz the element is within 7 2^-9 of the product of the two
columns' norms.  Over 896 rows with deltas of either sign an element is about a
thirtieth of that product: an element of another place is outside the bound."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2311_15088_gb300 import sph

pytestmark = pytest.mark.gpu

B, REL = 896, 7 * 2.0 ** -9


def _bf16(a):
    return torch.as_tensor(a, dtype=torch.float32).to(torch.bfloat16)


@pytest.mark.parametrize("max_batch", [896, 1024])
def test_every_gradient_element(max_batch):
    p = omlp.init_params(23)
    rng = np.random.default_rng(24)
    for w, b, n_out, _ in omlp.LAYERS:
        p[w] = _bf16(p[w]).double().numpy()
        p[b] = rng.uniform(-0.1, 0.1, size=n_out).astype(np.float32).astype(np.float64)
    packed = np.concatenate([np.concatenate([p[w].ravel(), p[b]]) for w, b, _, _ in omlp.LAYERS]).astype(np.float32)
    x = _bf16(rng.normal(size=(B, omlp.D_IN))).double().numpy()
    dy = (rng.normal(size=(B, omlp.D_OUT)) / B).astype(np.float32)
    m = sph.Mlp(max_batch)
    m.set_params(torch.from_numpy(packed))
    g = m.gradients(_bf16(x).cuda(), torch.from_numpy(dy).cuda()).double().cpu().numpy()
    assert m.status() == 0
    c = omlp.forward(p, x)
    starts = np.cumsum([0] + [n_out * n_in + n_out for _, _, n_out, n_in in omlp.LAYERS])
    delta = dy.astype(np.float64)
    for k in range(4, 0, -1):
        w, _, n_out, n_in = omlp.LAYERS[k - 1]
        h = c["x"] if k == 1 else c[f"h{k - 1}"]
        at = starts[k - 1]
        got = g[at:at + n_out * n_in].reshape(n_out, n_in)
        want = delta.T @ h
        norms = np.linalg.norm(delta, axis=0)
        bound = REL * norms[:, None] * np.linalg.norm(h, axis=0)[None, :]
        assert np.all(np.abs(got - want) <= bound), (w, np.max(np.abs(got - want) / bound))
        # the bound tells an element from its neighbours in either direction
        for axis in (0, 1):
            assert np.mean(np.abs(np.roll(want, 1, axis) - want) > bound) > 0.5
        got_b, want_b = g[at + n_out * n_in:at + n_out * n_in + n_out], delta.sum(axis=0)
        assert np.all(np.abs(got_b - want_b) <= REL * norms * np.sqrt(B))
        if k > 1:
            delta = (delta @ p[w]) * omlp.gelu_grad(c[f"z{k - 1}"])
