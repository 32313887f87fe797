"""Inference at the row numbers where its launch changes: 16 and 32 rows a CTA
up to 16 and 32 times the multiprocessors, 128-row tiles beyond (needs a
GB300)."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2311_15088_gb300 import sph

pytestmark = pytest.mark.gpu


def _bf16(a):
    return torch.as_tensor(a, dtype=torch.float32).to(torch.bfloat16)


# batches are multiples of 128: the last of a kernel and the first of the next
@pytest.mark.parametrize("per_sm,more", [(0, 1), (16, 0), (16, 1), (32, 0), (32, 1)])
def test_forward_at_the_edges_of_each_kernel(per_sm, more):
    """The outputs against the FP64 oracle (the bounds of the other forward
    tests: BF16 operands through four layers), and bit for bit what the same
    rows give inside a batch of 128-row tiles."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = per_sm * sms // 128 * 128 + 128 * more
    big = 40 * sms // 128 * 128 + 128
    assert B < big
    p = omlp.init_params(17)
    rng = np.random.default_rng(B)
    for w, b, n_out, _ in omlp.LAYERS:
        p[w] = _bf16(p[w]).double().numpy()
        p[b] = rng.uniform(-0.1, 0.1, size=n_out).astype(np.float32).astype(np.float64)
    packed = np.concatenate([np.concatenate([p[w].ravel(), p[b]]) for w, b, _, _ in omlp.LAYERS]).astype(np.float32)
    x = _bf16(rng.normal(size=(big, omlp.D_IN)))
    m = sph.Mlp(big)
    m.set_params(torch.from_numpy(packed))
    y = m.forward(x[:B].cuda())
    assert torch.equal(y, m.forward(x.cuda())[:B]) and m.status() == 0
    ref = omlp.forward(p, x[:B].double().numpy())["y"]
    y = y.double().cpu().numpy()
    assert np.linalg.norm(y - ref) <= 2e-2 * np.linalg.norm(ref)
    assert np.all(np.abs(y - ref) <= 2e-2 * np.abs(ref).max())
