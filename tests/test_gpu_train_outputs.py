"""Where the training calls' results go: gradients and loss at any byte address
(needs a GB300)."""
import pytest
import torch

from paper_2311_15088_gb300 import sph, surrogate

pytestmark = pytest.mark.gpu

B, N = 256, sph.SPH_MLP_PARAMS


@pytest.mark.parametrize("offset", [0, 1, 2, 4, 12])
def test_results_at_any_byte_offset(offset):
    """The bytes at an offset are those of an aligned call, and no byte beside
    them is written."""
    g = torch.Generator(device="cuda").manual_seed(9)
    x = torch.randn((B, sph.SPH_MLP_IN), generator=g, device="cuda").to(torch.bfloat16)
    dy = torch.randn((B, sph.SPH_MLP_OUT), generator=g, device="cuda")
    t = torch.randn((B, 4), generator=g, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    m, ref = sph.Mlp(B), sph.Mlp(B)
    for net in (m, ref):
        net.set_params(torch.from_numpy(surrogate.init_params(3)))
    want = ref.gradients(x, dy)
    grads = torch.full((4 * N + 32,), 7, dtype=torch.uint8, device="cuda")
    sph.sph_mlp_gradients(m.handle, x.data_ptr(), dy.data_ptr(), B, grads.data_ptr() + offset, s)
    assert torch.equal(grads[offset:offset + 4 * N], want.view(torch.uint8))
    assert bool((grads[:offset] == 7).all()) and bool((grads[offset + 4 * N:] == 7).all())
    loss = torch.full((32,), 7, dtype=torch.uint8, device="cuda")
    for phase in (0, 1):
        want = ref.train_step(x, t, 1e-3, phase).clone()
        sph.sph_mlp_train_step(m.handle, x.data_ptr(), t.data_ptr(), B, phase, 1e-3, loss.data_ptr() + offset, s)
        assert torch.equal(loss[offset:offset + 4], want.view(torch.uint8))
        assert bool((loss[:offset] == 7).all()) and bool((loss[offset + 4:] == 7).all())
    assert torch.equal(m.get_params(), ref.get_params()) and m.status() == 0
