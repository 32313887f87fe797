"""The network called from other host threads than the one that made it (needs
a GB300)."""
import threading

import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2311_15088_gb300 import sph

pytestmark = pytest.mark.gpu


def _packed():
    p = omlp.init_params(5)
    return torch.from_numpy(np.concatenate([np.concatenate([p[w].ravel(), p[b]]) for w, b, _, _ in omlp.LAYERS])
                            .astype(np.float32))


@pytest.mark.parametrize("call", ["forward", "gradients", "train_step"])
def test_first_cuda_call_of_a_thread(call):
    """A host thread whose first CUDA call is the network's (its buffers were
    made elsewhere, so it has not bound a context)."""
    B, s = 256, torch.cuda.current_stream().cuda_stream
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((B, sph.SPH_MLP_IN), generator=g, device="cuda").to(torch.bfloat16)
    t = torch.randn((B, 16 if call == "gradients" else 4), generator=g, device="cuda")
    out, rc = [], []
    for threaded in (False, True):
        m = sph.Mlp(B)
        m.set_params(_packed())
        o = torch.zeros(sph.SPH_MLP_PARAMS, device="cuda")
        torch.cuda.synchronize()

        def run():
            if call == "forward":
                rc.append(sph._lib.sph_mlp_forward(m.handle, x.data_ptr(), B, o.data_ptr(), s))
            elif call == "gradients":
                rc.append(sph._lib.sph_mlp_gradients(m.handle, x.data_ptr(), t.data_ptr(), B, o.data_ptr(), s))
            else:
                rc.append(sph._lib.sph_mlp_train_step(m.handle, x.data_ptr(), t.data_ptr(), B, 0, 1e-3, o.data_ptr(), s))

        if threaded:
            th = threading.Thread(target=run)
            th.start()
            th.join()
        else:
            run()
        torch.cuda.synchronize()
        assert m.status() == 0
        out += [o, m.get_params()]
    assert rc == [0, 0]
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3]) and bool(out[0].any())
