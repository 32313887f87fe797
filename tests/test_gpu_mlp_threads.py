"""The network called from other host threads than the one that made it, and from
several at once (needs a GB300)."""
import threading

import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2311_15088_gb300 import sph

pytestmark = pytest.mark.gpu

THREADS = 4


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


# rows for 16 and 32 rows a CTA and for the 128-row tiles
@pytest.mark.parametrize("rows_per_sm", [4, 20, 40])
def test_first_calls_of_a_handle_from_several_threads(rows_per_sm):
    B = rows_per_sm * torch.cuda.get_device_properties(0).multi_processor_count // 128 * 128
    packed = _packed()
    g = torch.Generator(device="cuda").manual_seed(B)
    x = [torch.randn((B, sph.SPH_MLP_IN), generator=g, device="cuda").to(torch.bfloat16) for _ in range(THREADS)]
    m = sph.Mlp(B)
    m.set_params(packed)
    want = [m.forward(v) for v in x]
    streams = [torch.cuda.Stream() for _ in range(THREADS)]
    for _ in range(8):
        m = sph.Mlp(B)
        m.set_params(packed)
        torch.cuda.synchronize()
        got, start = [None] * THREADS, threading.Barrier(THREADS)

        def first_call(k):
            with torch.cuda.stream(streams[k]):
                start.wait()
                got[k] = m.forward(x[k])

        threads = [threading.Thread(target=first_call, args=(k,)) for k in range(THREADS)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        assert m.status() == 0
        assert all(torch.equal(a, b) for a, b in zip(got, want))
