"""Device weights and gradients on an ensemble whose stream does not wait for the legacy stream: what
the legacy stream has queued on them comes first (the weights are still being written; the
destination is still being read)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_device_buffers_follow_the_legacy_stream():
    import torch

    import paper_2509_08968_gb300 as npf
    from paper_2509_08968_gb300 import build
    build.build()
    from paper_2509_08968_gb300.surrogate import init_weights
    lib = npf.load()
    widths = [4, 32, 16]
    W = init_weights(widths, 2, 3)
    side = torch.cuda.Stream()
    real = torch.tensor(W, device="cuda")
    dst = torch.zeros_like(real)
    late, seen = torch.zeros_like(real), torch.empty_like(real)
    torch.cuda.synchronize()
    wd = (ctypes.c_int * 3)(*widths)
    torch.cuda._sleep(200_000_000)         # about 0.1 s on the legacy stream
    late.copy_(real)
    h = ctypes.c_void_p(lib.npf_mlp_create(2, 2, wd, npf._ptr(late), ctypes.c_void_p(side.cuda_stream)))
    try:
        torch.cuda._sleep(200_000_000)
        seen.copy_(dst)                    # reads the old contents
        assert lib.npf_mlp_get_weights(h, npf._ptr(dst)) == npf.NPF_OK
        with torch.cuda.stream(side):      # (the call has returned: the weights are there)
            got = dst.clone()
        torch.cuda.synchronize()
        assert not seen.any() and np.array_equal(got.cpu().numpy(), W)
        X, T = torch.rand(8, 4, device="cuda"), torch.rand(8, 16, device="cuda")
        loss = np.empty(2, np.float32)
        torch.cuda.synchronize()
        torch.cuda._sleep(200_000_000)
        seen.copy_(dst)
        assert lib.npf_mlp_loss_grad(h, 8, npf._ptr(X), npf._ptr(T), npf._ptr(dst), npf._ptr(loss)) == npf.NPF_OK
        torch.cuda.synchronize()
        assert np.array_equal(seen.cpu().numpy(), W) and not np.array_equal(dst.cpu().numpy(), W)
    finally:
        lib.npf_mlp_destroy(h)
