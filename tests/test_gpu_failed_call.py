"""A call that fails after it has queued work returns once that work has finished, as every call does
(an order refused for its memory behind an order that ran), so that the caller may free or reuse what
the work reads and the plan may change streams."""
import time

import numpy as np
import pytest

import npf_synth as S
from tests._util import rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def npf():
    from paper_2509_08968_gb300 import build
    build.build()
    import paper_2509_08968_gb300 as m
    return m


@pytest.mark.parametrize("call", ["compute", "interaction"])
def test_refused_order_waits_for_the_others(npf, call):
    import torch
    n = 60
    sysm = S.config_n60(0, orders=(3,))
    stream = torch.cuda.Stream()
    with npf.Plan(sysm.lam, sysm.U, sysm.V, 4) as p:
        p.set_tensor(3, sysm.tensors[3])
        p.set_tensor(4, torch.zeros((n, S.packed_count(n, 4)), dtype=torch.float64, device="cuda"))
        ref = p.term(3)
        p.set_stream(stream.cuda_stream)
        p.set_option(npf.OPT_MEM_BUDGET, 1e9)   # order 3 in one batch; order 4 needs more
        p.term(3)
        for _ in range(2):   # (the first one builds order 4's tables, which waits for the device)
            with pytest.raises(npf.NpfError) as e:
                p.compute(4) if call == "compute" else p.interaction(4, 0.1)
            assert stream.query()
            assert e.value.status == npf.NPF_ERR_OOM
        assert rel_fro(p.term(3), ref) < 1e-12


def test_refused_system_waits_for_the_batch(npf):
    """Eight streams: the FP64 systems in front of a refused one run without a wait of their own."""
    import torch
    n, N = 60, 3
    sysm = S.config_n60(1, orders=(N,))
    plans = []
    for k in range(2):
        plans.append(npf.Plan(sysm.lam, sysm.U, sysm.V, N, precision="fp64"))
        plans[-1].set_tensor(N, sysm.tensors[N])
    plans[0].term(N)
    t0 = time.perf_counter()
    plans[0].term(N)
    alone = time.perf_counter() - t0
    plans[1].set_option(npf.OPT_MEM_BUDGET, 1e6)
    outs = [np.full((n, n), 3.0 + 0.0j) for _ in plans]
    torch.cuda.synchronize()
    with pytest.raises(npf.NpfError) as e:
        npf.batch_compute(plans, [N, N], outs)
    t0 = time.perf_counter()
    torch.cuda.synchronize()   # (the streams are the library's own)
    assert time.perf_counter() - t0 < 0.25 * alone
    assert e.value.status == npf.NPF_ERR_OOM
    assert all((o == 3.0).all() for o in outs)
    for p in plans:
        p.close()
