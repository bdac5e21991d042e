"""The tensor-core pipeline's bounded waits: a test hook withholds the first completion signal,
the epilogue's wait runs out (~2 s), the call reports NPF_ERR_TIMEOUT, and the CUDA context stays
usable (no fault, trap or hang is involved)."""
import time

import numpy as np
import pytest

import npf_synth as S
import oracle
from tests._util import make_plan, rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def npf():
    from paper_2509_08968_gb300 import build
    build.build()
    import paper_2509_08968_gb300 as m
    return m


def test_bounded_wait_reports_timeout_and_recovers(npf):
    sysm = S.config_small(0, orders=(2,))
    ref = oracle.psiN(sysm.tensors[2], 10, 2, sysm.U, sysm.V, sysm.lam, p1_block=10)
    with make_plan(npf, sysm, 2, "split_bf16") as p:
        p.set_option(npf.OPT_SLICES, 6)   # the tensor-core route at this size
        p.set_option(npf.OPT_DEBUG_STALL, 1)
        t0 = time.time()
        with pytest.raises(npf.NpfError) as e:
            p.term(2)
        assert e.value.status == npf.NPF_ERR_TIMEOUT
        assert time.time() - t0 < 60
        p.set_option(npf.OPT_DEBUG_STALL, 0)
        assert rel_fro(p.term(2), ref) < 1e-10


def test_a_failed_call_leaves_its_outputs_alone(npf):
    """Nothing is written to a call's outputs when a wait gave up: host and device outputs keep what
    they held (a batch's first pass included; its replays read the flag at the same place)."""
    import torch
    sysm = S.config_small(0, orders=(2, 3))
    n = 10
    with make_plan(npf, sysm, 3, "split_bf16") as p:
        p.set_option(npf.OPT_SLICES, 6)   # the tensor-core route at this size
        good = p.interaction(3, 0.1)
        p.set_option(npf.OPT_DEBUG_STALL, 1)
        host = np.full((3, n, n), 7.0 + 5.0j)
        dev = torch.full((n, n), 7.0 + 5.0j, dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        for call in (lambda: p.compute(3, host[0]), lambda: p.compute(3, dev), lambda: p.term(2, dev),
                     lambda: p.term(3, host[0]), lambda: p.term_rows(3, 0, n, host[0]), lambda: p.interaction(3, 0.1, host),
                     lambda: npf.batch_compute([p], [3], [host[0]])):
            with pytest.raises(npf.NpfError) as e:
                call()
            assert e.value.status == npf.NPF_ERR_TIMEOUT
            assert (host == 7.0 + 5.0j).all() and bool((dev == 7.0 + 5.0j).all())
        p.set_option(npf.OPT_DEBUG_STALL, 0)
        assert rel_fro(p.interaction(3, 0.1), good) < 1e-10
        assert rel_fro(good, oracle.interaction_npfs(sysm, 3, 0.1)) < 1e-10


def test_a_failed_tuning_is_not_kept(npf):
    """The autotuner's terms that gave up leave no tile width behind for the process."""
    n = 22
    sysm = S.modal_system(n, 5)
    sysm.tensors[2] = S.random_packed_tensor(n, 2, 6)
    with make_plan(npf, sysm, 2, "split_bf16") as p:
        p.set_option(npf.OPT_TILE_N, 0)
        p.set_option(npf.OPT_DEBUG_STALL, 1)
        with pytest.raises(npf.NpfError) as e:
            p.term(2)
        assert e.value.status == npf.NPF_ERR_TIMEOUT
        assert npf.tuned_tile(n, 2, "split_bf16") == 0
        p.set_option(npf.OPT_DEBUG_STALL, 0)
        ref = oracle.psiN(sysm.tensors[2], n, 2, sysm.U, sysm.V, sysm.lam, p1_block=n)
        assert rel_fro(p.term(2), ref) < 1e-10
        assert npf.tuned_tile(n, 2, "split_bf16") in (16, 32)
