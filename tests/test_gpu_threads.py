"""Two host threads with a handle each: one records and replays batches, the other makes plans whose
scratch grows from call to call. Neither may disturb the other."""
import threading

import numpy as np
import pytest

import npf_synth as S
import oracle
from tests._util import rel_fro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def npf():
    from paper_2509_08968_gb300 import build
    build.build()
    import paper_2509_08968_gb300 as m
    return m


def test_scratch_grows_beside_a_recording(npf):
    big, small = S.config_blocks(28, 1, orders=(3,)), S.modal_system(8, 2)
    small.tensors.update({N: S.random_packed_tensor(8, N, N) for N in (2, 3, 4)})
    want = {N: oracle.psiN(small.tensors[N], 8, N, small.U, small.V, small.lam, p1_block=8) for N in (2, 4)}
    plans = []
    for _ in range(64):
        plans.append(npf.Plan(big.lam, big.U, big.V, 3))
        plans[-1].set_tensor(3, big.tensors[3])
    outs = [np.empty((28, 28), np.complex128) for _ in plans]
    ref = oracle.npf(big.U, big.V, oracle.psiN(big.tensors[3], 28, 3, big.U, big.V, big.lam, p1_block=8))
    errors, stop, rounds = [], threading.Event(), [0]

    def grow():
        try:
            while not stop.is_set():
                with npf.Plan(small.lam, small.U, small.V, 4, precision="fp64") as p:
                    for N, t in small.tensors.items():
                        p.set_tensor(N, t)
                    for N in (2, 3, 4):   # each needs more scratch than the one before
                        got = p.term(N)
                        assert N == 3 or rel_fro(got, want[N]) < 1e-12
                rounds[0] += 1
        except Exception as e:   # (reported by the main thread)
            errors.append(e)

    t = threading.Thread(target=grow)
    t.start()
    try:
        for k in range(30):
            plans[k % 64].set_option(npf.OPT_EPS, 1e-8)   # a new list: run eagerly, then recorded
            for _ in range(2):
                npf.batch_compute(plans, [3] * 64, outs)
                assert all(rel_fro(o, ref) < 1e-10 for o in outs[::21])
    finally:
        stop.set()
        t.join()
        for p in plans:
            p.close()
    assert not errors, errors[0]
    assert rounds[0] > 10
