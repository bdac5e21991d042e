"""The FP64 chain in shared memory (k_chain.cu): the FP64 form at orders 2 to 4 and the small
systems of the tensor-core forms, on both sides of the sizes where the route changes, with odd n,
row ranges, a mode subset, no divide, weights other than Psi, batches and a budget that leaves
the general path. Tolerance: 1e-12 for FP64 sums of at most 40^4 terms (the FP64 bar of the library)."""
import threading
from types import SimpleNamespace

import numpy as np
import pytest

import oracle
from tests._util import ran, rel_fro
from tests.test_gpu_sorted import _odd_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def npf():
    from paper_2509_08968_gb300 import build
    build.build()
    import paper_2509_08968_gb300 as m
    return m


@pytest.mark.parametrize("n,N", [(1, 2), (2, 3), (3, 4), (25, 2), (26, 2), (16, 3), (17, 3), (10, 4), (11, 4),
                                 (45, 2), (40, 3), (21, 4)])
def test_both_sides_of_the_rule(npf, n, N):
    lam, U, V, A = _odd_system(n, N, 70 * n + N)
    ref = oracle.psiN(A, n, N, U, V, lam, p1_block=8)
    for precision, tol in (("fp64", 1e-12), ("split_bf16", 1e-10), ("fp32", 1e-5)):
        with npf.Plan(lam, U, V, N, precision=precision) as p:
            p.set_tensor(N, A)
            p.set_option(npf.OPT_PROFILE, 1)
            got = p.term(N)
            assert rel_fro(got, ref) < tol
            chain = precision == "fp64" or n <= {2: 25, 3: 16, 4: 10}[N]
            assert ("fp64_chain" in ran(p)) == chain
            if precision == "fp64":
                assert np.array_equal(got, p.term(N))   # fixed order of summation
                p.set_option(npf.OPT_DIVIDE, 0)
                ref0 = oracle.psiN(A, n, N, U, V, lam, divide=False, p1_block=8)
                assert rel_fro(p.term(N), ref0) < tol


@pytest.mark.parametrize("n,N", [(9, 2), (13, 2), (9, 3), (11, 3), (7, 4), (9, 4)])
def test_rows_subset_weights_and_batch(npf, n, N):
    lam, U, V, A = _odd_system(n, N, 80 * n + N)
    sysm = SimpleNamespace(n=n, lam=lam, U=U, V=V, tensors={N: A})
    ref = oracle.psiN(A, n, N, U, V, lam, p1_block=8)
    with npf.Plan(lam, U, V, N) as p, npf.Plan(lam, U, V, N, precision="fp64") as q:
        for x in (p, q):
            x.set_tensor(N, A)
            rows = x.term_rows(N, 2, 5)
            assert rel_fro(rows[2:5], ref[2:5]) < 1e-12
            assert not rows[:2].any() and not rows[5:].any()
            inter = x.interaction(N, 0.3)
            assert rel_fro(inter, oracle.interaction_npfs(sysm, N, 0.3)) < 1e-12
        outs = [np.empty((n, n), np.complex128) for _ in range(2)]
        for _ in range(3):   # eager, recorded, replayed
            npf.batch_compute([p, q], [N, N], outs)
            for o, tol in zip(outs, (1e-10, 1e-12)):   # (in a batch p leaves the chain at smaller n)
                assert rel_fro(o, U * (V + ref).T) < tol
        modes = [0, n - 1, 2]
        p.set_mode_subset(modes)
        assert rel_fro(p.term(N), oracle.psiN_subset(A, n, N, U, V, lam, modes)) < 1e-12


def test_budget_below_the_chain_uses_the_general_path(npf):
    n, N = 20, 3
    lam, U, V, A = _odd_system(n, N, 91)
    ref = oracle.psiN(A, n, N, U, V, lam, p1_block=8)
    with npf.Plan(lam, U, V, N, precision="fp64") as p:
        p.set_tensor(N, A)
        p.set_option(npf.OPT_MEM_BUDGET, (2 * n ** N + n ** (N - 1)) * 16)
        assert rel_fro(p.term(N), ref) < 1e-12
        p.set_option(npf.OPT_MEM_BUDGET, (2 * n ** N + n ** (N - 1)) * 16 - 1)
        with pytest.raises(npf.NpfError) as e:
            p.term(N)
        assert e.value.status == npf.NPF_ERR_OOM


def test_sizes_side_by_side(npf):
    """The chain's shared memory grows with n (54 KB at n = 45, 2 KB at n = 8, order 3): launches of one
    size do not change what another may have, be it in another thread or in a recorded batch."""
    N = 3
    systems = [_odd_system(n, N, 90 + n) for n in (45, 8)]
    refs = [oracle.psiN(A, len(lam), N, U, V, lam, p1_block=8) for lam, U, V, A in systems]
    plans = []
    for lam, U, V, A in systems:
        plans.append(npf.Plan(lam, U, V, N, precision="fp64"))
        plans[-1].set_tensor(N, A)
    outs = [np.empty(r.shape, np.complex128) for r in refs]
    for _ in range(3):   # eager, recorded, replayed
        npf.batch_compute(plans, [N, N], outs)
        for (lam, U, V, A), r, o in zip(systems, refs, outs):
            assert rel_fro(o, U * (V + r).T) < 1e-12
    errors, stop = [], threading.Event()

    def small():
        try:
            while not stop.is_set():
                plans[1].term(N)
        except npf.NpfError as e:
            errors.append(e)

    t = threading.Thread(target=small)
    t.start()
    try:
        for _ in range(300):
            got = plans[0].term(N)
    finally:
        stop.set()
        t.join()
        for p in plans:
            p.close()
    assert not errors
    assert rel_fro(got, refs[0]) < 1e-12
