"""Sorted-tuple operands of the tensor-core path: the first mode products' regathered rows, the
divide's slots (segments packed into 128-row tiles) and the reduction's colexicographic rows, at
the sizes where their tables have remainders: odd n, one mode, segments of length 1, tiles of
several short segments, n just past a row radix, a mode subset of odd size, batches of a few upper
indices, the FP32 form and a slab. Tolerances are the library's bars for the forms (1e-10, 1e-5)."""
from math import comb
from types import SimpleNamespace

import numpy as np
import pytest

import npf_synth as S
import oracle
from tests._util import ROUTES, assert_route, rel_fro, set_route

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def npf():
    from paper_2509_08968_gb300 import build
    build.build()
    import paper_2509_08968_gb300 as m
    return m


def _odd_system(n, N, seed):
    """Conjugate pairs and, for odd n, one real mode; eigenvectors from a real similarity."""
    rng = np.random.default_rng(seed)
    lam, W = np.empty(n, np.complex128), np.zeros((n, n), np.complex128)
    for b in range(n // 2):
        s, w = rng.uniform(-2.0, -0.05), rng.uniform(0.5, 15.0)
        lam[2 * b:2 * b + 2] = s + 1j * w, s - 1j * w
        W[2 * b, 2 * b:2 * b + 2] = 1.0
        W[2 * b + 1, 2 * b:2 * b + 2] = 1j, -1j
    if n % 2:
        lam[-1], W[-1, -1] = rng.uniform(-2.0, -0.05), 1.0
    U = (np.eye(n) + 0.3 / np.sqrt(n) * rng.standard_normal((n, n))) @ W
    return lam, U, np.linalg.inv(U), S.random_packed_tensor_dense_fill(n, N, seed + N)


@pytest.mark.parametrize("route", ROUTES)
@pytest.mark.parametrize("n,N,precision", [
    (1, 3, "split_bf16"), (3, 2, "split_bf16"), (3, 4, "split_bf16"), (9, 3, "split_bf16"),
    (11, 4, "split_bf16"), (33, 3, "split_bf16"), (35, 3, "fp32"), (17, 4, "fp32"), (19, 4, "split_bf16"),
    (65, 3, "split_bf16"), (67, 2, "split_bf16"), (71, 3, "fp32")])
def test_term_odd_sizes(npf, n, N, precision, route):
    lam, U, V, A = _odd_system(n, N, 40 * n + N)
    ref = oracle.psiN(A, n, N, U, V, lam, p1_block=8)
    with npf.Plan(lam, U, V, N, precision=precision) as p:
        set_route(npf, p, route, precision)
        p.set_tensor(N, A)
        assert rel_fro(p.term(N), ref) < (1e-10 if precision == "split_bf16" else 1e-5)
        assert_route(p, route, precision)


@pytest.mark.parametrize("route", ROUTES)
@pytest.mark.parametrize("n,N,m", [(9, 3, 1), (21, 3, 5), (13, 4, 7), (67, 3, 33)])
def test_subset_odd_sizes(npf, n, N, m, route):
    lam, U, V, A = _odd_system(n, N, 50 * n + N)
    modes = np.random.default_rng(n).permutation(n)[:m]
    ref = oracle.psiN_subset(A, n, N, U, V, lam, modes)
    with npf.Plan(lam, U, V, N) as p:
        set_route(npf, p, route)
        p.set_tensor(N, A)
        full = p.term(N)                       # the tables of every mode, then of the subset
        p.set_mode_subset(modes)
        assert rel_fro(p.term(N), ref) < 1e-10
        p.set_mode_subset(None)
        assert rel_fro(p.term(N), full) < 1e-12
        assert_route(p, route)


@pytest.mark.parametrize("n,N,tile", [(5, 3, 16), (70, 3, 16), (90, 2, 16), (100, 2, 16), (75, 2, 32)])
def test_reduction_groups(npf, n, N, tile):
    """One to seven column tiles, of which the last is narrower: the blocks of a reduction group."""
    lam, U, V, A = _odd_system(n, N, 70 * n + N)
    ref = oracle.psiN(A, n, N, U, V, lam, p1_block=8)
    with npf.Plan(lam, U, V, N) as p:
        p.set_option(npf.OPT_TILE_N, tile)
        p.set_tensor(N, A)
        assert rel_fro(p.term(N), ref) < 1e-10


@pytest.mark.parametrize("n,N,m", [(32, 4, 3), (33, 4, 3), (64, 3, 4), (96, 3, 3), (97, 3, 3)])
def test_regather_chunks(npf, n, N, m):
    """Sizes on both sides of the regather's variants (1 to 4 chunks of 32 entries a row)."""
    lam, U, V, A = _odd_system(n, N, 60 * n + N)
    modes = np.random.default_rng(n).permutation(n)[:m]
    ref = oracle.psiN_subset(A, n, N, U, V, lam, modes)
    with npf.Plan(lam, U, V, N) as p:
        p.set_tensor(N, A)
        p.set_mode_subset(modes)
        assert rel_fro(p.term(N), ref) < 1e-10


@pytest.mark.parametrize("route", ROUTES)
@pytest.mark.parametrize("n,N", [(9, 3), (11, 4), (35, 3)])
def test_few_upper_indices_and_new_modes(npf, n, N, route):
    """Batches of a few upper indices, and modal data replaced in a plan whose tables exist."""
    lam, U, V, A = _odd_system(n, N, 60 * n + N)
    lam2, U2, V2, _ = _odd_system(n, N, 61 * n + N)
    rad = 32 if n <= 32 else 64
    dense = 2 * (rad ** (N - 1) * (rad * 4 * 6 + 4)) + 4096
    fixed = n * (-(-comb(n + N - 1, N) // 128) * 128) * 16 + n * comb(n + N - 1, N) * 32
    with npf.Plan(lam2, U2, V2, N) as p:
        set_route(npf, p, route)
        p.set_tensor(N, A)
        p.term(N)
        p.set_option(npf.OPT_MEM_BUDGET, fixed + dense)
        p.set_modes(lam, U, V)
        assert rel_fro(p.term(N), oracle.psiN(A, n, N, U, V, lam, p1_block=8)) < 1e-10
        pre = [n - 1] * (N - 1)
        assert rel_fro(p.modal_slab(N, pre), oracle.h_slab(A, n, N, U, V, lam, pre)) < 1e-10
        p.set_option(npf.OPT_MEM_BUDGET, fixed + dense - 1)   # below one dense upper index: refused
        with pytest.raises(npf.NpfError) as e:
            p.term(N)
        assert e.value.status == npf.NPF_ERR_OOM
        assert_route(p, route)


@pytest.mark.parametrize("n,N,e", [(40, 2, 100), (9, 3, 100), (40, 3, 100), (70, 3, 100), (11, 4, 100), (35, 4, 100)])
def test_any_normalisation_of_the_eigenvectors(npf, n, N, e):
    """U 2^x, V 2^-x is the same system (Psi_N scales as V): the products of weights, 2^(-(N - 1) x), leave
    FP32's range, the sums over them must not."""
    lam, U, V, A = _odd_system(n, N, 30 * n + N)
    ref = oracle.psiN(A, n, N, U, V, lam, p1_block=8)
    for x in (e, -e):
        with npf.Plan(lam, U * 2.0 ** x, V * 2.0 ** -x, N) as p:
            set_route(npf, p, "tensor")
            p.set_tensor(N, A)
            assert rel_fro(p.term(N) * 2.0 ** x, ref) < 1e-10
            assert_route(p, "tensor")


@pytest.mark.parametrize("n,N", [(9, 2), (9, 3), (40, 3), (70, 3), (11, 4)])
def test_any_scale_of_the_tensor(npf, n, N):
    """Psi_N is linear in the tensor: scaled by 2^x beyond FP32's range, it is the same numbers times
    2^x; an interaction's second reduction starts from kept rows."""
    lam, U, V, A = _odd_system(n, N, 20 * n + N)
    ref = oracle.psiN(A, n, N, U, V, lam, p1_block=8)
    # far below the linear part: z(0) = 0.1 Psi, and pNN is linear in the tensor too
    small = SimpleNamespace(n=n, lam=lam, U=U, V=V, tensors={N: A * 2.0 ** -60})
    inter = oracle.interaction_npfs(small, N, 0.1)[N - 1] * 2.0 ** 60
    for x in (110, -110, 300, -300):
        with npf.Plan(lam, U, V, N) as p:
            set_route(npf, p, "tensor")
            p.set_tensor(N, A * 2.0 ** x)
            assert rel_fro(p.term(N) * 2.0 ** -x, ref) < 1e-10
            if x < 0:
                assert rel_fro(p.interaction(N, 0.1)[N - 1] * 2.0 ** -x, inter) < 1e-10
            assert_route(p, "tensor")


def test_interaction_of_a_tiny_excitation(npf):
    """pN3 is of the order delta^3 (1e-36), far below FP32's range for its low parts."""
    n, delta = 27, 1e-12
    lam, U, V, A = _odd_system(n, 3, 8)
    s = SimpleNamespace(n=n, lam=lam, U=U, V=V, tensors={3: A})
    ref = oracle.interaction_npfs(s, 3, delta)
    with npf.Plan(lam, U, V, 3) as p:
        p.set_tensor(3, A)
        got = p.interaction(3, delta)
    assert rel_fro(got[2], ref[2]) < 1e-10 and rel_fro(got[0], ref[0]) < 1e-10


def test_scratch_stays_in_the_budget(npf):
    """The upper indices of a batch are counted by the rows they take, which at 2 slices, order 3 and
    n = 32, 64, 128 are more than the dense rows that a budget is accepted by (17 MB here)."""
    import torch
    n, N = 128, 3
    P = comb(n + N - 1, N)
    lam, U, V, _ = _odd_system(n, 2, 5)
    budget = n * P * 16 + n * (n + 1) // 2 * n * 16 + n * (2 * (128 ** 2 * (128 * 4 * 2 + 4)) + 4096)
    with npf.Plan(lam, U, V, N) as p:
        p.set_option(npf.OPT_SLICES, 2)
        p.set_option(npf.OPT_MEM_BUDGET, budget)
        p.set_tensor(N, torch.zeros((n, P), dtype=torch.float64, device="cuda"))
        free = torch.cuda.mem_get_info()[0]
        assert not p.term(N).any()
        used = free - torch.cuda.mem_get_info()[0]
    assert budget / 2 < used < budget + 8e6   # (and a few MB of tables)


@pytest.mark.parametrize("n", [27, 35])
def test_interaction_shares_the_divided_entries(npf, n):
    """Mode interactions reduce each order twice from one set of divided entries when it runs in one
    batch: against the oracle, again after new modal data, and with a budget of few upper indices,
    where nothing is kept."""
    def system(seed):
        lam, U, V, A3 = _odd_system(n, 3, seed)
        return SimpleNamespace(n=n, lam=lam, U=U, V=V,
                               tensors={2: S.random_packed_tensor_dense_fill(n, 2, 5), 3: A3})
    one, two = system(3), system(4)
    two.tensors = one.tensors
    with npf.Plan(one.lam, one.U, one.V, 3) as p:
        for N, t in one.tensors.items():
            p.set_tensor(N, t)
        for s in (one, two):
            ref = oracle.interaction_npfs(s, 3, 0.1)
            p.set_modes(s.lam, s.U, s.V)
            for _ in range(2):
                assert rel_fro(p.interaction(3, 0.1), ref) < 1e-10
            assert rel_fro(p.term(3), oracle.psiN(s.tensors[3], n, 3, s.U, s.V, s.lam, p1_block=8)) < 1e-10
        p.set_option(npf.OPT_MEM_BUDGET, 60e6 if n > 32 else 20e6)
        assert rel_fro(p.interaction(3, 0.1), ref) < 1e-10


def test_interaction_gives_its_workspace_back(npf):
    """The divided entries that an interaction keeps (168 MB at n = 60, order 3) are workspace: another
    call that needs scratch, a batch's first pass and a caller's budget each free them; a recorded
    batch goes on, and the next interaction is right again."""
    import torch
    s = S.config_n60(0, orders=(3,))
    ref = oracle.interaction_npfs(s, 3, 0.1)
    term = oracle.psiN(s.tensors[3], 60, 3, s.U, s.V, s.lam, p1_block=4)
    free = lambda: torch.cuda.mem_get_info()[0]
    outs = [np.empty((60, 60), np.complex128)]
    with npf.Plan(s.lam, s.U, s.V, 4) as p:
        p.set_tensor(3, s.tensors[3])
        assert rel_fro(p.interaction(3, 0.1), ref) < 1e-10
        kept = free()
        p.set_option(npf.OPT_MEM_BUDGET, 1.5e9)
        assert rel_fro(p.term(3), term) < 1e-10
        assert free() - kept > 150e6
        p.set_option(npf.OPT_MEM_BUDGET, 0)
        for k in range(3):   # eager (gives back), recorded beside a kept workspace, replayed
            assert rel_fro(p.interaction(3, 0.1), ref) < 1e-10
            npf.batch_compute([p], [3], outs)
            assert rel_fro(outs[0], s.U * (s.V + term).T) < 1e-10
