import numpy as np


def rel_fro(got, ref):
    """Relative Frobenius error ||got - ref||_F / ||ref||_F."""
    got = np.asarray(got)
    ref = np.asarray(ref)
    return float(np.linalg.norm((got - ref).ravel()) / np.linalg.norm(ref.ravel()))


# Small systems of the tensor-core forms run the FP64 chain by default: "tensor" gives the form's own slice
# count as an option, which keeps them on the tensor-core path.
ROUTES = ("default", "tensor")


def set_route(npf, p, route, precision="split_bf16"):
    if route == "tensor" and precision != "fp64":
        p.set_option(npf.OPT_SLICES, 4 if precision == "fp32" else 6)
    p.set_option(npf.OPT_PROFILE, 1)


def ran(p):
    """Names of the kernels that the plan ran since the last look."""
    return {name for name, (count, _) in p.profile(reset=True).items() if count}


def assert_route(p, route, precision="split_bf16"):
    """On "tensor" the plan's terms ran on tensor cores, all of them."""
    names = ran(p)
    if route == "tensor" and precision != "fp64":
        assert {"split_mode_divide", "split_reduce"} <= names and "fp64_chain" not in names, names


def make_plan(npf, sysm, N_max, precision, **kw):
    p = npf.Plan(sysm.lam, sysm.U, sysm.V, N_max, precision=precision, **kw)
    for N, t in sysm.tensors.items():
        if N <= N_max:
            p.set_tensor(N, t)
    return p
