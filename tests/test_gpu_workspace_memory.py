"""The Lanczos workspaces where device memory is short.

A context keeps a few GB of Lanczos vectors between calls.  They are what one can do without: a queue that
finds no room for them runs the COCG kernels, an allocation that fails takes back the ones that no queue
uses, and a batch divides the slots' 8 GB among its contexts.  Memory is made short by an allocation that
leaves the stated bytes free.  Systems: an empty box, whose orbitals are products of 1D eigenvectors.
Tolerance: two solves that meet tol differ by at most 2 tol cond(A), and cond(A) <= top / omega < 2e2 (top of the
stencil's symbol at h = 0.4: 60): 2e-8 at tol = 1e-10, 4e-6 (asserted: 1e-5) at 1e-8; 1e-6 leaves room for the
Coulomb operator's and the orthonormalisation's conditioning.
"""
import contextlib

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GB = 1 << 30


@pytest.fixture(scope="module")
def rpa():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2504_01816_gb300 as m
    return m


@contextlib.contextmanager
def only(free_bytes):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    if free < free_bytes + GB:
        pytest.skip("the device's memory is in use")
    hog = torch.empty(free - free_bytes, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hog
        torch.cuda.empty_cache()


def box(n, n_s, h=0.4):
    w = synth.fornberg_second_derivative(6)
    d = np.zeros((n, n))
    for i in range(n):
        for j in range(max(0, i - 6), min(n, i + 7)):
            d[i, j] = -0.5 * w[abs(i - j)] / h ** 2
    mu, q = np.linalg.eigh(d)
    modes = sorted((mu[a] + mu[b] + mu[c], a, b, c) for a in range(4) for b in range(4) for c in range(4))[:n_s]
    psi = np.stack([np.einsum("z,y,x->zyx", q[:, c], q[:, b], q[:, a]).reshape(-1) for _, a, b, c in modes])
    return h, torch.zeros(n ** 3, dtype=torch.float64, device="cuda"), torch.as_tensor(psi, device="cuda"), \
        [m[0] for m in modes]


def context(rpa, n, n_s, **options):
    h, v, psi, eps = box(n, n_s)
    o = rpa.default_options()
    o.prec, o.tol = rpa.RPA_MIXED, 1e-10
    for k, val in options.items():
        setattr(o, k, val)
    return rpa.Context(n, n, n, h, v, psi, eps, o)


def block(k, n, seed=3):
    return torch.randn(k, n ** 3, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))


def near(a, b):
    return float(torch.linalg.norm(a - b)) <= 1e-6 * float(torch.linalg.norm(b))


def test_queue_without_room_runs_the_cocg_kernels(rpa):
    """128 systems of 40^3: the slots take 0.6 GB, the Lanczos vectors more than 3 GB."""
    v = block(16, 40)
    opt = dict(profile=1, n_omega=1, fixed_subspace_iters=1, n_atoms=1)
    with context(rpa, 40, 8, **opt) as ctx:
        full = ctx.ec(v)
    with context(rpa, 40, 8, **opt) as ctx, only(2 * GB):
        short = ctx.ec(v)
    assert any(k["name"].startswith("k_lanczos") for k in full.stats["kernels"]), full.stats["kernels"]
    assert not any(k["name"].startswith("k_lanczos") for k in short.stats["kernels"]), short.stats["kernels"]
    assert full.status == short.status == rpa.RPA_OK
    assert np.allclose(full.lambdas, short.lambdas, rtol=1e-6, atol=0)


def test_idle_workspaces_are_given_back(rpa):
    """A second context's call needs 0.6 GB where 0.4 are left; the first holds more than 3 GB that it does not use."""
    v = block(16, 40)
    with context(rpa, 40, 8) as first, context(rpa, 40, 8) as second:
        a, code = first.apply_nuchi0(0.5, v)
        assert code == rpa.RPA_OK
        with only(int(0.4 * GB)):
            b, code = second.apply_nuchi0(0.5, v)
            assert code == rpa.RPA_OK
            again, code2 = first.apply_nuchi0(0.5, v)
        assert code2 == rpa.RPA_OK
        assert near(b, a) and near(again, a)


def test_setup_takes_idle_workspaces_back(rpa):
    v = block(16, 40)
    with context(rpa, 40, 8) as first:
        a, _ = first.apply_nuchi0(0.5, v)
        args = box(100, 48)
        o = rpa.default_options()
        o.prec = rpa.RPA_MIXED
        with only(int(0.3 * GB)):                # psi in FP64 and FP32: 0.6 GB
            rpa.Context(100, 100, 100, args[0], args[1], args[2], args[3], o).close()
        again, code = first.apply_nuchi0(0.5, v)
        assert code == rpa.RPA_OK and near(again, a)


def test_batch_shares_the_slot_storage(rpa):
    """Four contexts of 512 systems of 64^3: 9.7 GB of slots each if each took what it takes alone."""
    n, n_s, k = 64, 8, 64
    vs = [block(k, n, seed) for seed in range(4)]
    with contextlib.ExitStack() as stack:
        ctxs = [stack.enter_context(context(rpa, n, n_s, tol=1e-8)) for _ in vs]
        with only(14 * GB):
            rs, code = rpa.rpa.apply_nuchi0_batch(ctxs, 0.8, vs)
        assert code == rpa.RPA_OK
    with context(rpa, n, n_s, tol=1e-8) as ctx:
        alone, code = ctx.apply_nuchi0(0.8, vs[2])
    assert code == rpa.RPA_OK
    assert float(torch.linalg.norm(rs[2] - alone)) <= 1e-5 * float(torch.linalg.norm(alone))
