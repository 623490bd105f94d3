"""What a context keeps between calls (the factor, the quantized coordinates,
side buffers, the report of a batch) must not reach a later call with other
points: each test mixes entry points on one context and checks the results
against plain FP64 arithmetic."""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

M = pytest.importorskip("paper_2607_23354_gb300")


def _dev(X):
    return torch.from_numpy(np.ascontiguousarray(X)).cuda()


def _rel(X, t, x, b):
    """||b - Z x|| / (||Z|| ||x||) in FP64, Z from the points."""
    d = torch.cdist(X, X, compute_mode="donot_use_mm_for_euclid_dist")
    Z = torch.exp(-t * d)
    return float((b - Z @ x).abs().max() / (Z.sum(1).max() * x.abs().max()))


# A solve with a kept factor refines with the points it was given: in between,
# another entry point quantizes other points at the same address (changed in
# place and restored, or the temporary FP64 copies of FP32 points).  The other
# points are 1e-6 away, so a refinement with them converges, to a residual of
# about 1e-7 here; 1e-14 is the library's tolerance, doubled for the check's own
# FP64 rounding.
@pytest.mark.parametrize("options", [dict(precision="fp64"), dict(residual_mode="matrix_free")])
@pytest.mark.parametrize("between", ["residual", "grad"])
@pytest.mark.parametrize("fp32", [False, True])
def test_kept_factor_refines_with_its_own_points(options, between, fp32):
    rng = np.random.default_rng(4)
    n, t = 700, 2.0
    A = _dev(rng.random((n, 6)))
    B = A + 1e-6 * _dev(rng.standard_normal((n, 6)))
    if fp32:
        A, B = A.float(), B.float()
    b = _dev(rng.standard_normal(n))
    c = M.Context(M.Options(**options))

    def other(P):
        if between == "residual":
            c.residual(P, t, b)
        else:
            c.grad(P, t, w=b)

    c.solve(A, t)
    if fp32:
        other(B)
    else:
        keep = A.clone()
        A.copy_(B)
        other(A)
        A.copy_(keep)
    x, info = c.solve_rhs(A, t, b)
    c.close()
    assert info["factor_reused"] == 1 or fp32  # the copies' address is the allocator's choice
    assert _rel(A.double(), t, x, b) <= 2e-14


# A kept factor is given up when an entry point lays the workspace out for more
# points (its tiles would be looked for at the other layout's offsets).
@pytest.mark.parametrize("between", ["min_distance", "residual", "similarity_matrix"])
def test_kept_factor_and_a_larger_layout(between):
    rng = np.random.default_rng(9)
    X, Y = _dev(rng.random((300, 4))), _dev(rng.random((2000, 4)))
    b = _dev(rng.standard_normal(300))
    c = M.Context()
    c.solve(X, 3.0)
    if between == "min_distance":
        c.min_distance(Y)
    elif between == "residual":
        c.residual(Y, 3.0, Y[:, 0])
    else:
        c.similarity_matrix(Y, 3.0)
    x, info = c.solve_rhs(X, 3.0, b)
    assert info["factor_reused"] == 0
    assert _rel(X, 3.0, x, b) <= 2e-14
    # and is used again without such a call
    c.solve(X, 3.0)
    x, info = c.solve_rhs(X, 3.0, b)
    c.close()
    assert info["factor_reused"] == 1
    assert _rel(X, 3.0, x, b) <= 2e-14


# A batch leaves its workspace (1.8 GB) in the context: a solve for which the free
# memory alone is too little takes it back and stays in core.
def test_side_buffers_are_given_back_to_a_solve():
    rng = np.random.default_rng(3)
    c = M.Context()
    clouds = [_dev(rng.standard_normal((2048, 8))) for _ in range(48)]
    c.solve_batch(clouds, [1.0])
    X = _dev(rng.random((8192, 8)))
    need = c.workspace_bytes(8192, 8)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    assert need > 0.9e9
    hog = torch.empty(int(torch.cuda.mem_get_info()[0] - 0.5e9), dtype=torch.uint8, device="cuda")
    try:
        w, mag, info = c.solve(X, 5.0)
        _, dx = c.grad(X, 5.0, w=w)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert info["slabs"] == 0 and bool(torch.isfinite(dx).all())
    assert _rel(X, 5.0, w, torch.ones_like(w)) <= 2e-14
    _, mags, sts = c.solve_batch(clouds[:2], [1.0])  # and the batch takes its own again
    c.close()
    assert int(sts.abs().sum()) == 0


# Partial sums and digits keep to the workspace limit together with the workspace,
# with the same results as without one.
def test_side_buffers_under_a_workspace_limit():
    rng = np.random.default_rng(5)
    X, w = _dev(rng.random((3000, 6))), _dev(rng.standard_normal(3000))
    g = torch.full((3000,), 0.7, dtype=torch.float64, device="cuda")  # constant: no solve
    clouds = [_dev(rng.standard_normal((n, 6))) for n in (1500, 700, 300, 1500)]
    out = []
    for limit in (0.0, 4e7):
        c = M.Context(M.Options(workspace_limit_bytes=limit))
        r, norms = c.residual(X, 2.0, w)
        dt, dx = c.grad(X, 2.0, w=w, dL_dw=g)
        ws, mags, sts = c.solve_batch(clouds, [0.5, 2.0])
        assert int(sts.abs().sum()) == 0
        out.append((r, dx, torch.tensor([dt, norms["r_norm_inf"], norms["z_norm_inf"]]), torch.cat(ws), mags))
        c.close()
    for a, b in zip(*out):
        assert float((a - b).abs().max()) <= 1e-11 * float(a.abs().max())


# A batch reports the launch shape of its own one-CTA launch, or none.
def test_batch_reports_its_own_launch():
    rng = np.random.default_rng(8)
    small, large = [_dev(rng.standard_normal((n, 5))) for n in (40, 300)]
    keys = ("batch_threads", "batch_ctas_per_sm", "batch_tensor_cores", "batch_left_looking")
    c = M.Context()
    seen = []
    for clouds in ([large], [small, large], [large]):
        c.solve_batch(clouds, [1.0])
        seen.append([c.last_batch_info[k] for k in keys])
    c.close()
    assert seen[0] == seen[2] == [0, 0, 0, 0]
    assert seen[1][0] in (256, 512) and seen[1][1] >= 1


# FP32 w and dL/dw are converted for the call: the copy of the one must not take the
# memory of the other's.
def test_gradient_of_converted_vectors():
    rng = np.random.default_rng(2)
    X = _dev(rng.random((400, 5)))
    w, g = _dev(rng.standard_normal(400)).float(), _dev(rng.standard_normal(400)).float()
    c = M.Context()
    dt, dx = c.grad(X, 1.5, w=w, dL_dw=g)
    dt64, dx64 = c.grad(X, 1.5, w=w.double(), dL_dw=g.double())
    c.close()
    assert dt == dt64 and torch.equal(dx, dx64)


# Contexts of two threads, each on its own stream, with points of different
# dimension: the kernels' shared memory depends on it, and their limit on it is one
# for the process.  Errors of a launch come back as MagnitudeError.
@pytest.mark.parametrize("call", ["similarity_matrix", "residual", "solve_batch", "residual_many_dimensions"])
def test_threads_with_different_dimensions(call):
    errors = []

    def work(m, seed):
        try:
            rng = np.random.default_rng(seed)
            n = 130 if call == "solve_batch" else 60
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                X, w = _dev(rng.standard_normal((n, m))), _dev(rng.standard_normal(n))
                c = M.Context(stream=stream)
                for _ in range(400):
                    if call == "similarity_matrix":
                        c.similarity_matrix(X, 0.2)
                    elif call == "solve_batch":
                        c.solve_batch([X], [0.5])
                    else:
                        c.residual(X, 0.2, w)
                c.close()
        except Exception as e:  # noqa: BLE001 (reported by the test's own thread)
            errors.append(e)

    dims = (1000, 1900) if call == "residual_many_dimensions" else (17, 32)
    threads = [threading.Thread(target=work, args=(m, i)) for i, m in enumerate(dims)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
