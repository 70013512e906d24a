"""The staged patch kernels (shared-memory neighbourhoods; integer limbs for FP64) against the
row-by-row colour kernels, at the sizes where their index rules change: meshes so small that
every patch touches a wall or two, the first mesh with interior patches, ragged counts of
patches per warp; every operator form; value ranges near the ends of FP64.

Tolerances: a sweep is a few dozen sums of products per unknown and colour; both sides round
each at 2^-53 or better of its largest term, and a colour's correction passes through at most
(p+1)^2 later colours: 1e-12 (FP64) and 5e-5 (FP32, the same with 2^-24) of the largest unknown.
"""
import numpy as np
import pytest

from paper_1705_09282_gb300 import inputs

pytestmark = pytest.mark.gpu


def _torch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


def _pair(monkeypatch, *args, **kw):
    from paper_1705_09282_gb300.solver import Solver
    S1 = Solver(*args, **kw)
    monkeypatch.setenv("IGAMG_SWEEP_FORM", "lanes1")
    monkeypatch.setenv("IGAMG_FUSED_LEVELS", "-1")
    S0 = Solver(*args, **kw)
    monkeypatch.delenv("IGAMG_SWEEP_FORM")
    monkeypatch.delenv("IGAMG_FUSED_LEVELS")
    return S0, S1


@pytest.mark.parametrize("p", [2, 3])
@pytest.mark.parametrize("n", [4, 6, 8, 10, 14, 22, 46])
@pytest.mark.parametrize("kind", ["stokes", "oseen", "annulus", "fp32"])
def test_staged_sweeps_equal_row_kernels(p, n, kind, monkeypatch):
    torch = _torch()
    from paper_1705_09282_gb300 import _lib
    kw = {}
    if kind == "oseen":
        kw["beta"] = inputs.oseen_advection(p, n, 0.5)
    elif kind == "annulus":
        kw["geometry"] = _lib.IGAMG_GEOM_QUARTER_ANNULUS
    elif kind == "fp32":
        kw["precision"] = _lib.IGAMG_FP32_IR
    S0, S1 = _pair(monkeypatch, p, n, 2, 10.0, 0.5, **kw)
    nd = S0.ndof()
    dt = torch.float32 if kind == "fp32" else torch.float64
    U = torch.tensor(inputs.random_vector(nd, seed=n), device="cuda").to(dt)
    F = torch.tensor(inputs.random_vector(nd, seed=n + 1), device="cuda").to(dt)
    U0, U1 = U.clone(), U.clone()
    for S, V in ((S0, U0), (S1, U1)):
        (S.smooth32 if kind == "fp32" else S.smooth)(V, F, sweeps=1)
    tol = 5e-5 if kind == "fp32" else 1e-12
    assert float((U0 - U1).abs().max()) <= tol * float(U0.abs().max())
    S0.close()
    S1.close()


@pytest.mark.parametrize("scale", [2.0 ** -600, 2.0 ** 600, 0.0])
def test_staged_sweep_at_extreme_scales(scale, monkeypatch):
    # the sweep is linear in (U, F): a power of two changes exponents only
    torch = _torch()
    from paper_1705_09282_gb300.solver import Solver
    S = Solver(2, 16, 2, 1.0, 1.0)
    nd = S.ndof()
    U = torch.tensor(inputs.random_vector(nd, seed=3), device="cuda")
    F = torch.tensor(inputs.random_vector(nd, seed=4), device="cuda")
    V, W = U.clone(), U * scale
    S.smooth(V, F, sweeps=2)
    S.smooth(W, F * scale, sweeps=2)
    assert torch.equal(W, V * scale)
    S.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("where", ["U", "F"])
def test_staged_sweep_spreads_nonfinite_values_as_the_row_kernel_does(bad, where, monkeypatch):
    torch = _torch()
    S0, S1 = _pair(monkeypatch, 2, 32, 2, 1.0, 1.0)
    nd = S0.ndof()
    g = nd // 3
    out = []
    for S in (S0, S1):
        U = torch.tensor(inputs.random_vector(nd, seed=5), device="cuda")
        F = torch.tensor(inputs.random_vector(nd, seed=6), device="cuda")
        (U if where == "U" else F)[g] = bad
        S.smooth(U, F, sweeps=1)
        out.append(torch.isfinite(U))
        S.close()
    assert not out[1][g] if where == "F" else True
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("p,n", [(2, 4), (2, 6), (2, 8), (2, 10), (2, 12), (3, 4), (3, 6), (3, 8), (3, 10)])
@pytest.mark.parametrize("kind", ["stokes", "oseen", "cylinder", "fp32", "cylinder-fp32"])
def test_staged_sweeps_3d_equal_row_kernels(p, n, kind, monkeypatch):
    torch = _torch()
    from paper_1705_09282_gb300 import _lib
    from paper_1705_09282_gb300.solver import Solver
    if n > 8 and kind != "stokes" and (p == 3 or "cylinder" in kind):
        pytest.skip("set-up of this form takes long; the index rules are those of the Stokes case")
    kw = {"dim": 3}
    if kind == "oseen":
        kw["beta"] = inputs.oseen_advection_3d(p, n, 0.5)
    if kind.startswith("cylinder"):
        kw["geometry"] = _lib.IGAMG_GEOM_HOLLOW_CYLINDER
    if kind.endswith("fp32"):
        kw["precision"] = _lib.IGAMG_FP32_IR
    monkeypatch.setenv("IGAMG_FUSED_LEVELS", "-1")
    S1 = Solver(p, n, 2, 10.0, 0.5, **kw)
    monkeypatch.setenv("IGAMG_SWEEP_FORM", "rows")
    S0 = Solver(p, n, 2, 10.0, 0.5, **kw)
    nd = S0.ndof()
    F = torch.tensor(inputs.random_vector(nd, seed=n + 1), device="cuda")
    if kind.endswith("fp32"):
        # one refinement step from zero: an FP32 V-cycle, its velocity lifted in FP64
        V0, V1 = S0.empty(), S1.empty()
        for S, V in ((S0, V0), (S1, V1)):
            S.vcycle(V, F)
        tol = 5e-5
    else:
        V0 = torch.tensor(inputs.random_vector(nd, seed=n), device="cuda")
        V1 = V0.clone()
        S0.smooth(V0, F, sweeps=1)
        S1.smooth(V1, F, sweeps=1)
        tol = 1e-12
    assert float((V0 - V1).abs().max()) <= tol * float(V0.abs().max())
    S0.close()
    S1.close()


@pytest.mark.parametrize("p,n,dim,kind", [(2, 16, 2, "stokes"), (3, 14, 2, "stokes"), (2, 12, 2, "oseen"), (2, 12, 2, "annulus"),
                                          (3, 12, 2, "annulus"), (2, 6, 3, "stokes"), (2, 6, 3, "oseen"), (2, 6, 3, "cylinder"),
                                          (3, 6, 3, "stokes"), (3, 6, 3, "cylinder")])
@pytest.mark.parametrize("small", ["none", "ux", "uy", "p", "uxp"])
def test_rows_keep_their_precision_when_components_differ(p, n, dim, kind, small, monkeypatch):
    # every patch row's local residual against the same sum in extended precision, component by component,
    # one or two of which are 1e-4 and 1e-8 of the others: no row may lose to values it does not read.
    # Bound, relative to D = |F| + sum over components of (sum |K_ij|) max |U_j|, with N terms in the
    # largest box: values cut at 2^-56, coefficients rounded at 2^-58 each, lo x lo products left out
    # at 2^-58 each, two shifts of 2^-57 per box and lane of the row, the result rounded at 2^-54.
    # And the root mean square must not exceed that of FP64 multiply-adds (k_residual on the records).
    torch = _torch()
    import ctypes

    from paper_1705_09282_gb300 import _lib
    from paper_1705_09282_gb300.solver import Solver, host_operator_rows
    monkeypatch.setenv("IGAMG_ADV_FORM", "records")
    kw = {"dim": 3} if dim == 3 else {}
    if kind == "oseen":
        kw["beta"] = inputs.oseen_advection_3d(p, n, 0.5) if dim == 3 else inputs.oseen_advection(p, n, 0.5)
    elif kind != "stokes":
        kw["geometry"] = _lib.IGAMG_GEOM_QUARTER_ANNULUS if dim == 2 else _lib.IGAMG_GEOM_HOLLOW_CYLINDER
    S = Solver(p, n, 2, 10.0, 0.5, **kw)
    nd = S.ndof()
    K = host_operator_rows(p, n, 2, 10.0, 0.5, 1, **kw)[: nd - 1]
    q = p - 1
    if dim == 2:
        nc = (n + p - 2) * (n + q)
        cuts = [0, nc, 2 * nc, nd - 1, nd]
        terms, lanes = max((2 * p + 1) * (2 * q + 1), 4 * p * p), 1
    else:
        nc = (n + p - 2) * (n + q) ** 2
        cuts = [0, nc, 2 * nc, 3 * nc, nd - 1, nd]
        terms, lanes = max((2 * p + 1) * (2 * q + 1) ** 2, 4 * p * p * (2 * q + 1)), 4 if p == 2 else 8
    comp = [slice(a, b) for a, b in zip(cuts, cuts[1:])]
    U = inputs.random_vector(nd, seed=n)
    scale = {"none": (), "ux": ((0, 1e-8),), "uy": ((1, 1e-4),), "p": ((dim, 1e-8),), "uxp": ((0, 1e-4), (dim, 1e-8))}[small]
    for c, x in scale:
        U[comp[c]] *= x
    F = np.zeros(nd)
    F[: nd - 1] = (K @ U) * (1.0 + 0.5 * inputs.random_vector(nd - 1, seed=n + 1))
    exact = F[: nd - 1].astype(np.longdouble) - np.array([(k.astype(np.longdouble) * U.astype(np.longdouble)).sum() for k in K])
    D = np.abs(F[: nd - 1])
    for c in comp:
        D = D + np.abs(K[:, c]).sum(axis=1) * np.abs(U[c]).max()
    Ud, Fd = torch.tensor(U, device="cuda"), torch.tensor(F, device="cuda")
    R = torch.full((nd,), float("nan"), dtype=torch.float64, device="cuda")
    _lib.check(_lib.lib().igamg_probe_patch_rows(S._h, 1, ctypes.c_void_p(Ud.data_ptr()), ctypes.c_void_p(Fd.data_ptr()),
                                                 ctypes.c_void_p(R.data_ptr())), "igamg_probe_patch_rows")
    got = R.cpu().numpy()[: nd - 1]
    fp64 = S.residual(Ud, Fd).cpu().numpy()[: nd - 1]
    assert torch.equal(Ud, torch.tensor(U, device="cuda"))
    rel = (np.abs(got - exact) / D).astype(float)
    ref = (np.abs(fp64 - exact) / D).astype(float)
    for k, c in enumerate(comp[:-1]):
        assert rel[c].max() <= (2 * terms + 4 + 16 * lanes) * 2.0 ** -58 + 2.0 ** -54, k
        assert np.sqrt((rel[c] ** 2).mean()) <= np.sqrt((ref[c] ** 2).mean()), k
    S.close()


@pytest.mark.parametrize("dim,p,n", [(2, 2, 16), (2, 3, 16), (3, 2, 8)])
@pytest.mark.parametrize("scale", [2.0 ** -920, 2.0 ** 940])
def test_staged_sweep_near_the_ends_of_the_exponent_range(dim, p, n, scale):
    # as test_staged_sweep_at_extreme_scales; the largest value of every component of a neighbourhood stays
    # above 2^-959 here, below which the staged rows give up low bits
    torch = _torch()
    from paper_1705_09282_gb300.solver import Solver
    S = Solver(p, n, 2, 1.0, 1.0, **({"dim": 3} if dim == 3 else {}))
    nd = S.ndof()
    U = torch.tensor(inputs.random_vector(nd, seed=3), device="cuda")
    F = torch.tensor(inputs.random_vector(nd, seed=4), device="cuda")
    V, W = U.clone(), U * scale
    S.smooth(V, F)
    S.smooth(W, F * scale)
    assert torch.equal(W, V * scale)
    S.close()


@pytest.mark.parametrize("p,n", [(2, 6), (2, 10), (3, 6)])
@pytest.mark.parametrize("kind", ["stokes", "oseen", "cylinder", "fp32", "cylinder-fp32"])
def test_3d_records_read_in_place_equal_records_fetched_ahead(p, n, kind, monkeypatch):
    # the variant for colours of many blocks, on meshes small enough to run every form: the FP64 rows are
    # integers, so both variants agree bit for bit (FP32: the tolerance of the sweep against the row kernels)
    torch = _torch()
    from paper_1705_09282_gb300 import _lib
    from paper_1705_09282_gb300.solver import Solver
    kw = {"dim": 3}
    if kind == "oseen":
        kw["beta"] = inputs.oseen_advection_3d(p, n, 0.5)
    if kind.startswith("cylinder"):
        kw["geometry"] = _lib.IGAMG_GEOM_HOLLOW_CYLINDER
    if kind.endswith("fp32"):
        kw["precision"] = _lib.IGAMG_FP32_IR
    monkeypatch.setenv("IGAMG_FUSED_LEVELS", "-1")
    out = []
    for blocks in ("0", str(1 << 30)):
        monkeypatch.setenv("IGAMG_PRE_BLOCKS", blocks)
        S = Solver(p, n, 2, 10.0, 0.5, **kw)
        F = torch.tensor(inputs.random_vector(S.ndof(), seed=n + 1), device="cuda")
        if kind.endswith("fp32"):
            V = S.empty()
            S.vcycle(V, F)
        else:
            V = torch.tensor(inputs.random_vector(S.ndof(), seed=n), device="cuda")
            S.smooth(V, F, sweeps=2)
        out.append(V.clone())
        S.close()
    if kind.endswith("fp32"):
        assert float((out[0] - out[1]).abs().max()) <= 5e-5 * float(out[1].abs().max())
    else:
        assert torch.equal(out[0], out[1])


def _staged(S):
    import ctypes

    from paper_1705_09282_gb300 import _lib
    U, R = S.empty(), S.empty()
    rc = _lib.lib().igamg_probe_patch_rows(S._h, 1, ctypes.c_void_p(U.data_ptr()), ctypes.c_void_p(U.data_ptr()),
                                           ctypes.c_void_p(R.data_ptr()))
    return rc == 0


@pytest.mark.parametrize("kind,p,n,dim", [("oseen", 2, 16, 2), ("annulus", 3, 16, 2), ("oseen", 2, 8, 3), ("cylinder-fp32", 2, 6, 3)])
def test_levels_without_memory_for_staged_tables_run_the_row_kernels(kind, p, n, dim, monkeypatch):
    torch = _torch()
    from paper_1705_09282_gb300 import _lib
    from paper_1705_09282_gb300.solver import Solver
    kw = {"dim": 3} if dim == 3 else {}
    if kind == "oseen":
        kw["beta"] = inputs.oseen_advection_3d(p, n, 0.5) if dim == 3 else inputs.oseen_advection(p, n, 0.5)
    else:
        kw["geometry"] = _lib.IGAMG_GEOM_QUARTER_ANNULUS if dim == 2 else _lib.IGAMG_GEOM_HOLLOW_CYLINDER
    if kind.endswith("fp32"):
        kw["precision"] = _lib.IGAMG_FP32_IR
    monkeypatch.setenv("IGAMG_FUSED_LEVELS", "-1")
    out = []
    for free in (None, "0"):
        if free is not None:
            monkeypatch.setenv("IGAMG_STAGED_FREE", free)
        S = Solver(p, n, 2, 10.0, 0.5, **kw)
        assert _staged(S) == (free is None)
        F = torch.tensor(inputs.random_vector(S.ndof(), seed=n + 1), device="cuda")
        V = S.empty()
        S.vcycle(V, F)
        out.append(V.clone())
        S.close()
    tol = 5e-5 if kind.endswith("fp32") else 1e-11            # four sweeps and a coarse solve of the sweeps' 1e-12
    assert float((out[0] - out[1]).abs().max()) <= tol * float(out[0].abs().max())


def test_staged_levels_hold_their_local_inverses_once(monkeypatch):
    # an operator with records and inverses per row and patch: the staged handle holds more than the row
    # kernels' one by its records (976 bytes a row), the wall patches' rows (64 entries of 16 bytes each) and
    # the padding of its inverses (8 to 10 entries a row of the 8 x 8 ones, under 12 % on the others), not by a
    # second copy of the inverses
    torch = _torch()
    from paper_1705_09282_gb300.solver import Solver
    n, L = 24, 3
    beta = inputs.oseen_advection_3d(2, n, 0.5)
    monkeypatch.setenv("IGAMG_FUSED_LEVELS", "-1")

    def held(form):
        if form:
            monkeypatch.setenv("IGAMG_SWEEP_FORM", form)
        else:
            monkeypatch.delenv("IGAMG_SWEEP_FORM", raising=False)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        S = Solver(2, n, L, 10.0, 0.5, dim=3, beta=beta)
        used = before - torch.cuda.mem_get_info()[0]
        rows = sum(S.ndof(l) for l in range(L))
        staged = _staged(S)
        S.close()
        return used, rows, staged

    held(None)                                                # loads the kernels
    used, rows, staged = held(None)
    base, _, rowform = held("rows")
    assert staged and not rowform
    inverses = base - 944 * rows
    walls = sum(3 * (m + 1) * m ** 2 - 3 * (m - 3) * (m - 4) ** 2 for m in (n, n // 2))
    assert used <= base + 976 * rows + 1024 * walls + 0.25 * inverses + (8 << 20)
