"""FP64 grade on the tensor cores at the edges of what it takes: waits that expire, rows and inverses
that are not finite, sums whose large terms cancel, no memory for its slices."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2304_13144_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api(native_lib):
    from paper_2304_13144_gb300 import api as A
    yield A
    for f in (A.MTP_FAULT_DEVICE_ALLOC, A.MTP_FAULT_ALLOC_SKIP, A.MTP_FAULT_GRADE_WAIT):
        A.mtp_debug_inject(f, 0)


def setup(api, types=2, lev=12, n=4, seed=5):
    """Model, batch and list of a perturbed crystal (m = 127 for two species at level 12)."""
    md = O.OracleModel(types, lev, 2.0, 5.0)
    nu_sum = [sum(nu for _, nu in labs) for labs, _ in md.basis]
    theta = synth.draw_theta(seed, types, md.n_rad, 8, nu_sum, [len(labs) for labs, _ in md.basis], 2.0, 5.0, 42.0)
    g = synth.rng(seed)
    pos, cell, _ = synth.cubic_supercell(synth._FCC, 3.6, n)
    b = api.Batch(synth.single(pos + g.normal(0, 0.1, pos.shape), g.integers(0, types, len(pos)), cell))
    model = api.mtp_load(api.make_desc(types, lev), theta)
    return model, b, api.mtp_build_neighbors(model, b)


def test_expired_waits_take_the_abort_path(api):
    """One try per wait: the kernel stops, drains its copies and products, frees tensor memory; the
    grades it did not finish are NaN, mtp_sync says so, and the next call is unaffected."""
    model, b, nb = setup(api)
    api.mtp_set_active_set(model, torch.tensor(synth.diag_dominant(6, model.n_params), device="cuda"))
    ref = api.mtp_grade(model, b, nb, "fp64")["gamma"].clone()
    api.mtp_sync(model)
    api.mtp_debug_inject(api.MTP_FAULT_GRADE_WAIT, 1)
    out = api.mtp_grade(model, b, nb, "fp64", threshold=2.0)
    with pytest.raises(api.MtpError) as e:
        api.mtp_sync(model)
    assert e.value.name == "MTP_ERR_TIMEOUT"
    g = out["gamma"]
    nan = torch.isnan(g)
    assert nan.any() and torch.equal(g[~nan], ref[~nan])
    assert int(out["n_flagged"].item()) == int((g[~nan] > 2.0).sum().item())
    again = api.mtp_grade(model, b, nb, "fp64")["gamma"]
    api.mtp_sync(model)
    assert torch.equal(again, ref)


def expected(rows, X):
    """gamma by the comparisons of the library: the largest |C|, a NaN column never the largest (-1 where
    every column is NaN)."""
    with np.errstate(all="ignore"):
        C = np.abs(rows @ X)
    return np.where(np.isnan(C), -1.0, C).max(1)


def check(gamma, ref, rel):
    plain = np.isfinite(ref) & (ref >= 0)
    np.testing.assert_array_equal(gamma[~plain], ref[~plain])
    np.testing.assert_allclose(gamma[plain], ref[plain], rtol=rel)


def test_overflowing_rows_leave_the_others_alone(api):
    """Radial coefficients of one species pair so large that the products of moments overflow: the rows
    of atoms with such a neighbor hold infinities, the others grade as if there were none."""
    types, lev, n = 2, 12, 5
    md = O.OracleModel(types, lev, 2.0, 5.0)
    nu_sum = [sum(nu for _, nu in labs) for labs, _ in md.basis]
    theta = synth.draw_theta(5, types, md.n_rad, 8, nu_sum, [len(labs) for labs, _ in md.basis], 2.0, 5.0, 42.0)
    big = theta.copy()
    n_c = types * types * md.n_rad * 8
    c = big[-n_c:].reshape(types, types, -1)
    c[0, 1] *= 1e200
    g = synth.rng(31)
    pos, cell, _ = synth.cubic_supercell(synth._FCC, 3.6, n)
    z = np.zeros(len(pos), int)
    z[[3, 250, 499]] = 1
    b = api.Batch(synth.single(pos + g.normal(0, 0.1, pos.shape), z, cell))
    A = torch.tensor(synth.diag_dominant(6, md.m), device="cuda")
    gam, rows = [], []
    for th in (theta, big):
        model = api.mtp_load(api.make_desc(types, lev), th)
        nb = api.mtp_build_neighbors(model, b)
        api.mtp_set_active_set(model, A)
        gam.append(api.mtp_grade(model, b, nb, "fp64")["gamma"].cpu().numpy())
        rows.append(api.mtp_param_rows(model, b, nb, "fp64").cpu().numpy())
        X = api.mtp_get_active_inverse(model).cpu().numpy()
    over = ~np.isfinite(rows[1]).all(1)
    same = (rows[0] == rows[1]).all(1)
    assert 50 < over.sum() < 300 and 200 < same.sum() < 450 and len(pos) % 64
    np.testing.assert_array_equal(gam[1][same], gam[0][same])
    check(gam[1][over], expected(rows[1][over], X), 1e-12)


def test_inverse_that_overflows(api):
    """A set whose every pivot is fine against max |A| and whose inverse has entries past 2^1024: the
    grades are those of plain sums over that inverse, infinities and NaN columns included."""
    model, b, nb = setup(api)
    m = model.n_params
    A = 2.0 ** -970 * (np.eye(m) - 2.0 ** 30 * np.eye(m, k=1))
    api.mtp_set_active_set(model, torch.tensor(A, device="cuda"))
    X = api.mtp_get_active_inverse(model).cpu().numpy()
    assert np.isfinite(X).any() and not np.isfinite(X).all()
    rows = api.mtp_param_rows(model, b, nb, "fp64").cpu().numpy()
    assert np.isfinite(rows).all()
    check(api.mtp_grade(model, b, nb, "fp64")["gamma"].cpu().numpy(), expected(rows, X), 1e-12)
    # and a set with a finite inverse again
    A = synth.diag_dominant(6, m)
    api.mtp_set_active_set(model, torch.tensor(A, device="cuda"))
    X = api.mtp_get_active_inverse(model).cpu().numpy()
    check(api.mtp_grade(model, b, nb, "fp64")["gamma"].cpu().numpy(), expected(rows, X), 1e-11)


@pytest.mark.parametrize("types,lev", [(2, 12), (3, 20)])
def test_winning_column_of_small_terms_beside_cancelling_large_ones(api, types, lev):
    """An inverse made for one atom's row b: its two largest terms, in two columns of their own, cancel
    to 2^-36, and every other column holds one product 2^-30 as large.  gamma is such a product, and must
    be as close to it as FP64 sums are bound to be: m 2^-53 sum_k |b_k X_kp| of its column."""
    model, b, nb = setup(api, types, lev)
    m = model.n_params
    rows = api.mtp_param_rows(model, b, nb, "fp64").cpu().numpy()
    atom = 17
    row = rows[atom]
    k1, k2 = np.argsort(-np.abs(row))[:2]
    g = synth.rng(9)
    top = abs(row[k1])
    X = np.diag(2.0 ** -30 * top * g.uniform(0.5, 1.0, m) / np.maximum(np.abs(row), 2.0 ** -6 * top))
    q, d = row[k1] / row[k2], 2.0 ** -36
    X[k1, k1] = X[k1, k2] = 1.0
    X[k2, k1], X[k2, k2] = -q * (1 + d), -q * (1 - d)
    A = np.diag(1.0 / np.diag(X))
    det = 2 * d * q
    A[np.ix_([k1, k2], [k1, k2])] = np.array([[X[k2, k2], -1.0], [-X[k2, k1], 1.0]]) / det
    api.mtp_set_active_set(model, torch.tensor(A, device="cuda"))
    X = api.mtp_get_active_inverse(model).cpu().numpy().astype(np.longdouble)
    out = api.mtp_grade(model, b, nb, "fp64")
    C = np.abs((row.astype(np.longdouble)[:, None] * X).sum(0))
    p = int(C.argmax())
    assert p not in (k1, k2)
    bound = m * 2.0 ** -53 * (np.abs(row) * np.abs(X[:, p])).sum()
    assert abs(out["gamma"][atom].item() - C[p]) <= bound
    # the other rows: within the bound of their largest products
    C = np.abs(np.stack([(r[:, None] * X).sum(0) for r in rows.astype(np.longdouble)])).max(1)
    tol = 2.0 ** -52 * C + m * 2.0 ** -53 * (np.abs(rows) * np.abs(X).max(1)).max(1)
    assert (np.abs(out["gamma"].cpu().numpy() - C) <= tol).all()


def regions(api, call):
    """The regions that a call runs."""
    torch.cuda.synchronize()
    api.mtp_profiler_enable(True)
    try:
        api.mtp_profiler_read()
        call()
        return set(api.mtp_profiler_read())
    finally:
        api.mtp_profiler_enable(False)


def fail_growth(api, after, call):
    """call() with the device allocation after `after` growths of its workspaces failing."""
    try:
        api.mtp_debug_inject(api.MTP_FAULT_ALLOC_SKIP, after)
        api.mtp_debug_inject(api.MTP_FAULT_DEVICE_ALLOC, 1)
        return call()
    finally:
        api.mtp_debug_inject(api.MTP_FAULT_DEVICE_ALLOC, 0)
        api.mtp_debug_inject(api.MTP_FAULT_ALLOC_SKIP, 0)


def test_without_memory_for_the_slices_of_rows(api):
    """The workspaces of the rows and of the flags exist, that of the slices cannot be had: the SIMT
    kernel answers."""
    model, b, nb = setup(api)
    api.mtp_set_active_set(model, torch.tensor(synth.diag_dominant(6, model.n_params), device="cuda"))
    api.mtp_config_rows(model, b, nb, "fp64")
    api.mtp_grade(model, b, nb, "mixed")
    out = []
    grade = lambda: out.append(api.mtp_grade(model, b, nb, "fp64")["gamma"].cpu().numpy())   # noqa: E731
    ran = regions(api, lambda: fail_growth(api, 0, grade))
    assert "grade_simt_fp64" in ran and "grade_fp64" not in ran
    ran = regions(api, grade)
    assert "grade_fp64" in ran and "grade_simt_fp64" not in ran
    np.testing.assert_allclose(out[0], out[1], rtol=1e-12)


def test_without_memory_for_the_slices_of_the_inverse(api):
    """Of the allocations of an active set only the first five have to succeed (A, the factors, a flag,
    the inverse, its mixed-precision copies); without the sixth FP64 grades take the SIMT kernel."""
    A = None
    out = []
    for after in range(7):
        model, b, nb = setup(api)
        A = torch.tensor(synth.diag_dominant(6, model.n_params), device="cuda") if A is None else A
        load = lambda: api.mtp_set_active_set(model, A)   # noqa: E731
        if after < 5:
            with pytest.raises(api.MtpError):
                fail_growth(api, after, load)
            load()
        else:
            fail_growth(api, after, load)
        ran = regions(api, lambda: out.append(api.mtp_grade(model, b, nb, "fp64")["gamma"].cpu().numpy()))
        assert ("grade_simt_fp64" if after == 5 else "grade_fp64") in ran, (after, ran)
        assert len({"grade_simt_fp64", "grade_fp64"} & ran) == 1
    for g in out:
        np.testing.assert_allclose(g, out[0], rtol=1e-12)
