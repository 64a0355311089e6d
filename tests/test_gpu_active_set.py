"""MaxVol active-set update (Section II.D) on the GPU through the C ABI vs the oracle."""
import numpy as np
import pytest
import torch

from oracle import active_set as AS
from oracle import oracle as O
from paper_2304_13144_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api(native_lib):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2304_13144_gb300 import api as A
    return A


def theta_for(md, seed, nbar=40.0):
    nu_sum = [sum(nu for _, nu in labs) for labs, _ in md.basis]
    nf = [len(labs) for labs, _ in md.basis]
    return synth.draw_theta(seed, md.n_types, md.n_rad, md.n_q, nu_sum, nf, md.r_min, md.r_cut, nbar)


def test_maxvol_random_rows_match_oracle(api):
    """A level-8 unary model only supplies m = 26; the active set and candidates are random."""
    md = O.OracleModel(1, 8, 2.0, 5.0)
    m = md.m
    model = api.mtp_load(api.make_desc(1, 8), theta_for(md, 3))
    g = synth.rng(21)
    A0 = synth.diag_dominant(22, m)
    B = g.normal(size=(300, m)) * np.abs(A0).max() * 0.5
    api.mtp_set_active_set(model, torch.tensor(A0, device="cuda"))
    src, ns = api.mtp_maxvol(model, torch.tensor(B), eps=1e-3)
    A_ref, src_ref, ns_ref = AS.maxvol(A0, B, 1e-3)
    assert ns == ns_ref and ns > 0
    np.testing.assert_array_equal(src.cpu().numpy(), src_ref)
    np.testing.assert_array_equal(api.mtp_get_active_set(model).cpu().numpy(), A_ref)
    Ainv = api.mtp_get_active_inverse(model).cpu().numpy()
    ref_inv = np.linalg.inv(A_ref)
    assert np.abs(Ainv - ref_inv).max() <= 1e-10 * np.abs(ref_inv).max()
    # every candidate now has grade <= 1 + eps against the updated set
    C = B @ ref_inv
    assert np.abs(C).max() <= 1 + 1e-3 + 1e-9


def test_maxvol_on_mtp_rows_then_grade(api):
    """Active set from one snapshot (gauge-completed), candidates = FP64 rows of a hotter
    snapshot; after the update every candidate neighborhood grades <= 1 + eps on the GPU."""
    md = O.OracleModel(2, 10, 2.0, 5.0)
    theta = theta_for(md, 31)
    desc = api.make_desc(2, 10)
    model = api.mtp_load(desc, theta)
    cold = synth.b2_binary(seed=31, n=4, sigma=0.05)
    hot = synth.b2_binary(seed=32, n=4, sigma=0.25)
    bc, bh = api.Batch(cold), api.Batch(hot)
    nc, nh = api.mtp_build_neighbors(model, bc), api.mtp_build_neighbors(model, bh)
    sz = model.model_sizes()
    m, ng = sz["n_params"], sz["n_gauge"]
    pick = torch.tensor(synth.sample_atoms(5, len(cold["type"]), m - ng))
    rows = api.mtp_param_rows(model, bc, nc, "fp64", pick).cpu().numpy()
    D = api.mtp_gauge_directions(desc, theta)
    A0 = np.vstack([rows, D / np.linalg.norm(D, axis=1, keepdims=True) * np.abs(rows).max()])
    api.mtp_set_active_set(model, torch.tensor(A0, device="cuda"))
    Bh = api.mtp_param_rows(model, bh, nh, "fp64")
    src, ns = api.mtp_maxvol(model, Bh, eps=1e-2)
    src = src.cpu().numpy()
    assert ns > 0
    assert (src[m - ng:] < 0).all()        # the gauge rows stay (candidates have no component there)
    # the rows of the new A are the recorded ones, and (oracle arithmetic on the GPU's result)
    # no candidate can raise |det A| by more than 1 + eps
    A = api.mtp_get_active_set(model).cpu().numpy()
    Bn = Bh.cpu().numpy()
    for j in range(m):
        np.testing.assert_array_equal(A[j], A0[j] if src[j] < 0 else Bn[src[j]])
    C = np.linalg.solve(A.T, Bn.T).T
    assert np.abs(C).max() <= 1 + 1e-2 + 1e-4   # slack: cond(A) ~ 1e10 for lattice snapshots
    assert abs(np.linalg.slogdet(A)[1]) >= 0 and np.linalg.slogdet(A)[1] > np.linalg.slogdet(A0)[1]
    # the same greedy sequence as the oracle's (well separated maxima at this size)
    A_ref, src_ref, ns_ref = AS.maxvol(A0, Bn, 1e-2)
    assert ns == ns_ref
    np.testing.assert_array_equal(src, src_ref)
    gam = api.mtp_grade(model, bh, nh, "fp64", threshold=2.0)["gamma"].cpu().numpy()
    assert gam.max() <= 1 + 1e-2 + 1e-4


def test_maxvol_edge_cases(api):
    md = O.OracleModel(1, 8, 2.0, 5.0)
    model = api.mtp_load(api.make_desc(1, 8), theta_for(md, 3))
    m = md.m
    with pytest.raises(api.MtpError):
        api.mtp_maxvol(model, torch.zeros((4, m)))          # no active set yet
    A0 = synth.diag_dominant(23, m)
    api.mtp_set_active_set(model, torch.tensor(A0, device="cuda"))
    src, ns = api.mtp_maxvol(model, torch.zeros((0, m)))
    assert ns == 0 and (src.cpu().numpy() < 0).all()
    src, ns = api.mtp_maxvol(model, torch.tensor(A0[:5] * 0.5))   # dominated candidates
    assert ns == 0
    with pytest.raises(api.MtpError):
        api.mtp_maxvol(model, torch.zeros((4, m)), eps=-1.0)
    src, ns = api.mtp_maxvol(model, torch.tensor(A0 * 3.0), max_swaps=2)
    assert ns == 2


@pytest.mark.parametrize("types,n_q", [(1, 1), (1, 13), (1, 14), (1, 15), (2, 32), (4, 32), (8, 16), (8, 31), (8, 32)])
def test_active_inverse_at_panel_edges(api, types, n_q):
    """A^-1 around the edges of the panels and of the rows a thread holds (m = 3, 15, 16, 17, 131, 517,
    1033, 1993 and, column by column, 2057): random matrices whose every pivot is off the diagonal."""
    desc = api.make_desc(types, 2, n_q)
    m = api.mtp_describe(desc)["n_params"]
    model = api.mtp_load(desc, np.zeros(m))
    g = synth.rng(m)
    A = g.normal(size=(m, m)) + np.roll(np.diag(g.uniform(2.0, 3.0, m) * np.sqrt(m)), 1 + m // 3, axis=1)
    api.mtp_set_active_set(model, torch.tensor(A, device="cuda"))
    ref = np.linalg.inv(A)
    err = np.abs(api.mtp_get_active_inverse(model).cpu().numpy() - ref).max() / np.abs(ref).max()
    # both inverses: a few m eps cond(A); the condition number of these is a few tens at most
    assert err <= 4 * m * np.finfo(float).eps * np.linalg.cond(A, 1)


@pytest.mark.parametrize("n,max_swaps", [(5, 100), (40, 3), (700, 1_000_000)])
def test_maxvol_fewer_and_more_candidates_than_parameters(api, n, max_swaps):
    """Candidates fewer than parameters, a limit on the swaps, several blocks' worth of entries."""
    desc = api.make_desc(2, 2, 24)
    m = api.mtp_describe(desc)["n_params"]
    model = api.mtp_load(desc, np.zeros(m))
    g = synth.rng(23)
    A0 = synth.diag_dominant(24, m)
    B = g.normal(size=(n, m)) * np.abs(A0).max()
    api.mtp_set_active_set(model, torch.tensor(A0, device="cuda"))
    src, ns = api.mtp_maxvol(model, torch.tensor(B), eps=1e-3, max_swaps=max_swaps)
    A_ref, src_ref, ns_ref = AS.maxvol(A0, B, 1e-3, max_swaps)
    assert ns == ns_ref and 0 < ns <= max_swaps
    np.testing.assert_array_equal(src.cpu().numpy(), src_ref)
    np.testing.assert_array_equal(api.mtp_get_active_set(model).cpu().numpy(), A_ref)


@pytest.mark.parametrize("n", [3, 700])
def test_expired_maxvol_barrier_leaves_no_active_set(api, n):
    """The swaps change A and A^-1 in place: when a barrier of theirs gives up, nothing may go on with
    what is left of them (few and many blocks)."""
    desc = api.make_desc(2, 2, 24)
    m = api.mtp_describe(desc)["n_params"]
    model = api.mtp_load(desc, np.zeros(m))
    A0 = torch.tensor(synth.diag_dominant(24, m))
    B = torch.tensor(synth.rng(25).normal(size=(n, m)) * A0.abs().max().item())
    api.mtp_set_active_set(model, A0.cuda())
    try:
        api.mtp_debug_inject(api.MTP_FAULT_MAXVOL_WAIT, 1)
        with pytest.raises(api.MtpError) as e:
            api.mtp_maxvol(model, B)
    finally:
        api.mtp_debug_inject(api.MTP_FAULT_MAXVOL_WAIT, 0)
    assert e.value.name == "MTP_ERR_TIMEOUT"
    b = api.Batch(synth.fcc_unary_108(seed=26))
    nb = api.mtp_build_neighbors(model, b)
    for call in (lambda: api.mtp_get_active_set(model), lambda: api.mtp_get_active_inverse(model),
                 lambda: api.mtp_grade(model, b, nb, "fp64"), lambda: api.mtp_maxvol(model, B)):
        with pytest.raises(api.MtpError) as e:
            call()
        assert "no active set" in str(e.value)
    api.mtp_set_active_set(model, A0.cuda())
    src, swaps = api.mtp_maxvol(model, B)
    A_ref, src_ref, swaps_ref = AS.maxvol(A0.numpy(), B.numpy(), 1e-3, 1_000_000)
    assert swaps == swaps_ref
    np.testing.assert_array_equal(api.mtp_get_active_set(model).cpu().numpy(), A_ref)
