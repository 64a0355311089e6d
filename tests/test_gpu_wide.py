"""FP64 and dual-number pass (lists of pairs shared by a warp's neighborhoods, Horner adjoint)
against the oracle: every parity of the level, one to four species, empty and one-pair
neighborhoods between full ones, lists of atoms in any order, more atoms than a launch has warps."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2304_13144_gb300 import synth

pytestmark = pytest.mark.gpu


def setup(types, lev, n, seed):
    md = O.OracleModel(types, lev, 2.0, 5.0)
    nu_sum = [sum(nu for _, nu in labs) for labs, _ in md.basis]
    theta = synth.draw_theta(seed, types, md.n_rad, 8, nu_sum, [len(labs) for labs, _ in md.basis], 2.0, 5.0, 42.0)
    g = synth.rng(seed)
    pos, cell, _ = synth.cubic_supercell(synth._FCC, 3.6, n)
    full = synth.single(pos + g.normal(0, 0.1, pos.shape), g.integers(0, types, len(pos)), cell)
    far = np.array([[0.0, 0, 0], [20, 0, 0], [22.5, 0, 0], [0, 20, 0], [0, 0, 30]])
    dilute = synth.single(far, g.integers(0, types, len(far)), 60.0 * np.eye(3), (0, 0, 0))
    return md, theta, synth.concat([dilute, full, dilute])


def rel(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("types,lev,n", [(1, 4, 2), (2, 7, 2), (3, 10, 2), (1, 14, 2), (2, 18, (3, 2, 2)), (4, 22, 1), (3, 12, 9)])
def test_fp64_pass_matches_oracle(native_lib, types, lev, n):
    from paper_2304_13144_gb300 import api
    md, theta, bnp = setup(types, lev, n, 80 + lev)
    ref = O.efs(md, theta, bnp)
    model = api.mtp_load(api.make_desc(types, lev), theta)
    b = api.Batch(bnp)
    nb = api.mtp_build_neighbors(model, b)
    o = {k: v.cpu().numpy() for k, v in api.mtp_energy_forces_stress_atoms(model, b, nb, "fp64").items()}
    assert np.abs(o["site_energy"] - ref["V"]).max() <= 1e-10 * max(1.0, np.abs(ref["V"]).max())
    assert rel(o["forces"], ref["F"]) <= 1e-10
    assert rel(o["virial"], ref["W"]) <= 1e-10
    N = len(bnp["type"])
    pick = np.r_[np.arange(N)[::-1][:40], 0, 1, 2, 1]        # any order, repeats, empty neighborhoods
    rows = O.site_rows(md, theta, bnp["type"], ref["nbr"])
    got = api.mtp_param_rows(model, b, nb, "fp64", torch.tensor(pick)).cpu().numpy()
    assert rel(got, rows[pick]) <= 1e-10
    assert rel(api.mtp_param_rows(model, b, nb, "mixed").cpu().numpy(), rows) <= 2e-5


@pytest.mark.parametrize("types,lev,prec", [(1, 6, "fp64"), (3, 10, "fp64"), (2, 16, "fp64"), (2, 10, "mixed"), (2, 20, "mixed")])
def test_train_step_matches_oracle(native_lib, types, lev, prec):
    from paper_2304_13144_gb300 import api
    md, theta, bnp = setup(types, lev, 2, 90 + lev)
    g = synth.rng(7)
    K, N = len(bnp["cell"]), len(bnp["type"])
    E, F, W = g.normal(size=K), g.normal(size=(N, 3)), g.normal(size=(K, 9))
    L, grad, _ = O.loss_and_grad(md, theta, bnp, E, F, W.reshape(K, 3, 3), 1.0, 0.01, 1e-3)
    model = api.mtp_load(api.make_desc(types, lev), theta)
    b = api.Batch(bnp)
    nb = api.mtp_build_neighbors(model, b)
    loss, got = api.mtp_train_step(model, b, nb, torch.tensor(E), torch.tensor(F), torch.tensor(W), 1.0, 0.01, 1e-3, prec)
    tol = 1e-10 if prec == "fp64" else 1e-5
    assert abs(loss.item() - L) <= tol * abs(L)
    assert rel(got.cpu().numpy(), grad) <= tol


def test_without_memory_for_the_workspace_the_generic_kernel_answers(native_lib):
    """Its moments cost a value per moment and neighborhood: a call that cannot have them still runs."""
    from paper_2304_13144_gb300 import api
    md, theta, bnp = setup(2, 12, 2, 97)
    model = api.mtp_load(api.make_desc(2, 12), theta)
    b = api.Batch(bnp)
    nb = api.mtp_build_neighbors(model, b)
    try:
        api.mtp_debug_inject(api.MTP_FAULT_DEVICE_ALLOC, 1)
        plain = api.mtp_param_rows(model, b, nb, "fp64").cpu().numpy()
    finally:
        api.mtp_debug_inject(api.MTP_FAULT_DEVICE_ALLOC, 0)
    assert rel(plain, api.mtp_param_rows(model, b, nb, "fp64").cpu().numpy()) <= 1e-10
