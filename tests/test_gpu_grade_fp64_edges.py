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
    for f in (A.MTP_FAULT_DEVICE_ALLOC, A.MTP_FAULT_GRADE_WAIT):
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
