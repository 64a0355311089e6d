"""FP64 grade from exact slice products against an extended-precision product of the same rows and
inverse: row counts around the 128-row tile, K around the 64-wide chunk and above one accumulation
(1,024), rows and columns of very different magnitudes."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2304_13144_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("types,lev,atoms,spread", [(1, 16, 1, 0), (2, 12, 127, 0), (2, 16, 129, 12), (1, 14, 128, 3), (3, 20, 300, 0),
                                                    (3, 20, 64, 10), (4, 24, 40, 6)])
def test_sliced_grade_matches_extended_precision(native_lib, types, lev, atoms, spread):
    from paper_2304_13144_gb300 import api
    md = O.OracleModel(types, lev, 2.0, 5.0)
    nu_sum = [sum(nu for _, nu in labs) for labs, _ in md.basis]
    theta = synth.draw_theta(7, types, md.n_rad, 8, nu_sum, [len(labs) for labs, _ in md.basis], 2.0, 5.0, 42.0)
    g = synth.rng(lev + atoms)
    pos, cell, _ = synth.cubic_supercell(synth._FCC, 3.6, 5)
    pos = (pos + g.normal(0, 0.1, pos.shape))[:atoms]
    b = api.Batch(synth.single(pos, g.integers(0, types, len(pos)), cell))
    model = api.mtp_load(api.make_desc(types, lev), theta)
    nb = api.mtp_build_neighbors(model, b)
    m = model.n_params
    # rows of A by powers of ten: the rows of A^-1 and the terms of the product differ as much
    A = synth.diag_dominant(8, m) * 10.0 ** g.uniform(-spread / 2, spread / 2, (m, 1))
    api.mtp_set_active_set(model, torch.tensor(A, device="cuda"))
    out = api.mtp_grade(model, b, nb, "fp64")
    rows = api.mtp_param_rows(model, b, nb, "fp64").cpu().numpy().astype(np.longdouble)
    X = api.mtp_get_active_inverse(model).cpu().numpy().astype(np.longdouble)
    C = np.abs(np.stack([(r[:, None] * X).sum(0) for r in rows]))
    ref = C.max(1)
    got = out["gamma"].cpu().numpy()
    # FP64 rounding of the result, and m terms cut at 2^-63 of the row's largest balanced entry
    # (scales to the next power of two on both factors, dropped slice pairs: 2^-58 in all)
    tol = 2.0 ** -52 * ref + m * 2.0 ** -58 * (np.abs(rows) * np.abs(X).max(1)).max(1)
    assert (np.abs(got - ref) <= tol).all(), float((np.abs(got - ref) / tol).max())
    am = out["argmax"].cpu().numpy()
    assert (C[np.arange(len(ref)), am] >= ref - tol).all()
