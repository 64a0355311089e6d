"""The grouped contraction (four neighborhoods side by side, the default of the three-kernel pass)
against the contraction with one neighborhood's arrays per warp lane word: the same terms in the
same order, so bitwise the same outputs.  Sizes: remainders of four, fewer atoms than groups in
flight (words from global memory), more (shared or tensor memory), the largest level."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2304_13144_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lev,types,n,cut", [(8, 3, 1, 3), (8, 1, 17, 1), (12, 2, 14, 2), (16, 3, 3, 1), (16, 2, 14, 3),
                                             (20, 3, 2, 2), (20, 3, 11, 1), (24, 4, 4, 3)])
def test_grouped_contraction_is_bitwise_the_plain_one(native_lib, lev, types, n, cut):
    from paper_2304_13144_gb300 import api
    md = O.OracleModel(types, lev, 2.0, 5.0)
    nu_sum = [sum(nu for _, nu in labs) for labs, _ in md.basis]
    theta = synth.draw_theta(5, types, md.n_rad, 8, nu_sum, [len(labs) for labs, _ in md.basis], 2.0, 5.0, 42.0)
    g = synth.rng(lev + n)
    pos, cell, _ = synth.cubic_supercell(synth._FCC, 3.6, n)
    pos = (pos + g.normal(0, 0.1, pos.shape))[:len(pos) - cut]
    b = api.Batch(synth.single(pos, g.integers(0, types, len(pos)), cell))
    model = api.mtp_load(api.make_desc(types, lev), theta)
    api.mtp_set_active_set(model, torch.tensor(synth.diag_dominant(6, md.m), device="cuda"))
    nb = api.mtp_build_neighbors(model, b)
    out = []
    for shape in ((0, 0, 0, 0), (8, 1, 2, 2 if lev == 24 else 1)):
        api.mtp_set_split_shape(model, *shape)
        o = api.mtp_step(model, b, nb, "mixed")
        o.update(api.mtp_energy_forces_stress_atoms(model, b, nb, "mixed"))
        out.append({k: v.cpu().numpy() for k, v in o.items() if k != "flagged"})
    for k, v in out[0].items():
        assert np.array_equal(v, out[1][k]), k
