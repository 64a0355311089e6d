"""Neighbor build on both sides of each size rule (one-block binning up to 8,192 atoms, count pass by
warps below 65,536, cells that scan more than 32 bins), and the kept plan of a reused list."""
import numpy as np
import pytest
import torch

from nbr_check import check_reverse
from oracle import oracle as O
from paper_2304_13144_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api(native_lib):
    from paper_2304_13144_gb300 import api as A
    return A


def model(api):
    desc = api.make_desc(1, 4)
    return api.mtp_load(desc, np.zeros(api.mtp_describe(desc)["n_params"]))


def listed(api, nb, b):
    ex = {k: v.cpu().numpy() for k, v in api.mtp_nbr_export(nb, b).items()}
    i = np.repeat(np.arange(len(ex["off"]) - 1), np.diff(ex["off"]))
    return np.column_stack([i, ex["j"], ex["img"]]), ex


def in_order(a):
    return a[np.lexsort(a.T[::-1])]


@pytest.mark.parametrize("reps,cut", [((16, 16, 16), 0), ((16, 16, 16), 1), ((16, 16, 17), 0), ((32, 32, 32), 1), ((32, 32, 32), 0),
                                      ((1, 2, 7), 0), ((2, 2, 2), 3), ((1, 182, 182), 0)])
def test_list_matches_oracle_around_the_rules(api, reps, cut):
    g = synth.rng(sum(reps) + cut)
    pos, cell, _ = synth.cubic_supercell(synth._BCC, 2.87, reps)
    bnp = synth.single((pos + g.normal(0, 0.1, pos.shape))[:len(pos) - cut], np.zeros(len(pos) - cut, int), cell)
    b = api.Batch(bnp)
    nb = api.mtp_build_neighbors(model(api), b)
    got, ex = listed(api, nb, b)
    ref = O.batch_neighbors(bnp, 5.0, brute=len(bnp["type"]) < 500)
    want = np.column_stack([O.pair_centers(ref["off"]), ref["j"], ref["img"]])
    np.testing.assert_array_equal(ex["off"], ref["off"])
    np.testing.assert_array_equal(in_order(got), in_order(want))
    check_reverse(api, nb, b)


def test_reused_list_follows_cells_offsets_and_periodicity(api):
    """A list built again after each change of the batch equals a new list, bit for bit."""
    a = synth.training_batch(seed=5, n_cfg=6, n_types=1, lo=8, hi=64)
    cells = dict(a, cell=a["cell"] * 1.02)
    opened = dict(a, pbc=np.where(np.arange(18).reshape(6, 3) % 4 == 0, 0, 1).astype(np.uint8))
    moved = dict(a, atom_offset=np.r_[0, a["atom_offset"][1:-1] + 1, a["atom_offset"][-1]])
    m = model(api)
    nb = None
    for x in (a, a, cells, a, opened, moved, a):
        b = api.Batch(x)
        nb = api.mtp_build_neighbors(m, b, nb)
        got, ex = listed(api, nb, b)
        new, ex2 = listed(api, api.mtp_build_neighbors(m, b), b)
        np.testing.assert_array_equal(got, new)
        np.testing.assert_array_equal(ex["r"], ex2["r"])


def test_more_pairs_than_an_index_holds_are_refused(api):
    """256 atoms of a cell of 256 A^3 with a cut-off of 130 A have 2.4e9 pairs (9.2 million each);
    with 7,936 atoms beyond each other's reach the list is one of the largest that one block sums."""
    desc = api.make_desc(1, 4, r_cut=130.0)
    m = api.mtp_load(desc, np.zeros(api.mtp_describe(desc)["n_params"]))
    dense = np.stack(np.meshgrid(np.arange(8), np.arange(8), np.arange(4), indexing="ij"), -1).reshape(-1, 3) * 1.0
    far = np.stack(np.meshgrid(*[np.arange(20)] * 3, indexing="ij"), -1).reshape(-1, 3)[:7936] * 131.0
    bnp = synth.concat([synth.single(dense, np.zeros(256, int), np.diag([8.0, 8.0, 4.0])),
                        synth.single(far, np.zeros(7936, int), 2620.0 * np.eye(3), (0, 0, 0))])
    with pytest.raises(api.MtpError) as e:
        api.mtp_build_neighbors(m, api.Batch(bnp))
    assert e.value.name == "MTP_ERR_UNSUPPORTED" and "pairs" in str(e.value)
