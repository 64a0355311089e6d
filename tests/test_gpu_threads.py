"""Neighbor lists of different batches built at once, in several threads and streams, with one model."""
import threading

import numpy as np
import pytest
import torch

from paper_2304_13144_gb300 import synth

pytestmark = pytest.mark.gpu

BUILDS = 40


def test_lists_built_at_once_with_one_model(native_lib):
    """Each thread rebuilds its own list for cells of its own size, and of another size and back, so
    that offsets, cells and pair counts differ between the builds in flight; every list must be the one
    that a build alone gives.  One thread's positions are not finite: only its builds fail."""
    from paper_2304_13144_gb300 import api
    model = api.mtp_load(api.make_desc(1, 4), np.zeros(api.mtp_describe(api.make_desc(1, 4))["n_params"]))
    g = synth.rng(77)

    def batch(n, sigma=0.1):
        pos, cell, _ = synth.cubic_supercell(synth._FCC, 3.6, n)
        return api.Batch(synth.single(pos + g.normal(0, sigma, pos.shape), np.zeros(len(pos), int), cell))

    work = [[batch(2), batch(3)], [batch(5), batch(4)], [batch(12), batch(9)], [batch(3), batch(14)]]
    bad = batch(4)
    bad.pos[7, 1] = float("nan")
    ref = [[api.mtp_nbr_export(api.mtp_build_neighbors(model, b), b) for b in w] for w in work]
    torch.cuda.synchronize()
    errors, got = [], [[None, None] for _ in work]
    start = threading.Barrier(len(work) + 1)

    def build(t):
        try:
            s = torch.cuda.Stream()
            lists = [None, None]
            start.wait()
            for k in range(BUILDS):
                for e, b in enumerate(work[t]):
                    lists[e] = api.mtp_build_neighbors(model, b, lists[e], stream=s)
                    n, pairs = lists[e].size()
                    assert n == b.n_atoms and pairs == ref[t][e]["j"].numel()
            got[t] = lists
        except Exception as e:   # reported by the test below
            errors.append(f"thread {t}: {e!r}")

    def fail():
        s = torch.cuda.Stream()
        start.wait()
        for k in range(BUILDS):
            try:
                api.mtp_build_neighbors(model, bad, stream=s)
                errors.append("non-finite positions accepted")
            except api.MtpError as e:
                if e.name != "MTP_ERR_NUMERIC":
                    errors.append(repr(e))

    threads = [threading.Thread(target=build, args=(t,)) for t in range(len(work))] + [threading.Thread(target=fail)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for t, w in enumerate(work):
        for e, b in enumerate(w):
            ex = api.mtp_nbr_export(got[t][e], b)
            for k in ("off", "j", "img", "r"):
                assert torch.equal(ex[k], ref[t][e][k]), (t, e, k)


@pytest.mark.parametrize("prec,lev", [("fp64", 12), ("mixed", 24)])
def test_parameter_rows_at_once_with_one_model(native_lib, prec, lev):
    """Threads take rows of lists of their own sizes (growing and shrinking the workspace), each on its
    stream, while another runs energies and forces: the rows of every call are those of a call alone."""
    from oracle import oracle as O
    from paper_2304_13144_gb300 import api
    types = 2
    md = O.OracleModel(types, lev, 2.0, 5.0)
    nu_sum = [sum(nu for _, nu in labs) for labs, _ in md.basis]
    theta = synth.draw_theta(5, types, md.n_rad, 8, nu_sum, [len(labs) for labs, _ in md.basis], 2.0, 5.0, 42.0)
    g = synth.rng(78)
    pos, cell, _ = synth.cubic_supercell(synth._FCC, 3.6, 6)
    b = api.Batch(synth.single(pos + g.normal(0, 0.1, pos.shape), g.integers(0, types, len(pos)), cell))
    model = api.mtp_load(api.make_desc(types, lev), theta)
    nb = api.mtp_build_neighbors(model, b)
    forces = api.mtp_energy_forces_stress(model, b, nb, prec)["forces"]
    lists = [[torch.tensor(g.integers(0, b.n_atoms, n), device="cuda") for n in sizes]
             for sizes in ((5, 700, 40), (864, 1, 300), (64, 900, 7))]
    ref = [[api.mtp_param_rows(model, b, nb, prec, a).clone() for a in ls] for ls in lists]
    model = api.mtp_load(api.make_desc(types, lev), theta)     # (no workspace yet)
    torch.cuda.synchronize()
    errors = []
    start = threading.Barrier(len(lists) + 1)

    def rows(t):
        try:
            s = torch.cuda.Stream()
            start.wait()
            with torch.cuda.stream(s):
                for k in range(20):
                    got = [api.mtp_param_rows(model, b, nb, prec, a) for a in lists[t]]
                    s.synchronize()
                    for x, y in zip(got, ref[t]):
                        if not torch.equal(x, y):
                            errors.append(f"thread {t}, pass {k}: rows differ")
        except Exception as e:
            errors.append(f"thread {t}: {e!r}")

    def energies():
        try:
            s = torch.cuda.Stream()
            start.wait()
            with torch.cuda.stream(s):
                for k in range(40):
                    f = api.mtp_energy_forces_stress(model, b, nb, prec)["forces"]
                    s.synchronize()
                    if not torch.equal(f, forces):
                        errors.append("forces differ")
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=rows, args=(t,)) for t in range(len(lists))] + [threading.Thread(target=energies)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:5]


def test_lists_of_different_shared_memory_built_at_once(native_lib):
    """One-block binning takes 57 KB of shared memory for one of these dilute gases and 87 KB for the
    other: neither thread's launches may find the kernel limited to the other's."""
    from paper_2304_13144_gb300 import api
    desc = api.make_desc(1, 4)
    model = api.mtp_load(desc, np.zeros(api.mtp_describe(desc)["n_params"]))
    g = synth.rng(79)
    batches = [api.Batch(synth.single(g.uniform(0, L, (n, 3)), np.zeros(n, int), L * np.eye(3)))
               for n, L in ((8000, 95.5), (6000, 80.5))]
    pairs = [api.mtp_build_neighbors(model, b).size()[1] for b in batches]
    torch.cuda.synchronize()
    errors = []
    start = threading.Barrier(2)

    def build(t):
        s = torch.cuda.Stream()
        nb = None
        start.wait()
        try:
            for k in range(400):
                nb = api.mtp_build_neighbors(model, batches[t], nb, stream=s)
                assert nb.size()[1] == pairs[t]
        except Exception as e:
            errors.append(f"thread {t}, build {k}: {e!r}")

    threads = [threading.Thread(target=build, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
