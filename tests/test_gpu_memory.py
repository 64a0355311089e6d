"""Calls near the limit of device memory (host-side injection of failing growths): what a call can do
without is taken last, and is what it goes without."""
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
    for f in (A.MTP_FAULT_DEVICE_ALLOC, A.MTP_FAULT_ALLOC_SKIP):
        A.mtp_debug_inject(f, 0)


class fail_growth:
    """Within: the device allocation after `after` growths of workspaces fails."""

    def __init__(self, api, after):
        self.api, self.after = api, after

    def __enter__(self):
        self.api.mtp_debug_inject(self.api.MTP_FAULT_ALLOC_SKIP, self.after)
        self.api.mtp_debug_inject(self.api.MTP_FAULT_DEVICE_ALLOC, 1)

    def __exit__(self, *exc):
        self.api.mtp_debug_inject(self.api.MTP_FAULT_DEVICE_ALLOC, 0)
        self.api.mtp_debug_inject(self.api.MTP_FAULT_ALLOC_SKIP, 0)


def theta_of(types, lev, seed=5):
    md = O.OracleModel(types, lev, 2.0, 5.0)
    nu_sum = [sum(nu for _, nu in labs) for labs, _ in md.basis]
    return synth.draw_theta(seed, types, md.n_rad, 8, nu_sum, [len(labs) for labs, _ in md.basis], 2.0, 5.0, 42.0)


CALLS = ["step", "config_rows", "vjp", "config_grade", "neighborhood_grade", "train"]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("what", CALLS)
def test_optional_growths_come_last(api, what, prec):
    """One failing growth after the other, each on a fresh model: from the first call that gets by on, all
    do (a failing growth that is not needed is never followed by one that is), with the results of a call
    that has what it wants."""
    types, lev = 2, 12
    theta = theta_of(types, lev)
    bnp = synth.training_batch(seed=4, n_cfg=6, n_types=types, lo=8, hi=64)
    b = api.Batch(bnp)
    K, N = b.n_cfg, b.n_atoms
    g = synth.rng(8)
    E, F, W = (torch.tensor(g.normal(size=s)) for s in (K, (N, 3), (K, 9)))
    gE = torch.tensor(g.normal(size=K), device="cuda")
    A = torch.tensor(synth.diag_dominant(6, theta.size), device="cuda")

    def fresh():
        model = api.mtp_load(api.make_desc(types, lev), theta)
        api.mtp_set_active_set(model, A)
        return model, api.mtp_build_neighbors(model, b)

    model, nb = fresh()
    forces = api.mtp_energy_forces_stress(model, b, nb, prec)["forces"]

    def call(model, nb):
        if what == "step":
            o = api.mtp_step(model, b, nb, prec)
            return [o["energy"], o["forces"], o["virial"], o["gamma"]]
        if what == "config_rows":
            return [api.mtp_config_rows(model, b, nb, prec)]
        if what == "vjp":
            return list(api.mtp_energy_vjp(model, b, nb, gE, forces, prec=prec))
        if what == "train":
            return list(api.mtp_train_step(model, b, nb, E, F, W, 1.0, 0.01, 1e-3, prec))
        mode = "configuration" if what == "config_grade" else "neighborhood"
        return [api.mtp_config_grade(model, b, nb, prec, mode)["gamma"]]

    ref = [t.cpu().numpy() for t in call(*fresh())]
    tol = 1e-10 if prec == "fp64" else 2e-5
    passed = []
    for after in range(16):
        model, nb = fresh()
        with fail_growth(api, after):
            try:
                out = call(model, nb)
                passed.append(True)
            except api.MtpError as e:
                assert e.name == "MTP_ERR_CUDA" and "injected" in str(e)
                passed.append(False)
                continue
        for x, y in zip(out, ref):
            x = x.cpu().numpy()
            assert np.abs(x - y).max() <= tol * max(1.0, np.abs(y).max()), (after, passed)
    assert passed == sorted(passed), passed
    assert passed[-1] and not passed[0]


def test_kept_workspace_is_given_back_where_a_call_needs_memory(api):
    """The FP64 pass keeps its workspace between calls.  A later call that cannot grow what it needs runs
    again after giving it back; a second failure is reported."""
    theta = theta_of(2, 12)
    b = api.Batch(synth.training_batch(seed=4, n_cfg=6, n_types=2, lo=8, hi=64))
    model = api.mtp_load(api.make_desc(2, 12), theta)
    nb = api.mtp_build_neighbors(model, b)
    ref = api.mtp_energy_forces_stress(api.mtp_load(api.make_desc(2, 12), theta), b, nb, "mixed")["forces"]
    rows = api.mtp_param_rows(model, b, nb, "fp64")          # takes the workspace, and nothing else
    with fail_growth(api, 0):
        out = api.mtp_energy_forces_stress(model, b, nb, "mixed")["forces"]
    assert torch.equal(out, ref)
    with fail_growth(api, 0):                                 # the workspace is gone: to be taken again
        plain = api.mtp_param_rows(model, b, nb, "fp64")
    assert not torch.equal(plain, rows)                       # (the generic kernel's rounding)
    assert (plain - rows).abs().max() <= 1e-10 * rows.abs().max()
    assert torch.equal(api.mtp_param_rows(model, b, nb, "fp64"), rows)
    other = api.mtp_load(api.make_desc(2, 12), theta)
    with fail_growth(api, 0):                                 # nothing to give back
        with pytest.raises(api.MtpError) as e:
            api.mtp_energy_forces_stress(other, b, nb, "mixed")
    assert e.value.name == "MTP_ERR_CUDA"


def test_a_captured_workspace_stays(api):
    """A graph holds the workspace's address: it is kept although another call fails for want of memory."""
    theta = theta_of(2, 12)
    b = api.Batch(synth.training_batch(seed=4, n_cfg=6, n_types=2, lo=8, hi=64))
    model = api.mtp_load(api.make_desc(2, 12), theta)
    nb = api.mtp_build_neighbors(model, b)
    dev = {"dtype": torch.float64, "device": "cuda"}
    out = {"energy": torch.empty(b.n_cfg, **dev), "forces": torch.empty((b.n_atoms, 3), **dev),
           "virial": torch.empty((b.n_cfg, 3, 3), **dev)}
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        api.mtp_step(model, b, nb, "fp64", out=out, grade=False)
    torch.cuda.synchronize()
    ref = {k: v.clone() for k, v in out.items()}
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        api.mtp_step(model, b, nb, "fp64", out=out, grade=False)
    big = api.Batch(synth.training_batch(seed=5, n_cfg=8, n_types=2, lo=100, hi=200))
    nb2 = api.mtp_build_neighbors(model, big)
    with fail_growth(api, 0):
        with pytest.raises(api.MtpError):
            api.mtp_config_rows(model, big, nb2, "mixed")
    for v in out.values():
        v.zero_()
    graph.replay()
    torch.cuda.synchronize()
    for k, v in out.items():
        assert torch.equal(v, ref[k]), k


@pytest.mark.parametrize("lev", [8, 16, 24])
def test_mixed_rows_take_no_workspace_that_nothing_uses(api, lev):
    """FP32 rows of the shapes of the single kernel (all levels of it but 24 here) need no growth: the
    armed failure is still there for the next call."""
    theta = theta_of(1, lev)
    b = api.Batch(synth.fcc_unary_108())
    model = api.mtp_load(api.make_desc(1, lev), theta)
    nb = api.mtp_build_neighbors(model, b)
    with fail_growth(api, 0):
        api.mtp_param_rows(model, b, nb, "mixed")
        if lev == 24:
            api.mtp_energy_forces_stress(model, b, nb, "mixed")
        else:
            with pytest.raises(api.MtpError) as e:
                api.mtp_energy_forces_stress(model, b, nb, "mixed")
            assert "injected" in str(e.value)


def test_autotune_gives_its_outputs_back(api):
    """Its energies, forces and grades (2 MB for this batch) go when it returns."""
    desc = api.make_desc(1, 4)
    model = api.mtp_load(desc, np.full(api.mtp_describe(desc)["n_params"], 0.01))
    pos, cell, _ = synth.cubic_supercell(synth._FCC, 3.6, 26)
    b = api.Batch(synth.single(pos + synth.rng(2).normal(0, 0.1, pos.shape), np.zeros(len(pos), int), cell))
    nb = api.mtp_build_neighbors(model, b)
    api.mtp_autotune(model, b, nb, "mixed")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(16):
        api.mtp_autotune(model, b, nb, "mixed")
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 8 << 20
