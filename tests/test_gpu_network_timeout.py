"""What a caller sees when the network kernel gives up waiting (the self-test
marks one launch as such; no wait runs out): no entry point hands on results of
a partial evaluation as valid ones, and the next evaluation is the usual one,
bit for bit."""
import numpy as np
import pytest

from paper_2310_08439_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _cleared(tmdlib):
    yield
    with pytest.raises(tmdlib.TmdError) as e:   # every test here has one
        tmdlib.device_status()
    assert e.value.status == tmdlib.ERR_TIMEOUT
    assert tmdlib.device_status() == 0


def _case(n_species=2, seed=3):
    rng = np.random.default_rng(seed)
    pos, box = I.lattice("fcc", (4, 4, 4), 3.7)
    types = rng.integers(0, n_species, len(pos)).astype(np.int32)
    masses = np.asarray([55.8, 63.5])[types]
    s = I.System(I.jitter_and_wrap(pos, box, 0.1, rng), types, box, np.ones(3, np.int32),
                 vel=I.maxwell_velocities(masses, 300.0, rng), masses=masses)
    return I.random_model(n_species, 16, 4.5, [64, 64], seed=seed), s


def _model(tmd, p, **kw):
    m = tmd.Model(p, **kw)
    m.tuning = {"tile_rows": 128, "pair_blocks_per_sm": 0}   # on the tensor cores
    return m


def _dev(s):
    import torch
    return torch.as_tensor(s.pos, device="cuda"), torch.as_tensor(s.types, device="cuda")


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_enqueued_calls_give_nan(tmdlib, precision):
    import torch
    p, s = _case()
    m = _model(tmdlib, p, precision=precision)
    nl = tmdlib.NeighborList()
    pos, types = _dev(s)
    nl.build(pos, types, s.box, s.pbc, p.rc)
    good = {k: v.cpu().numpy() for k, v in tmdlib.evaluate(m, nl, pos, types, s.box).items()}
    tmdlib.selftest_network_timeout()
    bad = {k: v.cpu().numpy() for k, v in tmdlib.evaluate(m, nl, pos, types, s.box).items()}
    assert np.isnan(bad["energy"]).all() and np.isnan(bad["virial"]).all() and np.isnan(bad["forces"]).all()
    assert np.isnan(bad["e_atom"]).sum() == len(s.pos) - (len(s.pos) - 1) // 128 * 128   # the last tile
    again = {k: v.cpu().numpy() for k, v in tmdlib.evaluate(m, nl, pos, types, s.box).items()}
    for k in good:
        assert np.array_equal(again[k], good[k]), k
    G, dG = tmdlib.descriptors(m, nl, pos, types, s.box, with_grad=True)
    tmdlib.selftest_network_timeout()
    G1, dG1 = tmdlib.descriptors(m, nl, pos, types, s.box, with_grad=True)
    assert torch.equal(G, G1) and torch.isnan(dG1).any() and not torch.isnan(dG).any()
    off, nbr, sh = nl.export()
    shift4 = np.ascontiguousarray(np.concatenate([sh, s.types[nbr].astype(np.int8)[:, None]], axis=1))
    dev = lambda a: torch.as_tensor(a, device="cuda")
    e, f = torch.zeros(1, dtype=torch.float64, device="cuda"), torch.zeros((s.n, 3), device="cuda")
    for armed in (False, True, False):
        if armed:
            tmdlib.selftest_network_timeout()
        tmdlib.compute_noalloc(m, dev(off), dev(nbr), dev(shift4), pos, types, s.box, energy=e, forces=f)
        assert bool(torch.isnan(e).all()) == armed and bool(torch.isnan(f).all()) == armed


def test_single_steps_report_it(tmdlib):
    p, s = _case()
    m = _model(tmdlib, p)
    g = tmdlib.System(s.n, s.box, s.pbc, skin=0.0)
    g.set_state(s.pos, s.vel, s.types, s.masses)
    ref = g.step(m, 1.0, 3)
    for thermo in (True, False):
        g.set_state(s.pos, s.vel, s.types, s.masses)
        g.step(m, 1.0, 1)
        tmdlib.selftest_network_timeout()
        with pytest.raises(tmdlib.TmdError) as e:
            g.step(m, 1.0, 1, thermo=thermo)
            g.get_state()
        assert e.value.status == tmdlib.ERR_TIMEOUT
        with pytest.raises(tmdlib.TmdError):    # until a state is set
            g.get_state()
    g.set_state(s.pos, s.vel, s.types, s.masses)
    assert g.step(m, 1.0, 3)["e_pot"] == ref["e_pot"]


@pytest.mark.parametrize("rebuild_every", [0, 5])
def test_a_run_of_steps_is_stepped_again(tmdlib, rebuild_every):
    p, s = _case()
    m = _model(tmdlib, p)
    out = []
    for armed in (False, True):
        g = tmdlib.System(s.n, s.box, s.pbc, skin=1.0)
        g.set_state(s.pos, s.vel, s.types, s.masses)
        g.step(m, 1.0, 4, rebuild_every=rebuild_every)
        if armed:
            tmdlib.selftest_network_timeout()
        th = g.step(m, 1.0, 5, rebuild_every=rebuild_every)
        c = g.counters()
        assert c["steps"] == 9 and (c["reruns"] >= 1) == armed
        out.append((*g.get_state(), th["e_pot"]))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_a_step_before_a_run_is_not_taken_for_one_of_it(tmdlib):
    p, s = _case()
    m = _model(tmdlib, p)
    g = tmdlib.System(s.n, s.box, s.pbc, skin=1.0)
    g.set_state(s.pos, s.vel, s.types, s.masses)
    tmdlib.selftest_network_timeout()
    g.step(m, 1.0, 0, thermo=False)             # the first forces
    with pytest.raises(tmdlib.TmdError) as e:
        g.step(m, 1.0, 6, thermo=False)
        g.get_state()
    assert e.value.status == tmdlib.ERR_TIMEOUT


def test_host_state_and_host_evaluation_report_it(tmdlib):
    p, s = _case()
    m = _model(tmdlib, p)
    g = tmdlib.System(s.n, s.box, s.pbc, skin=0.0)
    g.set_state(s.pos, s.vel, s.types, s.masses)
    first = None
    for armed in (False, True, False):
        pos, vel, f = s.pos.copy(), s.vel.copy(), np.zeros((s.n, 3), np.float32)
        if armed:
            tmdlib.selftest_network_timeout()
            with pytest.raises(tmdlib.TmdError) as e:
                g.step_host(m, pos, vel, f, 1.0, 1)
            assert e.value.status == tmdlib.ERR_TIMEOUT
        else:
            g.step_host(m, pos, vel, f, 1.0, 1)
            assert first is None or np.array_equal(first, f)
            first = f
    nl = tmdlib.NeighborList()
    e, f, w = np.zeros(1), np.zeros((s.n, 3), np.float32), np.zeros(9)
    for energy in (e, None):
        tmdlib.evaluate_host(m, nl, s.pos, s.types, s.box, s.pbc, energy, f, w)
        assert np.isfinite(f).all()
        tmdlib.selftest_network_timeout()
        with pytest.raises(tmdlib.TmdError) as err:
            tmdlib.evaluate_host(m, nl, s.pos, s.types, s.box, s.pbc, energy, f, w)
        assert err.value.status == tmdlib.ERR_TIMEOUT


def test_batches_report_it(tmdlib):
    p, s = _case()
    m = _model(tmdlib, p)
    b = tmdlib.Batch([s, s, s], skin=1.0)
    ids = [0, 1, 2]
    E, W = b.compute(m, ids)
    tmdlib.selftest_network_timeout()
    with pytest.raises(tmdlib.TmdError) as e:
        b.compute(m, ids)
    assert e.value.status == tmdlib.ERR_TIMEOUT
    E1, W1 = b.compute(m, ids)
    assert np.array_equal(E, E1) and np.array_equal(W, W1)
    tmdlib.selftest_network_timeout()
    with pytest.raises(tmdlib.TmdError) as e:
        b.step(m, ids, 1.0, 2)
    assert e.value.status == tmdlib.ERR_TIMEOUT
    b2 = tmdlib.Batch([s, s, s], skin=1.0)
    assert np.isfinite([t["e_pot"] for t in b2.step(m, ids, 1.0, 2)]).all()
