"""A configuration with atoms at one and the same place (no direction between
them: its own energy and forces are not numbers) leaves every other system of
the batch, and every atom out of its reach, bitwise what it is without it.
Several species: the pair batches of an atom are then staged in groups padded
to multiples of 8, in slots that earlier atoms of the same warp have used."""
import numpy as np
import pytest

from paper_2310_08439_gb300 import inputs as I

pytestmark = pytest.mark.gpu
RC = 5.0


def _systems(n_species, broken):
    """Four intact crystals (19,000 atoms: several for each warp of the pass) and one gas of 400 atoms in 200 places (broken) or
    in 400 places; the atom and species counts, and so the order of
    evaluation, are the same in both."""
    rng = np.random.default_rng(40 + n_species)
    out = []
    for reps, a in (((12, 12, 11), 3.7), ((11, 11, 11), 3.6), ((12, 12, 12), 3.65), ((5, 5, 4), 3.8)):
        pos, box = I.lattice("fcc", reps, a)
        types = rng.integers(0, n_species, len(pos)).astype(np.int32)
        out.append(I.System(I.jitter_and_wrap(pos, box, 0.1, rng), types, box, np.ones(3, np.int32)))
    pos, box = I.lattice("fcc", (5, 5, 4), 3.7)
    types = rng.integers(0, n_species, len(pos)).astype(np.int32)
    pos = I.jitter_and_wrap(pos, box, 0.1, rng)
    if broken:
        pos[1::2] = pos[::2]
    out.insert(2, I.System(pos, types, box, np.ones(3, np.int32)))
    return out


@pytest.mark.parametrize("n_species,K,table", [(2, 16, 0), (3, 8, 0), (5, 16, 0), (1, 16, 64), (2, 16, 64), (3, 8, 256)])
def test_other_systems_of_a_batch_stay_as_they_are(tmdlib, n_species, K, table):
    """With a table the coincident pair's interval stays inside it."""
    m = tmdlib.Model(I.random_model(n_species, K, RC, [32, 32], seed=K + n_species))
    if table:
        m.set_radial_table(table)
    res = []
    for broken in (False, True):
        systems = _systems(n_species, broken)
        b = tmdlib.Batch(systems)
        E, W = b.compute(m, list(range(len(systems))))
        res.append((E, W, [b.get_system(k)[2] for k in range(len(systems))]))
    for k in (0, 1, 3, 4):
        assert np.isfinite(res[0][0][k])
        assert res[1][0][k] == res[0][0][k], k
        assert np.array_equal(res[1][1][k], res[0][1][k]), k
        assert np.array_equal(res[1][2][k], res[0][2][k]), k
    assert not np.isfinite(res[1][0][2])


def test_atoms_out_of_reach_stay_as_they_are(tmdlib):
    """One evaluation: two atoms at one place in a corner of a large box."""
    import torch
    rng = np.random.default_rng(8)
    pos, box = I.lattice("fcc", (16, 16, 16), 3.7)
    types = rng.integers(0, 2, len(pos)).astype(np.int32)
    pos = I.jitter_and_wrap(pos, box, 0.1, rng)
    m = tmdlib.Model(I.random_model(2, 16, RC, [32, 32], seed=9))
    near = np.argsort(((pos - pos[0] + box / 2) % box - box / 2).__pow__(2).sum(1))[1:9]
    res = []
    for broken in (False, True):
        x = pos.copy()
        if broken:
            x[near] = x[0]
        nl = tmdlib.NeighborList()
        p, t = torch.as_tensor(x, device="cuda"), torch.as_tensor(types, device="cuda")
        nl.build(p, t, box, np.ones(3, np.int32), RC)
        res.append({k: v.cpu().numpy() for k, v in tmdlib.evaluate(m, nl, p, t, box).items()})
    d = (pos - pos[0] + box / 2) % box - box / 2
    far = np.sqrt((d ** 2).sum(1)) > 2 * RC + np.sqrt((d[near] ** 2).sum(1)).max() + 0.1
    assert 8000 < far.sum() < len(pos)
    assert np.isfinite(res[0]["e_atom"]).all() and not np.isfinite(res[1]["e_atom"]).all()
    assert np.array_equal(res[1]["e_atom"][far], res[0]["e_atom"][far])
    assert np.array_equal(res[1]["forces"][far], res[0]["forces"][far])
