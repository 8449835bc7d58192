"""Per-system sums of a batch (a cluster of blocks per system: E, W and the
kinetic terms) at the edges of its warps, blocks and strides: systems of 1 to
2,049 atoms together.  The kinetic energy is FP64 throughout: 1e-12 of numpy's
sum; E and W against the same system evaluated alone, whose totals come from
another reduction, at the FP32 bars."""
import numpy as np
import pytest

from paper_2310_08439_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SIZES = [1, 31, 32, 33, 255, 256, 257, 2047, 2048, 2049]


@pytest.mark.parametrize("n_species", [1, 3])
def test_sums_of_uneven_systems(tmdlib, n_species):
    import torch
    rng = np.random.default_rng(n_species)
    systems = []
    for n in SIZES:
        reps = int(np.ceil((n / 4) ** (1 / 3)))
        pos, box = I.lattice("fcc", (reps, reps, reps), 3.8)
        pos = I.jitter_and_wrap(pos, box, 0.1, rng)[:n]
        systems.append(I.System(pos, rng.integers(0, n_species, n).astype(np.int32), box, np.zeros(3, np.int32),
                                vel=rng.normal(0, 1e-3, (n, 3)), masses=rng.uniform(10, 200, n)))
    m = tmdlib.Model(I.random_model(n_species, 8, 4.5, [16], seed=1))
    b = tmdlib.Batch(systems)
    ids = list(range(len(SIZES)))
    E, W = b.compute(m, ids)
    th = b.step(m, ids, 1.0, 0)
    for k, s in enumerate(systems):
        nl = tmdlib.NeighborList()
        pos = torch.as_tensor(s.pos, dtype=torch.float64, device="cuda")
        types = torch.as_tensor(s.types, dtype=torch.int32, device="cuda")
        nl.build(pos, types, s.box, s.pbc, 4.5)
        out = tmdlib.evaluate(m, nl, pos, types, s.box)
        e, w = float(out["energy"].item()), out["virial"].cpu().numpy().reshape(3, 3)
        assert abs(E[k] - e) <= 1e-6 * abs(e) and abs(th[k]["e_pot"] - e) <= 1e-6 * abs(e), SIZES[k]
        assert np.abs(W[k] - w).max() <= 1e-5 * np.abs(w).max(), SIZES[k]
        kin = 0.5 * 103.6427 * float((s.masses[:, None] * s.vel ** 2).sum())
        assert abs(th[k]["e_kin"] - kin) <= 1e-12 * kin, SIZES[k]
