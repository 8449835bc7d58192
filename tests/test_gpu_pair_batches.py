"""The pair passes (k_desc, k_force) at the edges of their batches, against the
FP64 oracle at the FP32 bars.  A cluster of m + 1 atoms, all within the cutoff
of one another, gives every atom exactly m pairs: none, one, either side of 8
(operand columns of the descriptor contraction), 32 (one pair per lane), 58 to
64 (two pairs per lane, the batch length of each species count) and 96.
Several species fill the groups of a batch unevenly.  Each cluster is evaluated
alone (cached pairs), by the allocation-free call (pairs screened in the pass)
and all of them in one batch (virials per atom)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2310_08439_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PAIRS = [0, 1, 7, 8, 9, 31, 32, 33, 57, 58, 59, 60, 61, 62, 63, 64, 65, 95, 96, 97]
RC = 6.0


def _cluster(m, n_species, seed):
    rng = np.random.default_rng(seed)
    g = np.stack(np.meshgrid(*[np.arange(-4, 5)] * 3, indexing="ij"), -1).reshape(-1, 3) * 0.95
    g = g[np.argsort((g ** 2).sum(1), kind="stable")][:m + 1] + rng.uniform(-0.06, 0.06, (m + 1, 3))
    assert np.sqrt(((g[:, None] - g[None]) ** 2).sum(-1)).max() < RC
    box = np.full(3, 40.0)
    return I.System(g + 20.0, rng.integers(0, n_species, m + 1).astype(np.int32), box, np.zeros(3, np.int32))


def _model(S, K, systems):
    def make(scale=None):
        return I.random_model(S, K, RC, [16], seed=K + S, feature_scale=scale)
    s = systems[-1]
    G = O.evaluate(O.OracleModel(make()), s.pos, s.types, s.box, s.pbc, want_G=True)["G"]
    return make(np.repeat(np.sqrt((G ** 2).mean(axis=0)).reshape(1, -1), S, axis=0))


def _check(o, e, f, w, what):
    assert abs(e - o["energy"]) <= 1e-6 * abs(o["energy"]), what
    rms = float(np.sqrt((o["forces"] ** 2).mean()))
    assert np.abs(f - o["forces"]).max() <= 1e-5 * rms if rms else not f.any(), what
    assert np.abs(w - o["virial"]).max() <= 1e-5 * np.abs(o["virial"]).max(), what


@pytest.mark.parametrize("S,K,table", [(1, 8, 0), (1, 16, 256), (2, 16, 0), (3, 16, 256), (5, 8, 0), (1, 32, 0),
                                       (2, 64, 0), (1, 128, 0)])
def test_batch_edges(tmdlib, S, K, table):
    import torch
    systems = [_cluster(m, S, 100 * S + m) for m in PAIRS]
    p = _model(S, K, systems)
    m = tmdlib.Model(p)
    if table:
        m.set_radial_table(table)
    om = O.OracleModel(p, radial_table=table) if table else O.OracleModel(p)
    refs = [O.evaluate(om, s.pos, s.types, s.box, s.pbc) for s in systems]
    for s, o in zip(systems, refs):
        nl = tmdlib.NeighborList()
        pos = torch.as_tensor(s.pos, dtype=torch.float64, device="cuda")
        types = torch.as_tensor(s.types, dtype=torch.int32, device="cuda")
        nl.build(pos, types, s.box, s.pbc, RC)
        out = tmdlib.evaluate(m, nl, pos, types, s.box)
        _check(o, float(out["energy"].item()), out["forces"].double().cpu().numpy(),
               out["virial"].cpu().numpy().reshape(3, 3), ("alone", s.n))
        off, nbr, sh = nl.export()
        shift4 = np.zeros((len(nbr), 4), np.int8)
        shift4[:, :3] = sh
        shift4[:, 3] = s.types[nbr]
        if len(nbr):
            dev = lambda a, t: torch.as_tensor(np.ascontiguousarray(a), dtype=t, device="cuda")
            e, f = torch.zeros(1, dtype=torch.float64, device="cuda"), torch.zeros((s.n, 3), device="cuda")
            w = torch.zeros(9, dtype=torch.float64, device="cuda")
            tmdlib.compute_noalloc(m, dev(off, torch.int64), dev(nbr, torch.int32), dev(shift4, torch.int8), pos, types,
                                   s.box, energy=e, forces=f, virial=w)
            torch.cuda.synchronize()
            _check(o, float(e.item()), f.double().cpu().numpy(), w.cpu().numpy().reshape(3, 3), ("noalloc", s.n))
    b = tmdlib.Batch(systems)
    E, W = b.compute(m, list(range(len(systems))))
    for k, o in enumerate(refs):
        _check(o, E[k], b.get_system(k)[2].astype(np.float64), W[k], ("batch", systems[k].n))
