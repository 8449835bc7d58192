"""The FP32 network on the FP32 pipes (k_mlp, tiles of 32 and 64 atoms) against
the FP64 oracle, on networks that run there: hidden widths that are no multiples
of 16 or above 128, and all widths 64 with tile_rows 32 or 64.  The two tiles sum
the products in one order and give the same bits; where tile_rows selects the
kernel (all widths 64), the tensor cores' result is another one within FP32
rounding."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2310_08439_gb300 import inputs as I

pytestmark = pytest.mark.gpu

NETS = {   # species, K, hidden widths, activation, runs on the tensor cores by default
    "w36_20": (2, 8, [36, 20], "tanh", False),
    "w160": (1, 16, [160], "squareplus", False),
    "dd256_w60": (1, 64, [60], "tanh", False),
    "all64": (1, 16, [64, 64], "tanh", True),
    "all64_2sp": (2, 8, [64], "squareplus", True),
}


@pytest.mark.parametrize("n_cells", [(3, 3, 3), (5, 4, 4)])   # 108 and 320 atoms: ragged last tiles
@pytest.mark.parametrize("net", list(NETS))
def test_tiles_on_the_fp32_pipes(tmdlib, net, n_cells):
    import torch
    S, K, widths, act, split = NETS[net]
    rng = np.random.default_rng(K + n_cells[0])
    pos, box = I.lattice("fcc", n_cells, 3.8)
    pos = I.jitter_and_wrap(pos, box, 0.1, rng)
    types = rng.integers(0, S, len(pos)).astype(np.int32)
    pbc = np.ones(3, np.int32)
    make = lambda scale: I.random_model(S, K, 5.0, widths, seed=7, activation=act, feature_scale=scale)
    G = O.evaluate(O.OracleModel(make(None)), pos, types, box, pbc, want_G=True)["G"]
    p = make([np.sqrt((G[types == t] ** 2).mean(axis=0)) for t in range(S)])
    o = O.evaluate(O.OracleModel(p), pos, types, box, pbc)
    m = tmdlib.Model(p)
    nl = tmdlib.NeighborList()
    x, t = torch.as_tensor(pos, device="cuda"), torch.as_tensor(types, device="cuda")
    nl.build(x, t, box, pbc, p.rc)
    res = {}
    for rows in (0, 32, 64):
        m.tuning = {"tile_rows": rows, "pair_blocks_per_sm": 0}
        out = {k: v.double().cpu().numpy() for k, v in tmdlib.evaluate(m, nl, x, t, box).items()}
        rms = float(np.sqrt((o["forces"] ** 2).mean()))
        assert abs(out["energy"].item() - o["energy"]) <= 1e-6 * abs(o["energy"])
        assert np.abs(out["e_atom"] - o["e_atom"]).max() <= 1e-5 * np.abs(o["e_atom"]).max()
        assert np.abs(out["forces"] - o["forces"]).max() <= 1e-5 * rms
        assert np.abs(out["virial"].reshape(3, 3) - o["virial"]).max() <= 1e-5 * np.abs(o["virial"]).max()
        res[rows] = out
    assert np.array_equal(res[32]["forces"], res[64]["forces"])
    assert np.array_equal(res[32]["e_atom"], res[64]["e_atom"])
    assert np.array_equal(res[0]["forces"], res[32]["forces"]) != split


@pytest.mark.parametrize("n", [1, 127, 128, 129, 300])
@pytest.mark.parametrize("shape", ["dd96_w64x4", "dd192_w32_16", "dd512_2sp_w64"])
def test_tensor_core_tiles_of_few_atoms(tmdlib, shape, n):
    """The tensor-core kernel selected by tile_rows 128, at the edges of its tiles,
    species by species; the built-in choice beside it, within the same bars."""
    import torch

    import test_gpu_network_split as split
    S, K, _, _ = split.SHAPES[shape]
    s = split._system(n, S, seed=n + K)
    p, o = split._model(shape, s.pos, s.types, s.box, s.pbc)
    m = tmdlib.Model(p)
    nl = tmdlib.NeighborList()
    x, t = torch.as_tensor(s.pos, device="cuda"), torch.as_tensor(s.types, device="cuda")
    nl.build(x, t, s.box, s.pbc, p.rc)
    for rows in (128, 0):
        m.tuning = {"tile_rows": rows, "pair_blocks_per_sm": 0}
        out = {k: v.double().cpu().numpy() for k, v in tmdlib.evaluate(m, nl, x, t, s.box).items()}
        assert abs(out["energy"].item() - o["energy"]) <= 1e-6 * abs(o["energy"])
        assert np.abs(out["e_atom"] - o["e_atom"]).max() <= 1e-5 * np.abs(o["e_atom"]).max()
        rms = float(np.sqrt((o["forces"] ** 2).mean()))
        assert np.abs(out["forces"] - o["forces"]).max() <= 1e-5 * rms if rms else not out["forces"].any()
        assert np.abs(out["virial"].reshape(3, 3) - o["virial"]).max() <= 1e-5 * np.abs(o["virial"]).max()


@pytest.mark.parametrize("counts", [(1, 0, 5), (128, 129, 127), (0, 0, 256), (3, 260, 1)])
def test_tiles_begin_where_a_species_begins(tmdlib, counts):
    """Species of none, one, and around 128 atoms: more tiles than 32-atom ones in
    the smallest case (their energies have room of their own), tiles of a species
    that end short of 128, and the per-atom energies that add up to the total."""
    import torch
    rng = np.random.default_rng(sum(counts))
    n = sum(counts)
    reps = int(np.ceil((n / 4) ** (1 / 3)))
    pos, box = I.lattice("fcc", (reps, reps, reps), 3.8)
    pos = I.jitter_and_wrap(pos, box, 0.1, rng)[:n]
    types = rng.permutation(np.repeat(np.arange(3), counts)).astype(np.int32)
    p = I.random_model(3, 8, 4.5, [64, 32], seed=5)
    pbc = np.zeros(3, np.int32)
    o = O.evaluate(O.OracleModel(p), pos, types, box, pbc)
    nl = tmdlib.NeighborList()
    x, t = torch.as_tensor(pos, device="cuda"), torch.as_tensor(types, device="cuda")
    nl.build(x, t, box, pbc, p.rc)
    out = {k: v.double().cpu().numpy() for k, v in tmdlib.evaluate(tmdlib.Model(p), nl, x, t, box).items()}
    assert np.abs(out["e_atom"] - o["e_atom"]).max() <= 1e-5 * np.abs(o["e_atom"]).max()
    assert abs(out["energy"].item() - out["e_atom"].sum()) <= 1e-12 * abs(o["energy"])
    rms = float(np.sqrt((o["forces"] ** 2).mean()))
    assert np.abs(out["forces"] - o["forces"]).max() <= 1e-5 * rms
    assert np.abs(out["virial"].reshape(3, 3) - o["virial"]).max() <= 1e-5 * np.abs(o["virial"]).max()
