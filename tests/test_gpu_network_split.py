"""The FP32 network on tensor cores with split operands (k_mlp_tf32: 128-atom
tiles, 32-wide weight chunks, the descriptor in groups of operand columns)
against the FP64 oracle at the plain FP32 bars, at the edges of its tiles and
of its range: one atom, a tile less one, full and plus one, three tiles with a
ragged end; one and several chunks and groups of the descriptor; widths 16 to
128 that do and do not fill a chunk; one to four hidden layers; tiles holding
several species; and more tiles than resident blocks."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2310_08439_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SHAPES = {   # species, K, hidden widths, activation -> descriptor columns 4 K S
    "dd32_w16": (1, 8, [16], "tanh"),
    "dd64_w48_32": (2, 8, [48, 32], "squareplus"),
    "dd96_w64x4": (3, 8, [64, 64, 64, 64], "tanh"),
    "dd128_w128_80_128": (1, 32, [128, 80, 128], "squareplus"),
    "dd192_w32_16": (3, 16, [32, 16], "tanh"),
    "dd512_w128_112": (1, 128, [128, 112], "squareplus"),
    "dd512_2sp_w64": (2, 64, [64], "tanh"),
}


def _system(n, n_species, seed):
    """n atoms of a jittered fcc lattice in an open box."""
    rng = np.random.default_rng(seed)
    reps = int(np.ceil((n / 4) ** (1 / 3)))
    pos, box = I.lattice("fcc", (reps, reps, reps), 3.8)
    pos = I.jitter_and_wrap(pos, box, 0.1, rng)[:n]
    return I.System(pos, rng.integers(0, n_species, n).astype(np.int32), box, np.zeros(3, np.int32))


def _model(shape, pos, types, box, pbc):
    """Random model, its first layer normalised by the descriptor RMS of this
    configuration (the way the workloads' models are built)."""
    S, K, widths, act = SHAPES[shape]
    p = I.random_model(S, K, 4.5, widths, seed=K + len(widths), activation=act)
    G = O.evaluate(O.OracleModel(p), pos, types, box, pbc, want_G=True)["G"]
    rms = np.repeat(np.sqrt((G ** 2).mean(axis=0)).reshape(1, -1), S, axis=0)
    p = I.random_model(S, K, 4.5, widths, seed=K + len(widths), activation=act, feature_scale=rms)
    return p, O.evaluate(O.OracleModel(p), pos, types, box, pbc)


def _check(tmd, p, s, o):
    import torch
    nl = tmd.NeighborList()
    pos = torch.as_tensor(s.pos, dtype=torch.float64, device="cuda")
    types = torch.as_tensor(s.types, dtype=torch.int32, device="cuda")
    nl.build(pos, types, s.box, s.pbc, p.rc)
    out = tmd.evaluate(tmd.Model(p), nl, pos, types, s.box)
    e, f = float(out["energy"].item()), out["forces"].double().cpu().numpy()
    ea = out["e_atom"].double().cpu().numpy()
    assert tmd.device_status() == 0
    assert abs(e - o["energy"]) <= 1e-6 * abs(o["energy"])
    assert np.abs(ea - o["e_atom"]).max() <= 1e-5 * np.abs(o["e_atom"]).max()
    rms = float(np.sqrt((o["forces"] ** 2).mean()))
    assert np.abs(f - o["forces"]).max() <= 1e-5 * rms if rms else not f.any()
    w = out["virial"].cpu().numpy().reshape(3, 3)
    assert np.abs(w - o["virial"]).max() <= 1e-5 * np.abs(o["virial"]).max()


@pytest.mark.parametrize("n", [1, 127, 128, 129, 300])
@pytest.mark.parametrize("shape", list(SHAPES))
def test_tile_and_chunk_edges(tmdlib, shape, n):
    S, K, _, _ = SHAPES[shape]
    s = _system(n, S, seed=n + K)
    p, o = _model(shape, s.pos, s.types, s.box, s.pbc)
    _check(tmdlib, p, s, o)


@pytest.mark.parametrize("shape", ["dd64_w48_32", "dd128_w128_80_128"])
def test_more_tiles_than_blocks(tmdlib, shape):
    """A jittered 108-atom cell 8 x 7 x 7 times over (42,336 atoms, 331 tiles):
    every copy has the cell's energies and forces."""
    S = SHAPES[shape][0]
    rng = np.random.default_rng(5)
    pos, box = I.lattice("fcc", (3, 3, 3), 3.8)
    pos = I.jitter_and_wrap(pos, box, 0.1, rng)
    types = rng.integers(0, S, len(pos)).astype(np.int32)
    p, one = _model(shape, pos, types, box, np.ones(3, np.int32))
    reps = (8, 7, 7)
    shift = np.stack(np.meshgrid(*[np.arange(r) for r in reps], indexing="ij"), -1).reshape(-1, 1, 3) * box
    m = len(shift)
    big = I.System((pos[None] + shift).reshape(-1, 3), np.tile(types, m), box * np.array(reps), np.ones(3, np.int32))
    _check(tmdlib, p, big, {"energy": one["energy"] * m, "e_atom": np.tile(one["e_atom"], m),
                            "forces": np.tile(one["forces"], (m, 1)), "virial": one["virial"] * m})
