"""Systematic parts of the errors of the split tensor-core sums, against FP64:
what all atoms have in common does not average out in the virial, however
small it is in one atom.

Descriptors: H is read from a table (no special function in it) and G compared
with the oracle's.  FP32 sums that round as they go are off by a few units in
the last place in each atom and by nothing on average: the mean relative error
of a rank over all atoms and channels that are not nearly empty stays below
half a unit in the last place of G_0 (2^-25), twice that for G_1 .. G_3, which
are squares."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2310_08439_gb300 import inputs as I

pytestmark = pytest.mark.gpu
RC = 5.0


def _system(n_species, seed, reps=(6, 6, 6), a=3.7, lattice="fcc"):
    rng = np.random.default_rng(seed)
    pos, box = I.lattice(lattice, reps, a)
    types = rng.integers(0, n_species, len(pos)).astype(np.int32)
    return I.System(I.jitter_and_wrap(pos, box, 0.1, rng), types, box, np.ones(3, np.int32))


def _descriptors(tmd, m, s):
    import torch
    pos = torch.as_tensor(s.pos, dtype=torch.float64, device="cuda")
    types = torch.as_tensor(s.types, dtype=torch.int32, device="cuda")
    nl = tmd.NeighborList()
    nl.build(pos, types, s.box, s.pbc, RC)
    G, dG = tmd.descriptors(m, nl, pos, types, s.box, with_grad=True)
    return G.double().cpu().numpy(), dG.double().cpu().numpy()


CASES = [(1, 16, "fcc"), (1, 32, "bcc"), (2, 16, "fcc"), (3, 8, "bcc")]


def _mean_errors(tmd, S, K, lattice):
    s = _system(S, 10 * S + K, *(((6, 6, 6), 3.7) if lattice == "fcc" else ((8, 8, 8), 2.95)), lattice)
    p = I.random_model(S, K, RC, [16], seed=1)
    m = tmd.Model(p)
    m.set_radial_table(256)
    o = O.evaluate(O.OracleModel(p, radial_table=256), s.pos, s.types, s.box, s.pbc, want_G=True)["G"]
    G = _descriptors(tmd, m, s)[0]
    G, o = G.reshape(len(G), S * K, 4), o.reshape(len(G), S * K, 4)
    rms = np.sqrt((o ** 2).mean(axis=0))
    mean = []
    for rank in range(4):
        big = o[:, :, rank] > 0.1 * rms[None, :, rank].max()
        mean.append(float(((G[:, :, rank] - o[:, :, rank])[big] / o[:, :, rank][big]).mean()))
    return np.array(mean)


@pytest.mark.parametrize("S,K,lattice", CASES)
def test_descriptor_sums_have_no_common_error(tmdlib, S, K, lattice, capsys):
    mean = _mean_errors(tmdlib, S, K, lattice)
    with capsys.disabled():
        print(f"\n[S={S} K={K} {lattice}] mean relative error of G_0 .. G_3: " + " ".join(f"{x:.2e}" for x in mean))
    assert abs(mean[0]) <= 2.0 ** -25
    assert np.abs(mean[1:]).max() <= 2.0 ** -24


def test_constants_of_the_ranks(tmdlib):
    """1/3 and 3/5, with which the lower degrees enter G_2 and G_3, are off by
    3e-8 and 4e-8 as FP32 numbers.  Over the four cases the mean error stays
    below a quarter of a unit in the last place, half of either."""
    mean = np.mean([_mean_errors(tmdlib, *c) for c in CASES], axis=0)
    assert np.abs(mean[2:]).max() <= 2.0 ** -26


def _gradient64(p, G, types):
    """dE_a/dG_a of the network at these descriptors, in FP64."""
    dG = np.zeros_like(G)
    for t in range(p.n_species):
        layers = p.unpack(t)
        rows = types == t
        a, d = G[rows], []
        for W, b in layers[:-1]:
            z = a @ W.T + b
            if p.activation == "tanh":
                a = np.tanh(z)
                d.append(1.0 - a * a)
            else:
                q = np.sqrt(z * z + p.squareplus_b)
                a = 0.5 * (z + q)
                d.append(a / q)
        g = np.repeat(layers[-1][0], rows.sum(), axis=0)
        for (W, _), da in zip(layers[:-1][::-1], d[::-1]):
            g = (g * da) @ W
        dG[rows] = g
    return dG


@pytest.mark.parametrize("floor", [0.1, 1e-4])   # 1e-4: columns of very different weights
@pytest.mark.parametrize("S,K,widths,act", [(1, 16, [64], "tanh"), (1, 16, [64, 64], "tanh"),
                                            (2, 8, [64, 64], "squareplus"), (3, 16, [128, 128], "tanh"),
                                            (1, 32, [128, 128, 128], "squareplus"), (1, 8, [16, 48], "tanh"),
                                            # 160 (in 5 passes of G'), 256, 320 and 640 columns
                                            (5, 8, [64, 64], "tanh"), (1, 64, [128, 128], "squareplus"),
                                            (5, 16, [112], "tanh"), (5, 32, [64, 32], "tanh")])
def test_network_sums_are_as_exact_as_their_rounding(tmdlib, S, K, widths, act, floor, capsys):
    """dE/dG of the network against FP64 at the descriptors that it was given.
    A hidden layer rounds about 12 numbers one after the other (the sums and the
    bias, the activation and its derivative, the way back); each is off by at most
    half a unit, 2^-24 / sqrt(12) rms, and what is off early goes through the rest
    twice: 2 sqrt(12 L) 2^-24 / sqrt(12) = 2^-23 sqrt(L) for L layers.  The products
    themselves must add nothing to that."""
    s = _system(S, 3 * S + K)
    def model(scale):
        return I.random_model(S, K, RC, widths, seed=K + len(widths), activation=act, feature_scale=scale, scale_floor=floor)
    G0 = O.evaluate(O.OracleModel(model(None)), s.pos, s.types, s.box, s.pbc, want_G=True)["G"]
    p = model([np.sqrt((G0[s.types == t] ** 2).mean(axis=0)) for t in range(S)])
    m = tmdlib.Model(p)
    m.tuning = {"tile_rows": 128, "pair_blocks_per_sm": 0}   # on the tensor cores
    G, dG = _descriptors(tmdlib, m, s)
    ref = _gradient64(p, G, s.types)
    err = float(np.linalg.norm(dG - ref) / np.linalg.norm(ref))
    with capsys.disabled():
        print(f"\n[S={S} K={K} {widths} {act} floor {floor}] dE/dG error {err:.2e}")
    assert err <= 2.0 ** -23 * np.sqrt(len(widths))
