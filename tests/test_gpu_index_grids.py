"""The index of grids where the fixed-point ion bins are certain, where every
ion lies on a bin edge (the FP64 form decides), where the FP64 form serves alone,
and lists too long for shared memory: the CSR against the oracle's ion bins, and a
search (forward lists, bitmaps, score table) against the oracle's."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2102_02286_gb300 import configs, synth
from paper_2102_02286_gb300 import hicops as hc
from paper_2102_02286_gb300.configs import Mod

from parity import assert_parity

pytestmark = pytest.mark.gpu

PROTON = 1.007276466812
MASS = dict(A=71.037114, R=156.101111, N=114.042927, D=115.026943, C=103.009185, E=129.042593, Q=128.058578,
            G=57.021464, H=137.058912, I=113.084064, L=113.084064, K=128.094963, M=131.040485, F=147.068414,
            P=97.052764, S=87.032028, T=101.047679, W=186.079313, Y=163.063329, V=99.068414)
# fixed modifications that make every residue a whole number of protons: b ions on bin edges
ON_EDGES = tuple(Mod(c, round(m / PROTON) * PROTON - m, 0, True) for c, m in MASS.items())

# modification rules, parameters
CASES = {
    "fine": ((configs.OX_M(2),), dict(bin_width_da=0.0007)),
    "coarse": ((configs.OX_M(2),), dict(bin_width_da=37.0, frag_mz_min=300.0)),
    "edges": (ON_EDGES, dict(bin_width_da=PROTON)),
    "narrow_range": ((configs.OX_M(1),), dict(frag_mz_min=400.0, frag_mz_max=410.0)),
    "long": ((configs.OX_M(1),), dict(min_len=40, max_len=64, max_mass=9000.0, frag_mz_max=9000.0,
                                      intensity_scale=1000)),
    "not_positive": ((Mod("M", -131.040485, 1), Mod("S", -95.0, 1)), dict()),
}


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("name", CASES)
def test_index_of_grid(gpu, oracle_lib, name):
    mods, params = CASES[name]
    w = replace(configs.OPEN_MEDIUM, mods=mods).with_proteins(40).with_spectra(40)
    w = replace(w, params=replace(w.params, missed_cleavages=4, **params))
    prot = synth.make_proteome(w.n_proteins, w.db_seed)
    idx = hc.Index(prot.seq, prot.off, w.mods, w.params)
    db = oracle_lib.OracleDb(prot.seq, prot.off, w.mods, w.params)
    off, ent = idx.copy_csr()
    assert idx.stats().n_peptides == db.n and off[-1] == len(ent) > 0
    bins = np.repeat(np.arange(len(off) - 1), np.diff(off.astype(np.int64)))
    order = np.lexsort((bins, ent >> 1))
    got = np.stack([(ent >> 1)[order], bins[order], (ent & 1)[order]], 1)
    want = []
    for p in range(db.n):
        b, t = db.bins(p)
        want.append(np.stack([np.full(len(b), p), b, t], 1))
    np.testing.assert_array_equal(got, np.concatenate(want))
    spec = synth.make_spectra(prot, w)
    assert_parity(idx.search(spec), db.search(spec), label=name)
