"""The ways a super-chunk can go, each against the oracle: folded planes and the
second plane (windows of several planes), the scan of the plane with the hot
bitmaps, a full repeat table (halving, then one counter a peptide), a full
queue of peptides to score, and the shared-memory layouts of the largest
query-bin counts and top-k lists."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2102_02286_gb300 import configs, synth
from paper_2102_02286_gb300 import hicops as hc

from parity import assert_parity

pytestmark = pytest.mark.gpu

# proteins, peaks, tolerance (Da), spectra, parameters
CASES = {
    # 1.3 M peptides in one window: several planes of either CTA shape
    "deep": (2000, 100, 6000.0, 3, dict()),
    "deep_two_hits_left": (2000, 400, 6000.0, 3, dict(top_n_peaks=400, min_shared=5, top_k=16)),
    # every repeat (and with 1, every hit) is scored: the queue runs full
    "every_hit": (60, 100, 6000.0, 4, dict(min_shared=1)),
    "every_repeat": (600, 100, 6000.0, 4, dict(min_shared=2)),
    "three": (600, 150, 6000.0, 4, dict(top_n_peaks=150, min_shared=3, top_k=32)),
    "seven": (300, 100, 6000.0, 4, dict(min_shared=7)),
    # nearly every peptide of a column is hit: the repeat table never holds a column's
    "dense_bins": (300, 1000, 6000.0, 3, dict(top_n_peaks=1000, bin_width_da=0.1, min_shared=4, top_k=32,
                                              intensity_scale=1000)),
    "dense_bins_many_slices": (300, 1000, 300.0, 3, dict(top_n_peaks=1024, bin_width_da=0.5, min_shared=6,
                                                         intensity_scale=1000)),
}


@pytest.mark.parametrize("threads", [0, 256, 384, 512])
@pytest.mark.parametrize("name", CASES)
def test_search_paths(oracle_lib, name, threads):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    proteins, peaks, tol, n, params = CASES[name]
    w = configs.OPEN_MEDIUM.with_proteins(proteins)
    w = replace(w, params=replace(w.params, **params),
                spectra=replace(w.spectra, n_spectra=n, target_peaks=(peaks, peaks), tol_da=(tol,)))
    key = (name,)
    if key not in _REF:
        _REF.clear()
        prot = synth.make_proteome(w.n_proteins, w.seed)
        spec = synth.make_spectra(prot, w)
        db = oracle_lib.OracleDb(prot.seq, prot.off, w.mods, w.params)
        _REF[key] = (hc.Index(prot.seq, prot.off, w.mods, w.params), spec, db.search(spec))
    idx, spec, ref = _REF[key]
    # one unit a spectrum where the shape is given, so that a window's super-chunks follow one another
    idx.set_config(hc.SearchConfig(threads, 0, 0, 0x7fffffff if threads else 0))
    assert_parity(idx.search(spec), ref, label=f"{name}, {threads} threads")
    assert int(ref.n_scored.sum()) > 0


_REF = {}
