"""Query preprocessing at the sizes where its forms meet (a warp's rounds, the
largest spectrum of a warp, the chunks of a block) and on peak lists that take its
turns: out of order, many peaks a bin, equal intensities at the cut, unusable
peaks, intensities from the smallest to the largest float.  Each against the
oracle's windows, retained counts and search."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2102_02286_gb300 import configs, synth
from paper_2102_02286_gb300 import hicops as hc

from parity import assert_parity

pytestmark = pytest.mark.gpu

COUNTS = (1, 31, 32, 33, 100, 257, 511, 512, 513, 1500, 4097, 9000)


def kinds(rng, mz, it):
    """The same peaks in the ways a list can come."""
    yield "ascending", mz, it
    p = rng.permutation(len(mz))
    yield "shuffled", mz[p], it[p]
    yield "crowded", np.sort(np.float32(100.0) + np.float32(0.004) * rng.integers(0, 200, len(mz)).astype(np.float32)), it
    yield "ties", mz, np.float32(1.0) + rng.integers(0, 3, len(mz)).astype(np.float32)
    bad_mz, bad_it = mz.copy(), it.copy()
    hit = rng.integers(0, 5, len(mz))
    bad_it[hit == 0] = 0.0
    bad_it[hit == 1] = np.inf
    bad_mz[hit == 2] = np.nan
    bad_mz[(hit == 3) & (rng.random(len(mz)) < 0.5)] = 99.0
    yield "unusable", bad_mz, bad_it
    yield "wide", mz, (10.0 ** rng.uniform(-45, 38, len(mz))).astype(np.float32)


@pytest.mark.parametrize("topn", [1, 100, 1024])
def test_prep_forms(oracle_lib, topn):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    w = configs.OPEN_MEDIUM.with_proteins(60)
    w = replace(w, params=replace(w.params, top_n_peaks=topn, min_shared=1 if topn == 1 else 3, intensity_scale=8000))
    prot = synth.make_proteome(w.n_proteins, w.db_seed)
    rng = np.random.default_rng(7)
    mzs, its, prec, z, tol = [], [], [], [], []
    for n in COUNTS:
        s = synth.make_spectra(prot, replace(w, spectra=replace(w.spectra, n_spectra=1, target_peaks=(n, n))))
        mz, it = np.array(s.mz[:n]), np.array(s.intensity[:n])
        o = np.argsort(mz, kind="stable")
        for _, m, i in kinds(rng, mz[o], it[o]):
            mzs.append(m); its.append(i)
            prec.append(s.prec_mz[0]); z.append(s.charge[0]); tol.append(rng.choice([0.0, 10.0, 500.0, 1e9]))
    n = len(mzs)
    spec = synth.Spectra(np.concatenate([[0], np.cumsum([len(m) for m in mzs])]).astype(np.uint64),
                         np.concatenate(mzs), np.concatenate(its), np.array(prec), np.array(z, np.uint8),
                         np.array(tol), *([np.zeros(n, np.uint64)] * 4))
    idx = hc.Index(prot.seq, prot.off, w.mods, w.params)
    ref = oracle_lib.OracleDb(prot.seq, prot.off, w.mods, w.params).search(spec)
    lo, hi, npk, _ = idx.search_work(spec)
    np.testing.assert_array_equal(lo, ref.lo)
    np.testing.assert_array_equal(hi, ref.hi)
    for q in range(n):
        bins = oracle_lib.preprocess(w.params, mzs[q], its[q], prec[q], int(z[q]), float(tol[q]))[0]
        assert npk[q] == len(bins)
    assert_parity(idx.search(spec), ref, label=f"top {topn}")
    assert int(ref.n_scored.sum()) > 0
