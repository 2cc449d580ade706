"""Planning of batches at the sizes where its forms meet (a warp's spectra, the
small and the large block, one step and several), with spectra of common fragments
that are split and empty ones between: the rows, histograms and counts of the same
spectra searched a few at a time with pieces of a given size."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2102_02286_gb300 import configs, synth
from paper_2102_02286_gb300 import hicops as hc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    out = {}
    for tol_bins in (0, 1):
        w = configs.OPEN_MEDIUM.with_proteins(400).with_spectra(300)
        w = replace(w, params=replace(w.params, tol_bins=tol_bins))
        prot = synth.make_proteome(w.n_proteins, w.db_seed)
        spec = synth.make_spectra(prot, w)
        z = spec.charge.copy()
        z[5::17] = 0                       # invalid: no units
        t = spec.tol_da.copy()
        t[3::7] = 1e6                      # the whole database
        t[4::7] = 0.0
        spec = replace(spec, charge=z, tol_da=t)
        idx = hc.Index(prot.seq, prot.off, w.mods, w.params)
        idx.set_config(hc.SearchConfig(0, 0, 0, 1 << 15))
        ref = [idx.search(spec.subset(range(a, a + 50))) for a in range(0, spec.n, 50)]
        idx.set_config(None)
        out[tol_bins] = idx, spec, [np.concatenate([getattr(r, f) for r in ref]) for f in ("psm", "hist", "n_scored")]
    return out


@pytest.mark.parametrize("tol_bins", [0, 1])
@pytest.mark.parametrize("n", [1, 4, 33, 127, 128, 129, 512, 513, 4096, 4097, 9001])
def test_plan_sizes(setup, tol_bins, n):
    idx, spec, (psm, hist, ns) = setup[tol_bins]
    pick = (np.arange(n) * 7) % spec.n
    got = idx.search(spec.subset(pick))
    want = psm[pick].copy()
    want["query"] = np.arange(n)[:, None]
    np.testing.assert_array_equal(got.psm, want)
    np.testing.assert_array_equal(got.hist, hist[pick])
    np.testing.assert_array_equal(got.n_scored, ns[pick])
