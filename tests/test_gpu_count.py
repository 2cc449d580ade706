"""Units counted peptide by peptide (min_shared 1 and 2, coarse grids) against the
oracle: the queue of qualifying peptides and its overflow, columns cut by the
window and by pieces of a given size, more peaks than threads, and batches of
which some spectra are counted and others are not."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2102_02286_gb300 import configs, synth
from paper_2102_02286_gb300 import hicops as hc

from parity import assert_parity

pytestmark = pytest.mark.gpu

# proteins, parameters, kernels a search launches
CASES = {
    "one": (80, dict(min_shared=1), 4),
    "one_many_peaks": (80, dict(min_shared=1, top_n_peaks=700, top_k=32), 4),
    "two": (120, dict(min_shared=2), 5),
    "two_tolerance": (80, dict(min_shared=2, tol_bins=2, bin_width_da=0.02), 6),
    "coarse": (80, dict(min_shared=4, bin_width_da=0.5), 5),
    "coarse_six": (80, dict(min_shared=6, bin_width_da=1.0005, top_k=32), 5),
    "fine": (80, dict(min_shared=3), 4),
}


@pytest.mark.parametrize("name", CASES)
def test_counted_units(oracle_lib, name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    proteins, params, launches = CASES[name]
    w = configs.OPEN_MEDIUM.with_proteins(proteins)
    w = replace(w, params=replace(w.params, **params))
    prot = synth.make_proteome(w.n_proteins, w.seed)
    parts = []
    for peaks, tol, n in ((3, 6000.0, 2), (40, 500.0, 3), (100, 6000.0, 3), (100, 3.0, 4), (100, 0.01, 3), (600, 300.0, 3)):
        parts.append(synth.make_spectra(prot, replace(w, spectra=replace(w.spectra, target_peaks=(peaks, peaks),
                                                                         tol_da=(tol,))), n, seed=peaks + int(tol)))
    off = np.cumsum([0] + [int(p.peak_off[-1]) for p in parts])
    cat = lambda f: np.concatenate([getattr(p, f) for p in parts])   # noqa: E731
    spec = replace(parts[0], peak_off=np.concatenate([p.peak_off[:-1].astype(np.uint64) + np.uint64(o) for p, o in
                                                      zip(parts, off)] + [off[-1:].astype(np.uint64)]),
                   **{f: cat(f) for f in ("mz", "intensity", "prec_mz", "charge", "tol_da")})
    ref = oracle_lib.OracleDb(prot.seq, prot.off, w.mods, w.params).search(spec)
    idx = hc.Index(prot.seq, prot.off, w.mods, w.params)
    for seg in (0, 1 << 14, 12_345, 0x7fffffff):
        idx.set_config(hc.SearchConfig(0, 0, 0, seg))
        before = hc.kernel_launches()
        got = idx.search(spec)
        assert hc.kernel_launches() - before == launches
        assert_parity(got, ref, label=f"{name}, pieces of {seg}")
    assert int(ref.n_scored.sum()) > 0
    # the same launches captured and replayed, one after another on a stream
    idx.set_config(None)
    plan, stream = idx.plan(spec.n), torch.cuda.Stream()
    batch, out = hc.DeviceBatch.from_spectra(spec), hc.DeviceResult.alloc(spec.n, w.params.top_k)
    torch.cuda.synchronize()
    for graph in (False, True, True, True):
        out.psm.zero_()
        out.hist.zero_()
        torch.cuda.synchronize()
        for _ in range(3):
            plan.search(batch, out, stream, graph=graph)
        torch.cuda.synchronize()
        assert_parity(out.to_host(spec.n, w.params.top_k), ref, label=f"{name}, plan, graph {graph}")
    plan.close()
