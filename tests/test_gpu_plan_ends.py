"""A plan made for exactly its batch, at numbers of spectra that leave the last
16-byte vector of the windows and costs ragged, over one step of the planning
block and several: the rows, histograms and counts of hicops_search."""
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
    w = configs.OPEN_MEDIUM.with_proteins(200).with_spectra(400)
    prot = synth.make_proteome(w.n_proteins, w.db_seed)
    return torch, w, hc.Index(prot.seq, prot.off, w.mods, w.params), synth.make_spectra(prot, w)


@pytest.mark.parametrize("n", [1, 2, 3, 5, 126, 131, 4095, 4098, 12_345])
def test_plan_of_its_batch(setup, n):
    torch, w, idx, spec = setup
    sub = spec.subset(np.arange(n) % spec.n)
    want = idx.search(sub)
    batch = hc.DeviceBatch.from_spectra(sub)
    out = hc.DeviceResult.alloc(n, w.params.top_k)
    plan = idx.plan(n)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for graph in (False, True, True):
        out.psm.zero_()
        out.hist.zero_()
        out.n_scored.zero_()
        torch.cuda.synchronize()
        plan.search(batch, out, stream, graph=graph)
        torch.cuda.synchronize()
        got = out.to_host(n, w.params.top_k)
        np.testing.assert_array_equal(got.psm, want.psm)
        np.testing.assert_array_equal(got.hist, want.hist)
        np.testing.assert_array_equal(got.n_scored, want.n_scored)
    plan.close()
