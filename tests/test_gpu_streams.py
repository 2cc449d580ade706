"""Searches of one index at the same time, from threads with streams of their own
and from host and device arrays, in scratch pieces of the index's pool that it
keeps and pieces too large for it to keep: each the result of the same search alone."""
import threading
from dataclasses import replace

import numpy as np
import pytest

from paper_2102_02286_gb300 import configs, synth
from paper_2102_02286_gb300 import hicops as hc

pytestmark = pytest.mark.gpu


def test_searches_at_the_same_time():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    w = configs.OPEN_MEDIUM.with_proteins(150)
    w = replace(w, params=replace(w.params, top_n_peaks=1024, intensity_scale=8000))
    prot = synth.make_proteome(w.n_proteins, w.db_seed)
    idx = hc.Index(prot.seq, prot.off, w.mods, w.params)
    base = synth.make_spectra(prot, w, 300, seed=5)
    # the last one's scratch: 20,000 x 2 x 4 KB of query bins and more, above the 128 MB that a pool keeps
    parts = [base.subset((np.arange(n) * s) % base.n) for n, s in ((1, 1), (50, 7), (1100, 11), (20_000, 13))]
    assert idx.search_scratch_bytes(20_000) > 128 << 20
    want = [idx.search(p) for p in parts]
    errors = []

    def same(got, i):
        np.testing.assert_array_equal(got.psm, want[i].psm)
        np.testing.assert_array_equal(got.hist, want[i].hist)
        np.testing.assert_array_equal(got.n_scored, want[i].n_scored)

    def client(t):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                batches = [hc.DeviceBatch.from_spectra(p) for p in parts]
                outs = [hc.DeviceResult.alloc(p.n, w.params.top_k) for p in parts]
                for r in range(3):
                    order = [(i + t + r) % len(parts) for i in range(len(parts))]
                    for i in order:
                        outs[i].psm.zero_()
                        idx.search_device(batches[i], outs[i], stream)
                    stream.synchronize()
                    for i in order:
                        same(outs[i].to_host(parts[i].n, w.params.top_k), i)
                    same(idx.search(parts[order[0]]), order[0])
        except Exception as e:   # reported below
            errors.append(e)

    threads = [threading.Thread(target=client, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
