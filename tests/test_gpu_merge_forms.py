"""The merge of parts where its forms meet: one list to 64 (a lane's second list),
lists that end early, k up to 32, spectra that fill the last block in part,
histograms at any 4-byte address, results written over an input; and sampling of
counts that need 64-bit keys.  Against a sort on the host and the oracle's fit."""
import numpy as np
import pytest

from paper_2102_02286_gb300 import hicops as hc

from parity import EV_RTOL

pytestmark = pytest.mark.gpu

NONE = 0xFFFFFFFF


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def parts_of(rng, P, n, k):
    """P parts' sorted rows: some lists short or empty, keys that tie across parts."""
    rows = np.zeros((P, n, k), hc.PSM_DTYPE)
    rows["pid"], rows["key"], rows["evalue"] = NONE, np.iinfo(np.int64).min, np.inf
    for p in range(P):
        for q in range(n):
            m = int(rng.integers(0, k + 1)) if (p + q) % 3 else k
            if q % 7 == 3:
                m = 0
            key = rng.integers(0, 40, m) * (1 << 32) + rng.integers(0, 2, m)
            pid = rng.choice(1000, m, replace=False) * P + p
            o = np.lexsort((pid, -key))
            rows["key"][p, q, :m], rows["pid"][p, q, :m] = key[o], pid[o]
            rows["nb"][p, q, :m], rows["ny"][p, q, :m] = rng.integers(0, 60, m), rng.integers(0, 60, m)
    return rows


@pytest.mark.parametrize("P,n,k,mode", [(1, 9, 5, 2), (3, 1, 1, 0), (33, 16, 7, 3), (64, 21, 32, 2), (8, 50, 10, 1)])
def test_merge_of_parts(gpu, oracle_lib, P, n, k, mode):
    torch = gpu
    rng = np.random.default_rng(P)
    rows = parts_of(rng, P, n, k)
    hist = np.zeros((P, n, 256), np.uint32)
    for q in range(n):
        x = rng.gumbel(rng.uniform(5, 60), rng.uniform(0.5, 9), size=(P, 300))
        for p in range(P):
            np.add.at(hist[p, q], np.clip(x[p].astype(int), 0, 255), 1)
    ns = hist.sum(2, dtype=np.uint32)
    total = hist.sum(0, dtype=np.uint32)

    def check(psm, h, c):
        np.testing.assert_array_equal(h, total)
        np.testing.assert_array_equal(c, ns.sum(0))
        for q in range(n):
            f = rows[:, q].reshape(-1)
            f = f[f["pid"] != NONE]
            f = f[np.lexsort((f["pid"], -f["key"]))][:k]
            got = psm[q][: len(f)]
            for name in ("pid", "key", "nb", "ny"):
                np.testing.assert_array_equal(got[name], f[name])
            assert np.all(psm[q]["pid"][len(f):] == NONE)
            np.testing.assert_array_equal(psm[q]["query"], q)
            if len(f):
                ev = oracle_lib.evalue(total[q], psm[q]["key"], psm[q]["pid"], mode)
                np.testing.assert_allclose(got["evalue"], ev[: len(f)], rtol=EV_RTOL, atol=0)

    def dev(a, words=0):
        """On the device, `words` 4-byte words past an aligned address."""
        b = torch.zeros(a.nbytes // 4 + words, dtype=torch.int32, device="cuda")
        b[words:] = torch.from_numpy(a.reshape(-1).view(np.int32))
        return b[words:]

    lib = hc.load()
    s = torch.cuda.current_stream().cuda_stream
    for h_in, c_in, words in ((hist, ns, 0), (total, total.sum(1, dtype=np.uint32), 1), (hist, ns, 3)):
        d_rows, d_h, d_c = dev(rows), dev(h_in, words), dev(c_in)
        for over in (False, True):       # the merged rows over the first part's, the last time
            out = d_rows if over else torch.zeros(n * k * 8, dtype=torch.int32, device="cuda")
            o_h, o_c = dev(np.zeros_like(total), words), dev(np.zeros(n, np.uint32))
            assert lib.hicops_merge_shards(P, n, k, d_rows.data_ptr(), d_h.data_ptr(), d_c.data_ptr(),
                                           len(h_in) if h_in is hist else 1, mode, 1, s, out.data_ptr(),
                                           o_h.data_ptr(), o_c.data_ptr()) == 0
            torch.cuda.synchronize()
            check(out[: n * k * 8].cpu().numpy().view(hc.PSM_DTYPE).reshape(n, k),
                  o_h.cpu().numpy().view(np.uint32).reshape(n, 256), o_c.cpu().numpy().view(np.uint32))


@pytest.mark.parametrize("words", [0, 1])
@pytest.mark.parametrize("top", [(1 << 24) - 1, 1 << 24, (1 << 32) - 1])
def test_sampling_of_large_counts(gpu, oracle_lib, top, words):
    torch = gpu
    rng = np.random.default_rng(3)
    h = rng.integers(0, 4, (40, 256)).astype(np.uint32)
    for q in range(40):
        h[q, rng.choice(256, 4, replace=False)] = [top, top, top - q % 3, top - 1]
    d = torch.zeros(h.size + words, dtype=torch.int32, device="cuda")
    d[words:] = torch.from_numpy(h.reshape(-1).view(np.int32))
    for s in (1, 9, 120):
        got = hc.hist_sample(d[words:], s).cpu().numpy().view(np.uint32).reshape(-1, s + 1)
        for q in range(40):
            lo, ln, _ = oracle_lib.hist_sample(h[q], s)
            assert got[q, 0] == lo | ln << 16
            np.testing.assert_array_equal(got[q, 1:1 + ln], h[q, lo:lo + ln])
            assert not got[q, 1 + ln:].any()
