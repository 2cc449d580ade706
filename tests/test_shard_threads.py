"""Parts of a database on a host that gives no more threads (an address-space limit
below their stacks): the call does the work itself, and gives the same part."""
import os
import resource
import subprocess
import sys

ROOT = os.path.abspath(os.path.join(os.path.dirname(__file__), ".."))

CHILD = """
import resource, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
from paper_2102_02286_gb300 import configs, synth
from paper_2102_02286_gb300 import hicops as hc
w = configs.OPEN_MEDIUM.with_proteins(400)
prot = synth.make_proteome(w.n_proteins, w.db_seed, w.protein_len)
full = hc.Index(prot.seq, prot.off, w.mods, w.params, upload=False)
P = full.n_peptides
assert P > 1 << 17                       # from there on threads take a part's entries
want = [full.peptide(p) for p in range(0, P, 997)]
pids = np.arange(P, dtype=np.uint32)
now = 4096 * int(open("/proc/self/statm").read().split()[0])
resource.setrlimit(resource.RLIMIT_AS, (now + (40 << 20), resource.RLIM_INFINITY))
for part in (full.shard(1, 0, upload=False), full.subset(pids, upload=False)):
    assert part.n_peptides == P
    assert [part.peptide(p) for p in range(0, P, 997)] == want
print("ok")
"""


def test_parts_without_more_threads():
    from paper_2102_02286_gb300 import build as pkg_build
    pkg_build.build()

    def stacks():                            # of 128 MB, which no cache of ended threads keeps
        hard = resource.getrlimit(resource.RLIMIT_STACK)[1]
        soft = 128 << 20 if hard == resource.RLIM_INFINITY else min(128 << 20, hard)
        resource.setrlimit(resource.RLIMIT_STACK, (soft, hard))

    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=300, preexec_fn=stacks)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr[-2000:])
    assert r.stdout.strip() == "ok"
