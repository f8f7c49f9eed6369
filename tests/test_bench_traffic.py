"""bench.py's DRAM traffic of one attend call is read from the committed profile
of the kernels the call runs; the profile has to carry the fields it reads."""
import hashlib
import os

import bench
from paper_2609_26425_gb300 import synth


def test_attend_traffic_reads_the_committed_profile(monkeypatch):
    with open(os.path.join(bench.ROOT, "profiles", "attend_dense_wan14b_layer.md")) as f:
        fields = dict(line.strip().split(": ", 1) for line in f if line.startswith(("workload: ", "traffic_", "source_")))
    assert fields["workload"] in synth.WORKLOADS and len(fields["source_sha256"]) == 64

    class Digest:   # the source as it was when the counters were taken
        def hexdigest(self):
            return fields["source_sha256"]

    monkeypatch.setattr(hashlib, "sha256", lambda data: Digest())
    assert bench.attend_traffic(fields["workload"]) == int(fields["traffic_bytes_per_launch"]) > 0
    assert bench.attend_traffic("another") is None
