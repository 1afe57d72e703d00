"""The committed ncu summaries that carry counters into the benchmark lines name the kernel headers
as they stand: part of the profiled kernels' code lies in them."""
import hashlib
import os

import lbw_workloads as W


def test_committed_profiles_match_the_kernel_headers():
    import bench
    csrc = os.path.join(bench.ROOT, "paper_1705_01801_gb300", "csrc")
    text = b"".join(open(os.path.join(csrc, n), "rb").read() for n in ("lbw_march.cuh", "lbw_tma.cuh"))
    headers = hashlib.sha256(text).hexdigest()[:16]
    for path in (bench.PROFILES[("torus", W.PREC_F32)], bench.PROFILES[("cylinder", W.PREC_F32)], bench.ENSEMBLE_PROFILE):
        assert bench._profile_fields(path)["headers_sha256_16"] == headers, path
