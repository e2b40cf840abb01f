"""The committed DRAM-traffic records: there is one for the dominant kernel of every
workload that the default bench line reports a bandwidth for, taken from device
code that has not changed since, and the bench attaches it."""
import json
import os

import pytest

import bench
from paper_1602_02306_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("kernel,workload", [
    ("csr_gather_kernel", "powerlaw_2M_jacobi_m128_k50"),
    ("reorth_dots_kernel", "powerlaw_2M_jacobi_m128_k50"),
    ("reorth_update_kernel", "powerlaw_2M_jacobi_m128_k50"),
    ("stencil_pair_kernel", "fd_hamiltonian_64^3_7pt_cheb8_m64_k30"),
    ("stencil_patch_kernel", "slicing_96^3_13pt_cheb8_S32_m64_tol0.25"),
])
def test_record_exists_and_is_attached(kernel, workload):
    rec = os.path.join(ROOT, "profiles", f"{kernel}_{workload}_traffic.json")
    with open(rec) as f:
        d = json.load(f)
    assert d["kernel"] == kernel and os.path.exists(os.path.join(ROOT, d["profile"]))
    assert bench._device_code_sha(d["device_code"]) == d["device_code_sha256"]
    assert 0.3 < d["dram_bytes"] / d["algorithmic_bytes"] < 1.5

    class _W:
        name = workload
    roof = {"kernel": kernel, "bytes_per_launch_avg": 1e9}
    bench._attach_traffic(roof, _W)
    assert roof["traffic"] == pytest.approx(1e9 * d["dram_bytes"] / d["algorithmic_bytes"])


def test_the_workloads_of_the_records_are_the_bench_s():
    src = open(W.__file__).read()
    for name in ("powerlaw_2M_jacobi_m128_k50", "fd_hamiltonian_64^3_7pt_cheb8_m64_k30",
                 "slicing_96^3_13pt_cheb8_S32_m64_tol0.25"):
        assert name in src
