"""Register spills of every unit that holds a hot kernel, from ptxas's resource
report on a CPU-only cross-compile for sm_103a: no kernel may spill, except those
listed with the bytes of spill stores they had when measured.  An entry that
matches no kernel fails, so that a kernel that moves to another file or changes
its name does not drop out of the test.  Skipped without nvcc.
"""
import concurrent.futures
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1805_07801_gb300", "csrc")

# unit -> {mangled-name fragment: largest spill-store bytes allowed}
KNOWN = {
    "closure.cu": {},
    "fft_pruned.cu": {},
    "fft_radix3.cu": {},
    "fft_sc.cu": {"k_scpassILi2048ELb": 32, "k_scpassILi4096ELb": 24},  # 1024 threads at 64 registers
    "fft_stream.cu": {
        "k_cpass_pipeILi1024ELin1ELb0ELi1E": 96,  # two radix-32 stages and the mirror exchange, 128 registers
        "k_cpass_pipeILi1024ELin1ELb1ELi1E": 96,
        "k_cpass_pipeILi1024ELin1ELb0ELi2E": 96,
        "k_cpass_pipeILi1024ELin1ELb1ELi2E": 96,
        "k_cpass_pipeILi1024ELi1ELb": 4,
        "k_cpass_pipeILi512E": 8,
        "k_cpass_pipeILi256E": 8,
    },
    "fft_tc.cu": {},
    "mlp_train.cu": {},
    "ns_diag.cu": {},
    "ns_fwdx.cu": {},
    "ns_fwdx3.cu": {},
    "ns_radix3.cu": {"k_ns_zILi192E": 60, "k_ns_zILi384E": 40, "k_ns_zILi768E": 64, "k_ns_invxILi384E": 8},
    "ns_shell.cu": {
        "k_shell_invxILi256E": 112,
        "k_shell_invxILi512E": 128,
        "k_shell_invxILi1024E": 128,
        "k_shell_invyILi1024E": 4,
        "k_shell_zILi128E": 8,
        "k_shell_zILi256E": 4,
        "k_shell_zILi1024E": 20,
    },
    "ns_ypass.cu": {},
    "rbc.cu": {},
    "rbc_pow2.cu": {"k_ns_invxILi512ELb1E": 12, "k_ns_invxILi1024ELb1E": 188},  # two fields of 16 values at 128
    "rbc_radix3.cu": {"k_rbc_fwdxILi192E": 28, "k_ns_invxILi384ELb1E": 52, "k_ns_invxILi768ELb1E": 48},
}


def _spills(nvcc, src, out):
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", f"-I{CSRC}",
           f"-I{os.path.join(ROOT, 'include')}", "-Xptxas", "-v", "-c", os.path.join(CSRC, src), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    res, name = {}, None
    for line in r.stderr.splitlines():
        m = re.search(r"Function properties for (\S+)", line)
        if m:
            name = m.group(1)
            continue
        m = re.search(r"(\d+) bytes spill stores", line)
        if m and name:
            res[name] = int(m.group(1))
            name = None
    return res


@pytest.fixture(scope="module")
def spills(tmp_path_factory):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    tmp = tmp_path_factory.mktemp("res")
    with concurrent.futures.ThreadPoolExecutor(os.cpu_count() or 4) as pool:
        jobs = {src: pool.submit(_spills, nvcc, src, str(tmp / (src + ".o"))) for src in KNOWN}
        return {src: j.result() for src, j in jobs.items()}


@pytest.mark.parametrize("src", sorted(KNOWN))
def test_no_kernel_spills_more_than_measured(spills, src):
    kernels = {k: v for k, v in spills[src].items() if re.search(r"\d+k_", k)}
    assert kernels
    for name, stores in kernels.items():
        allowed = max((b for frag, b in KNOWN[src].items() if frag in name), default=0)
        assert stores <= allowed, (name, stores)
    for frag in KNOWN[src]:
        assert any(frag in k for k in kernels), f"{frag} matches no kernel of {src}"


def test_every_unit_with_kernels_is_covered():
    covered = set(KNOWN) | {"ns.cu", "fft_passes.cu"}  # these two: test_kernel_resources_cpu.py
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu") and f not in covered:
            text = open(os.path.join(CSRC, f)).read()
            assert "__global__" not in text or f == "inputs.cu", f
