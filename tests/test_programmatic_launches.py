"""Kernels that may be scheduled before their predecessor has finished (programmatic stream serialisation) read memory only through
loads that stay behind their wait: not through the read-only path, which requires data that nobody writes while the kernel
lives."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2608_24070_b200" / "csrc"
READ_ONLY = re.compile(r"__ldg\s*\(|__ldc[agsv]\s*\(|ld\.global\.nc|ld\.global\.ca\.nc")


def _kernels():
    for path in sorted(CSRC.glob("*.cuh")):
        code = re.sub(r"//[^\n]*", "", path.read_text())
        for part in code.split("__global__")[1:]:
            yield path.name, re.search(r"(\w+_kernel)\s*\(", part).group(1), part


def test_no_read_only_loads_behind_a_programmatic_wait():
    assert [name for _, name, body in _kernels() if "griddep_" in body and READ_ONLY.search(body)] == []


def test_the_kernels_are_found():
    found = {name for _, name, body in _kernels() if "griddep_" in body}
    assert {"dw_adapter_pair_kernel", "dense_gemm_pair_kernel", "prune24_kernel", "prune_nm_kernel"} <= found
