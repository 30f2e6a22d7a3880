"""A kernel's dynamic shared memory limit is process-wide state: it is set only
through GBSP_SMEM_LIMIT, which takes constants alone, so that no host thread
can lower it under another's launch."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_0910_4836_gb300" / "csrc"


def test_limits_are_constants():
    sources = {p.name: p.read_text() for p in CSRC.iterdir() if p.suffix in (".cu", ".cuh")}
    named = {f for f, s in sources.items() if "MaxDynamicSharedMemorySize" in s}
    assert named == {"internal.cuh"}
    macro = re.search(r"#define GBSP_SMEM_LIMIT.*?while \(0\)", sources["internal.cuh"], re.S).group(0)
    assert "constexpr int limit__" in macro and macro.count("limit__") == 2
    assert sum(s.count("GBSP_SMEM_LIMIT(") for s in sources.values()) > 1
