"""The bench's work table knows every kernel that the library names."""
import pathlib
import re

import bench
import synth

CSRC = pathlib.Path(bench.__file__).parent / "paper_2608_28511_gb300" / "csrc"


def _names():
    src = "\n".join(p.read_text() for p in sorted(CSRC.glob("*.cu")))
    names = set(re.findall(r'KernelScope ks\("([a-z0-9_]+)"', src)) | set(re.findall(r'"([a-z0-9_]+_(?:tc|simt))"', src))
    assert {"topk", "perm_dispatch", "ffn_bwd_simt", "shared_wgrad_tc"} <= names
    return sorted(names)


def test_every_kernel_has_its_work():
    w = synth.Workload("w", S=64, GBS=1, D=128, E=8, K=2, F=64, H=256)
    for n in _names():
        bound, work = bench.kernel_work(n, w, w.T, 64)
        # (setup work of no algorithmic size is counted as 0, a product never)
        assert bound in ("tensor", "hbm") and work >= 0.0, n
        if n.endswith(("_tc", "_simt")) and n.rsplit("_", 1)[0] != "router_gemm":
            assert bound == "tensor" and work > 0.0 and bench.gemm_bytes(n, w, w.T, 64) > 0.0, n


def test_merged_launches_count_as_their_parts():
    w = synth.Workload("w", S=64, GBS=1, D=128, E=8, K=2, F=64)
    parts = sum(bench.kernel_work(n, w, w.T)[1] for n in ("ffn2_wgrad_simt", "ffn1_wgrad_simt", "ffn1_dgrad_simt"))
    assert bench.kernel_work("ffn_bwd_simt", w, w.T) == ("tensor", parts)
    assert bench.kernel_work("perm_dispatch", w, w.T)[1] >= bench.kernel_work("dispatch_rows", w, w.T)[1] - 4 * w.T * w.K
    assert {"dispatch_rows", "perm_dispatch"} <= set(bench.PERM_KERNELS)
