"""The bounded waits of the tensor-core contraction, read from its source (a wait that runs
out cannot be made to happen on a GPU without breaking the kernel): a role of one lane may
wait for itself, a role of whole warps only as a warp, because the loads of the accumulators
behind its wait take every lane."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1907_12334_gb300", "csrc", "kl_tc.cu")


def test_whole_warps_wait_as_warps():
    src = open(SRC).read()
    kernel = src[src.index("k_kl_tc(const __grid_constant__"):src.index("struct TcLayout")]
    roles = re.findall(r"if \(([^{]*)\) \{  // ---- (\w+)\n(.*?)(?=\n    \} else if|\n    \}\n    __syncwarp)", kernel, re.S)
    assert [name for _, name, _ in roles] == ["loads", "MMAs", "epilogue"]
    for cond, name, body in roles:
        one = "lane == 0" in cond
        assert re.search(r"\bmbar_wait\(" if one else r"\bwarp_wait\(", body), name
        assert one or not re.search(r"\bmbar_wait\(", body), name
    assert re.search(r"bool warp_wait\([^)]*\)\s*\{\s*return __all_sync\(0xffffffffu, mbar_wait\(", src)
