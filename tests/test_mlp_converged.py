"""The tcgen05 kernels' warps are converged again after a wait on an mbarrier (which
lanes may leave at different times) before any instruction that takes a whole warp
(tcgen05.ld.sync.aligned, bar.sync): checked on the source, without a GPU."""
import os
import re

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_10290_gb300", "csrc",
                      "mlp_tc.cu")


def test_waits_are_followed_by_a_convergence():
    with open(SOURCE) as f:
        code = "\n".join(line.split("//")[0] for line in f.read().splitlines())
    code = code[code.index("forward"):].split("__device__ bool wait_phase")[-1]
    waits = [m for m in re.finditer(r"wait_phase\(bar, [^)]*\)", code)]
    assert len(waits) >= 8
    for m in waits:
        if code[:m.start()].endswith("__syncthreads_and("):
            continue
        after = code[m.end():].split("} else")[0]
        sync = re.search(r"__syncwarp\(\)|__syncthreads\(\)", after)
        aligned = re.search(r"tm_ld\d+\(|group_sync\(\)|tcgen05\.(ld|dealloc)|layer\(", after)
        assert aligned is None or (sync and sync.start() < aligned.start()), after[:200]
