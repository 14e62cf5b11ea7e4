"""Orders inside the kernels that a run cannot show safely, read from the
sources: a wrong one hangs the GPU or writes into another CTA's memory."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2110_06037_gb300", "csrc")


def kernels():
    """(name, body without comments) of every __global__ function."""
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(f).read())
        for m in re.finditer(r"__global__", text):
            brace = text.index("{", m.end())
            name = re.findall(r"(\w+)\s*\(", re.sub(r"__launch_bounds__\([^)]*\)", "", text[m.end():brace]))[0]
            depth, i = 1, brace + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            yield name, text[brace:i]


def test_no_kernel_lets_its_successor_start_before_it_holds_its_tensor_memory():
    """tcgen05.alloc waits without a limit.  Were the next kernel's CTA resident
    before this one has allocated, it could hold the columns that this one needs
    while it waits for this one to complete."""
    seen = {}
    for name, body in kernels():
        if "tmem_alloc<" in body:
            alloc = body.index("tmem_alloc<")
            barrier = min(p for p in (body.find("__syncthreads()", alloc), body.find("cluster_sync_all()", alloc)) if p > 0)
            launches = [m.start() for m in re.finditer(r"griddep_launch\(\)", body)]
            seen[name] = len(launches) == 1 and launches[0] > barrier
    assert {"conv_tc_kernel", "conv_tc_lat_kernel", "conv_split_kernel", "expand_dw_kernel", "conv_chain_kernel"} <= set(seen)
    assert all(seen.values()), seen


def test_a_cluster_tile_that_gives_up_still_sends_and_receives_its_sums():
    """A peer's st.async completes only through the mbarrier of the CTA that it
    writes into: a CTA may leave once x_bar has counted every byte, on the error
    path too, and so every CTA has to send, on the error path too."""
    body = dict(kernels())["conv_tc_lat_kernel"]
    drain = body[body.index("if (abort_sh && lane == 0)"):]
    assert "x_bar" in drain[:drain.index("tmem_dealloc")]
    failed = body[body.rindex("ERR_ACC_WAIT"):]  # in the epilogue of a cluster, the last of the roles
    assert "st_async_v4" in failed[:failed.index("} else {")]
