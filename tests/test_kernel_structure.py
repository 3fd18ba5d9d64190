"""What the order of a few calls inside the kernels has to be, read off the sources: a kernel that breaks one of these would hang or
race on the GPU, so nothing here runs one."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_04127_b200", "csrc")


def _kernels():
    """(file, name, body) of every __global__ function, comments removed."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        with open(path) as f:
            src = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s+)?(\w+)\s*\(", src):
            start = src.index("{", m.end())
            depth, i = 0, start
            while True:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                if depth == 0:
                    break
                i += 1
            out.append((os.path.basename(path), m.group(1), src[start:i + 1]))
    return out


KERNELS = _kernels()
TENSOR_MEMORY = [k for k in KERNELS if "tmem_alloc(" in k[2]]


def test_the_kernels_are_found():
    assert {"split_gemm_kernel", "tc_fwd_causal_kernel", "tc_bwd_nc_kernel", "tc_bwd_k_kernel"} <= {k[1] for k in TENSOR_MEMORY}


@pytest.mark.parametrize("file,name,body", TENSOR_MEMORY, ids=[k[1] for k in TENSOR_MEMORY])
def test_tensor_memory_is_taken_before_dependents_may_start(file, name, body):
    """A dependent kernel holds all of an SM's tensor memory while it waits for this kernel's end; a block of this kernel that had
    yet to take its own would wait for it, for good."""
    trigger = re.search(r"pdl_wait\w*\(\)|griddepcontrol\.launch_dependents", body)
    if trigger:
        assert re.search(r"tmem_alloc\(.*__syncthreads\(\)", body[:trigger.start()], re.S), f"{file}: {name}"


@pytest.mark.parametrize("file,name,body", TENSOR_MEMORY, ids=[k[1] for k in TENSOR_MEMORY])
def test_a_kernel_that_gave_up_waits_for_its_copies(file, name, body):
    """After a wait ran into its limit, loads into the block's shared memory may still be in flight: it sleeps before it ends."""
    assert re.search(r"__nanosleep\(200000\);(?!.*\bmbar_).*tmem_dealloc\(", body, re.S), f"{file}: {name}"


TMA = [k for k in KERNELS if re.search(r"tma_load_\w+\(|bulk_load\(", k[2])]


@pytest.mark.parametrize("file,name,body", TMA, ids=[k[1] for k in TMA])
def test_tma_reads_behind_a_proxy_fence(file, name, body):
    """What a kernel before wrote with ordinary stores is read by TMA only behind the fence that goes with the early start."""
    wait = re.search(r"pdl_wait_tma\(\)", body)
    assert wait and wait.start() < re.search(r"tma_load_\w+\(|bulk_load\(", body).start(), f"{file}: {name}"
    assert not re.search(r"pdl_wait\(\)|griddepcontrol", body), f"{file}: {name}"


@pytest.mark.parametrize("file,name,body", TENSOR_MEMORY, ids=[k[1] for k in TENSOR_MEMORY])
def test_a_wait_has_one_answer_before_tensor_memory_is_read(file, name, body):
    """Tensor-memory loads and stores are instructions of a whole warp: where the lanes of a warp could leave a wait with different
    answers, half of it would enter one. The warp votes in between."""
    for wait in re.finditer(r"(?<!__all_sync\(0xffffffffu, )\b(?:wait_or_abort|mbar_wait)\(", body):
        access = re.search(r"\btmem_(?:ld|st|row_to_tile)\w*\(", body[wait.end():])
        if access:
            between = body[wait.end():wait.end() + access.start()]
            assert "__all_sync(" in between or "warp_wait(" in between, f"{file}: {name}: {body[wait.start():wait.start() + 60]}"
