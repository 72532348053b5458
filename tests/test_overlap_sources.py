"""Ordering of launches that overlap (programmatic dependent launch), checked on the sources: a kernel set up while the
one before it runs may read what that one wrote only behind griddepcontrol.wait or an acquire that pairs with a release.
A missing wait shows on a GPU as wrong bytes at best, so it is looked for here, without one."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1902_05320_gb300", "csrc")


def sources():
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            out[os.path.basename(path)] = re.sub(r"//[^\n]*", "", f.read())
    return out


def block(text, at, pair):
    """The text of the bracketed group that opens at or after `at`, and where it ends."""
    start = text.index(pair[0], at)
    depth, i = 0, start
    while True:
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        i += 1
        if depth == 0:
            return text[start:i], i


def kernels():
    """name -> (parameters, body) of every __global__ function."""
    out = {}
    for text in sources().values():
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\s*)?", text):
            at = m.end()
            if text[at] == "(":
                _, at = block(text, at, "()")
            name = re.compile(r"\s*(\w+)\s*").match(text, at)
            params, at = block(text, name.end(), "()")
            body, _ = block(text, at, "{}")
            out[name.group(1)] = (params, body)
    return out


def test_the_parser_sees_the_kernels():
    found = kernels()
    assert {"k_sha3_uniform", "k_sha3_uniform_coop", "k_sha3_queue", "k_sha3_lanes", "k_scatter", "k_merkle_climb",
            "k_stream_step", "k_keccak_p_1600"} <= set(found)
    assert "launch_wait()" in found["k_sha3_lanes"][1]


def test_queue_kernel_takes_the_plan_over_before_it_reads_it():
    """k_sha3_queue starts once the blocks of k_sha3_lanes have let it, without waiting for that kernel's end; what it
    reads was written by the kernel before both, so one block of k_sha3_lanes, which has waited for that one, hands it
    over by a release, and the queue kernel acquires it (or waits) before its first read."""
    found = kernels()
    lanes, queue = found["k_sha3_lanes"][1], found["k_sha3_queue"][1]
    assert lanes.index("launch_wait()") < lanes.index("hand_over(&ctl->ready)") < lanes.index("launch_next()")
    assert lanes.index("hand_over(&ctl->ready)") < lanes.index("return")  # on the early exit as well
    take = queue.index("taken_over(&ctl->ready)")
    handed = queue[queue.index("if (beside)"):queue.index("__syncthreads();") + 16]
    assert "if (threadIdx.x < 32 && !taken_over(&ctl->ready)) launch_wait();" in handed, "no wait without the flag"
    take = queue.index("__syncthreads();")  # the other warps of the block go on behind it
    for read in ("ctl->queue_start", "ctl->queue_mid", "ctl->slots", "ctl->ends", "order[", "out_off"):
        assert take < queue.index(read), read
    assert "__restrict__" not in found["k_sha3_queue"][0], "read-only loads may be moved before the acquire"
    queue_cuh = sources()["queue.cuh"]
    assert "st.release.gpu" in block(queue_cuh, queue_cuh.index("void hand_over("), "{}")[0]
    assert "ld.acquire.gpu" in block(queue_cuh, queue_cuh.index("bool taken_over("), "{}")[0]


def test_no_read_only_loads():
    """A read-only load (__ldg, ld.global.nc, or a plain one of a const __restrict__ parameter) is for data that does not
    change while the kernel runs, set-up included, so a compiler may move it before griddepcontrol.wait.  The sponge's
    loads are shared by all kernels, so there are none at all; __restrict__ is left to kernels launched plainly."""
    for name, text in sources().items():
        assert "__ldg" not in text and "global.nc" not in text, name
    for name, (params, body) in kernels().items():
        if "launch_wait()" in body:
            assert "__restrict__" not in params, name


def test_overlapped_kernels_wait_before_they_read():
    found = kernels()
    launched = set()
    for text in sources().values():
        for m in re.finditer(r"\b(?:launch_overlapped|launch_tiled|book)\s*\(", text):
            launched |= set(re.findall(r"\bk_\w+", block(text, m.start(), "()")[0]))
    assert len(launched) >= 18 and launched <= set(found)
    keccak_p = sources()["keccak_p.cu"]
    tile, _ = block(keccak_p, keccak_p.index("void run_tile("), "{}")
    assert tile.index("launch_wait()") < tile.index("cp.async.ca")
    for name in launched:
        params, body = found[name]
        wait = re.search(r"launch_wait\(\)|run_tile\(", body)
        assert wait, name
        before = body[:wait.start()]
        for pointer in re.findall(r"\*\s*(\w+)", params):
            assert not re.search(rf"\b{pointer}\s*(\[|->)|[^&\w]\*{pointer}\b", before), (name, pointer)
