"""Rules that a wrong kernel breaks only now and then on a GPU, checked where they can be decided: in the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_24377_b200", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def code(name):
    """A source file without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def kernels(name):
    """(name, body) of the __global__ functions of a file."""
    src = code(name)
    for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\((?:[^(){}]|\([^(){}]*\))*\)\s*\{", src):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        yield m.group(1), src[m.end():i]


def test_remote_shared_memory_is_written_behind_a_cluster_barrier():
    # the CTA that owns the memory must have started: a whole barrier (arrive, wait) lies in front of the first access
    seen = 0
    for f in FILES:
        for name, body in kernels(f):
            at = body.find("st.shared::cluster")
            if at < 0:
                continue
            seen += 1
            before = re.findall(r"barrier\.cluster\.(arrive|wait)", body[:at])
            assert before == ["arrive", "wait"], f"{f}: {name}"
            assert re.findall(r"barrier\.cluster\.(arrive|wait)", body[at:]) == ["arrive", "wait"], f"{f}: {name}: nor may it end early"
    assert seen == 1


def included(name):
    """The headers of this folder that a source file includes, and theirs."""
    direct = re.findall(r'#include "([^"/]+)"', code(name))
    return set(direct).union(*map(included, direct))


def test_what_a_launch_before_may_write_is_not_read_as_read_only():
    # kernels that start while their predecessor runs: no read-only loads, neither asked for nor left to the compiler, also not in
    # the headers that hold their bodies
    files = [f for f in FILES if "pdl_wait()" in code(f)]
    assert len(files) >= 6
    files = sorted(set(files).union(*map(included, files)))
    assert "walk.cuh" in files
    for f in files:
        src = code(f)
        assert not re.search(r"__ldg\b|ld\.global\.nc", src), f
        for name in set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", src)):
            assert not re.search(rf"[=(,?:+*/&|-]\s*{name}\s*\[|[=(,]\s*\*\s*{name}\b", src), f"{f}: {name} is read through a const __restrict__ pointer"


def test_attention_kernels_check_where_their_tensor_memory_starts():
    # they address it from column 0: were it elsewhere, a void output would have to show in the status word
    for f in ("forward.cu", "forward_walk.cu", "forward_rows.cu", "forward_bf16.cu", "forward_nvfp4.cu"):
        bodies = [body for _, body in kernels(f) if "tcgen05.alloc" in body]
        assert len(bodies) == 1, f
        at_end = re.search(r"check_tmem_base\(\*tmem_slot, lane, p\.status\);\s*asm volatile\(\"tcgen05\.dealloc", bodies[0])
        at_start = re.search(r"if \(\*tmem_slot != 0\) \*abort_flag = kCodeTmemBase;\s*const int role", bodies[0])
        reported = re.search(r"if \(tid == 0 && \*abort_flag != 0\) atomicCAS\(p\.status, 0, \*abort_flag\);", bodies[0])
        assert at_end or (at_start and reported), f
