"""Rules on the kernel sources whose breach no run shows reliably: the compiler may
or may not use the freedom that the source gives it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_13947_gb300", "csrc")


def _sources():
    return {os.path.basename(p): open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cu")))}


def _kernels(src):
    """(name, arguments, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+(?:__launch_bounds__\([^{;]*?\)\s+)?void\s+(k_\w+)\s*\(([^{;]*?)\)\s*\n\{", src):
        end = src.index("\n}\n", m.end())
        yield m.group(1), m.group(2), src[m.end():end]


def test_kernels_launched_ahead_promise_nothing_about_their_predecessors_output():
    """A kernel that may start before its predecessor ends (pdl_wait) reads the
    predecessor's output: the weights Wb and the partial sums.  const __restrict__ would
    declare them read-only for the kernel's whole lifetime."""
    seen = 0
    for src in _sources().values():
        for name, args, body in _kernels(src):
            if "pdl_wait();" not in body:
                continue
            seen += 1
            for arg in args.split(","):
                if re.search(r"\b(Wb|partial|master|mom|vel)\b", arg):
                    assert "__restrict__" not in arg, (name, arg.strip())
        for fn in re.findall(r"void load_net\(([^)]*)\)", src):
            assert "__restrict__" not in fn
    assert seen == 2


def test_aligned_instructions_follow_a_warp_synchronisation():
    """An .aligned barrier or tensor-memory instruction wants all threads of the warp
    together.  After a branch that only some of them took, nothing but a warp
    (or block) synchronisation says that they are."""
    seen = 0
    for name, src in _sources().items():
        lines = src.split("\n")
        for i, line in enumerate(lines):
            if not re.search(r'"(barrier\.cluster\.arrive\S*\.aligned|bar\.(sync|red)|tcgen05\.(alloc|dealloc|ld)\.)', line):
                continue
            seen += 1
            before = "\n".join(lines[max(0, i - 7):i])
            assert "__syncwarp();" in before or "__syncthreads();" in before, (name, i + 1, line.strip())
    assert seen >= 10
