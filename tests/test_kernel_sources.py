"""Rules of the kernels' source text that no run can show: a violation works until a compiler or a neighbouring
kernel changes."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1207_0486_gb300", "csrc")


def _early_kernels():
    """(name, parameters, body after the wait) of every kernel that waits for its predecessor inside."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = re.sub(r"//[^\n]*|__launch_bounds__\s*\([^)]*\)", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\(([^{]*?)\)\s*\{", src):
            body, depth = src[m.end():], 1
            for e, ch in enumerate(body):
                depth += {"{": 1, "}": -1}.get(ch, 0)
                if depth == 0:
                    break
            if "griddepcontrol.wait" in body[:e]:
                out.append((m.group(1), m.group(2), body[:e].split("griddepcontrol.wait", 1)[1]))
    return out


def test_nothing_of_a_device_is_kept_for_the_process():
    """A kernel's shared-memory limit and occupancy belong to the device that was current. Kept in a function's static, they
    would hold for the first device alone: an operator on a second one could not launch tiles above 48 KB."""
    kept = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        src = open(path).read()
        kept += [(os.path.basename(path), m.group(0).strip())
                 for m in re.finditer(r"^[ \t]+static (?:const )?(?:bool|int|size_t) \w+[^;(]*[;=].*$", src, re.M)
                 if "constexpr" not in m.group(0)]
    assert not kept, kept


def test_kernels_launched_early_read_nothing_as_constant_after_their_wait():
    """A kernel launched ahead of its predecessor's end is resident while that one still writes. A const
    __restrict__ parameter or __ldg may be a read-only load, which is defined only for data that nobody writes
    during the kernel's life, and may be moved above the wait."""
    kernels = _early_kernels()
    assert [k[0] for k in kernels] == ["k_ic0_sweep"]
    for name, params, after in kernels:
        constant = re.findall(r"const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", params)
        used = [p for p in constant if re.search(rf"\b{p}\b", after)]
        assert not used, (name, used)
        assert "__ldg" not in after, name
