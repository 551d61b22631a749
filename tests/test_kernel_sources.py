"""Rules of the kernel sources that no result shows reliably, checked on the
text of the CUDA files."""
import glob
import os
import re

from tests.conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1507_05988_gb300", "csrc")


def _kernels():
    """name -> text from the kernel's opening brace to its closing one."""
    out = {}
    for path in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^{;]*?\)\s*)?(\w+)\([^{;]*\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            out[m.group(1)] = text[m.end():i]
    return out


def test_kernels_of_programmatic_launches_wait_for_their_predecessor():
    """launch_k can let a kernel start while the one before it still stores
    (FCN_PDL=1): each of its kernels waits (pdl_enter) before the first access
    to global memory, that is, before its first use of an argument."""
    kernels = _kernels()
    assert len(kernels) > 20
    names = set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")):
        for arg in re.findall(r"launch_k\(\s*([\w:]+)", re.sub(r"//[^\n]*", "", open(path).read())):
            names.add(arg)
    names -= {"void"}                     # its own declaration
    assert names >= {"k", "cn_kernel", "cn_pair_kernel", "cn_block_kernel", "cn_seq_kernel", "xy_line_kernel"}
    names = (names - {"k"}) | {"row_kernel"}        # RowForm::launch picks the mode's row_kernel
    for name in names:
        body = kernels[name]
        head, sep, _ = body.partition("pdl_enter();")
        assert sep, f"{name} does not wait"
        assert not re.search(r"\w+\[|->|\*\s*\w+\s*=|\b[am]\.\w+", re.sub(r"extern __shared__[^;]*;", "", head)), name


def test_cartesian_field_accesses_are_checked():
    """The self-checking build sees every access of the Cartesian kernels to
    the field: no pointer in them is followed but through FCN_PTR, and the
    field is not indexed."""
    kernels = _kernels()
    for name in ("xy_line_kernel", "xy_point_kernel"):
        body = re.sub(r",\s*\*\w+\s*=", ",", kernels[name])            # further pointers of a declaration
        followed = re.findall(r"(?:^|[=(;{?:,)])\s*\*(\w+)", body)
        assert followed and set(followed) == {"FCN_PTR"}, (name, followed)
        assert not re.search(r"\b(field|p|p1|p2|l1|l2)\[(?!k)", body), name
