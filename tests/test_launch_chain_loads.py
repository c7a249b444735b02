"""A kernel that may start before the one ahead of it has ended reads what that one
writes only after its wait, and with ordinary loads: the read-only path (__ldg, or a
const __restrict__ argument, which the compiler may read by it) is specified for data
that nothing writes while the kernel runs."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_01775_gb300", "csrc")


def block(text, at, opening, closing):
    """The text of the bracketed block that starts at text[at]."""
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == opening) - (text[i] == closing)
        if depth == 0:
            return text[at:i + 1]
    raise ValueError("unbalanced")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*(?=\()", text):
            args = block(text, m.end(), "(", ")")
            yield m.group(1), args, block(text, text.index("{", m.end() + len(args)), "{", "}")


def test_chained_kernels_read_with_ordinary_loads():
    chained = [(n, a, b) for n, a, b in kernels() if "after_previous()" in b]
    names = {n for n, _, _ in chained}
    assert {"phi_kernel", "adam_kernel", "scan_kernel", "mlp_bwd_kernel", "struct_phi_kernel",
            "sur_fwd_cluster_kernel", "rollout_fwd_kernel"} <= names
    for name, args, body in chained:
        assert "__ldg" not in body, name
        for arg in args.split(","):
            assert not ("const" in arg.split("*")[0] and "__restrict__" in arg), (name, arg)
