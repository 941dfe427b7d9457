"""Source check (no GPU): a kernel of the dependent-launch chain reads through no
`const T *__restrict__` parameter.  Such loads may take the read-only path and may
be moved ahead of the wait for the kernel before, which may still be writing
what they read."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1707_08900_gb300", "csrc")


def _kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__", text):
        i = text.index("(", m.end())
        while re.search(r"__launch_bounds__\s*$", text[m.end():i]):  # skip its arguments
            depth = 0
            while True:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
                if depth == 0:
                    break
            i = text.index("(", i)
        name = re.search(r"(\w+)\s*$", text[m.end():i]).group(1)
        j = text.index("{", i)
        depth, k = 0, j
        while True:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
            if depth == 0:
                break
        yield name, text[i:j], text[j:k]


def test_chained_kernels_read_plainly():
    chained, bad = [], []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        for name, params, body in _kernels(open(path).read()):
            if "chain_wait()" in body:
                chained.append(name)
                bad += [(name, p.strip()) for p in params.split(",")
                        if re.search(r"\bconst\b[^*]*\*\s*(const\s*)?__restrict__", p)]
    assert {"k_substep_lag", "k_substep_lag64", "k_input_compact", "k_loss", "k_fill_ghosts_z"} <= set(chained)
    assert not bad, bad
