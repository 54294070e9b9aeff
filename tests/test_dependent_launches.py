"""Kernels that may start while the kernel before them still runs read nothing that
it writes through the read-only path.

A kernel that waits in grid_wait is launched beside its predecessor, so the
predecessor's output is not read-only for the kernel's life: no `const T*
__restrict__` parameter and no __ldg may reach it.  Read from the sources, since
the results are usually right all the same.
"""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0901_3293_gb300", "csrc")

# complete before the kernel is launched: the host's tables and force field, and what the step before wrote (the
# kernel between them starts this one only after its own wait)
COMPLETE = {"reps", "order", "bext", "f", "Qin"}


def functions():
    """(name, parameters, body) of every device function and kernel."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        text = re.sub(r"__launch_bounds__\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)", "", text)
        for m in re.finditer(r"__(?:global|device)__\s+(?:__forceinline__\s+)?void\s+(\w+)\s*\(", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            params = text[m.end():i - 1]
            if text[i:].lstrip()[:1] != "{":
                continue
            start = text.index("{", i)
            depth, k = 1, start + 1
            while depth:
                depth += {"{": 1, "}": -1}.get(text[k], 0)
                k += 1
            yield m.group(1), params, text[start:k]


def test_dependent_kernels_read_through_plain_pointers():
    found = list(functions())
    waiting = {name for name, _, body in found if "grid_wait()" in body}
    waiting |= {name for name, _, body in found if any(re.search(rf"\b{w}<", body) for w in waiting)}
    assert {"k_conv_win", "k_dw_tc", "k_dw_reduce", "k_sur_loss", "k_sum", "k_adam", "k_qside", "k_lbq", "k_heun",
            "k_qsite", "k_rate_input"} <= waiting
    wrong = [(name, p) for name, params, _ in found if name in waiting
             for p in re.findall(r"const\s+[\w:]+(?:<\w+>)?\s*\*\s*__restrict__\s+(\w+)", params) if p not in COMPLETE]
    wrong += [(name, p) for name, _, body in found if name in waiting
              for p in re.findall(r"__ldg\(\s*&?\s*\(?(\w+)", body) if p not in COMPLETE]
    assert not wrong
