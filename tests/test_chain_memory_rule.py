"""What an earlier kernel of a chain (or a pre-pass) writes must not be read through the read-only path: its lines may be
older than the wait.  `const T* __restrict__` lets the compiler choose that path, so in a kernel that waits for an earlier one
only the caller's own inputs and the job records may carry the qualifier."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_14090_b200", "csrc")
CALLERS_OWN = {"jobs", "w", "scale", "bias", "net_input", "labels"}


def _kernels(text):
    """(name, parameter list, body) of every __global__ function."""
    for m in re.finditer(r"__global__", text):
        head = text[m.end():]
        head = re.sub(r"^\s*void\s*__launch_bounds__\s*\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)", "", head)
        head = re.sub(r"^\s*void", "", head)
        name = re.match(r"\s*(\w+)\s*\(", head)
        if not name:
            continue
        depth, i = 1, name.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(head[i], 0)
            i += 1
        params, j = head[name.end():i - 1], head.index("{", i)
        depth, k = 1, j + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(head[k], 0)
            k += 1
        yield name.group(1), params, head[j:k]


def test_no_read_only_path_for_what_an_earlier_kernel_writes():
    waiting = 0
    for f in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for name, params, body in _kernels(text):
            if "chain_wait()" not in body and "griddepcontrol.wait" not in body:
                continue
            waiting += 1
            for p in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params):
                assert p in CALLERS_OWN, f"{f}: {name} may read {p} through the read-only path"
            for p in re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params):
                assert not re.search(r"ld_chain\(\s*%s\b" % p, body), f"{f}: {name}: ld_chain({p}) of a __restrict__ pointer"
    assert waiting >= 12
