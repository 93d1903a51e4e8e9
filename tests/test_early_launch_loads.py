"""A kernel that may be launched before the one that writes its input has ended (it
calls pdl_wait) must not read that input on the read-only path, whose loads nothing
keeps behind the wait: no __ldg, no ld.global.nc, and no const __restrict__
parameter, from which the compiler makes them."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1602_08604_gb300", "csrc")
# the tensor-core operand, written once with the context, and the grouped records of
# the variant that is launched plainly
ALLOWED = {"fold_first6_mma": {"gA", "entries", "offs"}}


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _kernels(src):
    """(name, parameters, body) of every __global__ function defined in src."""
    for m in re.finditer(r"__global__ void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", src):
        i, depth = m.end(), 1
        while depth:
            depth += {"(": 1, ")": -1}.get(src[i], 0)
            i += 1
        params = src[m.end():i - 1]
        if not re.match(r"\s*\{", src[i:]):
            continue
        j = src.index("{", i) + 1
        depth, k = 1, j
        while depth:
            depth += {"{": 1, "}": -1}.get(src[k], 0)
            k += 1
        yield m.group(1), params, src[j:k]


def test_no_read_only_loads_in_early_kernels():
    early = {}
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu"):
            for name, params, body in _kernels(_read(f)):
                if "pdl_wait" in body:
                    early[name] = (params, body)
    assert {"fold_generic", "fold_first6_weighted", "estimate_small", "assemble_low6", "fold_tma"} <= set(early)
    for name, (params, body) in early.items():
        assert not re.search(r"__ldg\s*\(|\.nc\.", body), name
        const = set(re.findall(r"const\s+[\w:<> ]+\*\s*__restrict__\s+(\w+)", params))
        assert const <= ALLOWED.get(name, set()), (name, const)
    # the bodies they share
    shared = _read("passes.cuh")
    assert not re.search(r"__ldg\s*\(|\.nc\.|const\s+[\w:<> ]+\*\s*__restrict__", shared)
    for body in (f for f in ("estimate_small.cu", "assemble_top.cu", "assemble.cu", "fold.cu")):
        assert not re.search(r"__ldg\s*\(|\.nc\.", _read(body)), body
