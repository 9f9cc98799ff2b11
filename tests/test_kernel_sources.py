"""What every kernel keeps because it is launched while the one before it still runs (no GPU needed: the sources are read)."""
import glob
import os
import re

import paper_2605_04478_b200 as ccld

CSRC = os.path.join(os.path.dirname(ccld.__file__), "csrc")
# read-only for as long as a kernel runs: the registry's tables; the caller's columns, which a call's first kernel does not touch this way
REGISTRY = {"mem", "R.members", "trees"}
COLUMNS = {"c_te", "c_tx", "c_by", "c_op", "c_sc", "c_rc", "pc", "ps", "tn", "rank", "t_enter", "t_exit"}


def sources():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))):
        yield os.path.basename(f), re.sub(r"//[^\n]*", "", open(f).read())


def kernels(src):
    """(name, parameters, body from its brace on)"""
    for m in re.finditer(r"__global__\s+void\s+__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s+(\w+)\(([^)]*)\)\s*\{", src):
        yield m.group(1), m.group(2), src[m.end():]


def test_every_kernel_waits_first():
    names = []
    for _, src in sources():
        assert src.count("__global__") == len(list(kernels(src)))
        for name, _, body in kernels(src):
            names.append(name)
            assert body.lstrip().startswith("begin_after();"), name
    assert len(names) >= 20


def test_memory_of_the_kernel_before_is_not_read_as_read_only():
    for f, src in sources():
        for name, params, _ in kernels(src):
            for p in params.split(","):
                m = re.match(r"\s*const\s+[\w:]+\s*\*\s*__restrict__\s+(\w+)", p)
                assert not m or m.group(1) in REGISTRY | COLUMNS, (f, name, p)
        for m in re.finditer(r"__ldg\((?:reinterpret_cast<[^>]*>\()?\s*([\w.]+)", src):
            assert m.group(1) in REGISTRY | COLUMNS, (f, m.group(0))
