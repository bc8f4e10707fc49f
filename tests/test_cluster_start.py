"""Every kernel that reaches into another CTA's shared memory first waits, at a
cluster barrier, until the whole cluster runs: before that the target CTA may
not have started, and the access is undefined.  Read from the sources (no GPU):
in the order in which a kernel's body runs, the first of its cluster barriers
and its accesses through map_shared_rank has to be a barrier.  Accesses inside a
lambda count where the lambda is used."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2302_13524_gb300", "csrc")
TOUCH, SYNC = "map_shared_rank", "cluster.sync()"


def _block(text, start):
    """The text between the braces that open at or after start, and where it ends."""
    i = text.index("{", start)
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i + 1:j], j + 1
        j += 1


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__", text):
            head = re.compile(r"\b(k_\w+)\(").search(text, m.end())
            body, _ = _block(text, text.index(")", head.end()))
            if TOUCH in body:
                yield f"{os.path.basename(path)}:{head.group(1)}", body


KERNELS = dict(_kernels())


def test_the_cluster_kernels_are_found():
    assert {k.split(":")[1] for k in KERNELS} >= {"k_solver", "k_solver_row", "k_prep_select_int"}


@pytest.mark.parametrize("kernel", sorted(KERNELS))
def test_a_cluster_barrier_comes_before_the_first_remote_access(kernel):
    body, lambdas = KERNELS[kernel], {}
    while (m := re.search(r"auto (\w+) = \[[^\]]*\]", body)) is not None:
        inner, end = _block(body, m.end())
        lambdas[m.group(1)] = inner
        body = body[:m.start()] + body[end:]
    touching = {n for n, t in lambdas.items() if TOUCH in t}
    for _ in lambdas:  # lambdas that call such ones
        touching |= {n for n, t in lambdas.items() if any(re.search(rf"\b{x}\b", t) for x in touching)}
    names = "|".join([TOUCH, re.escape(SYNC)] + sorted(touching))
    first = re.search(rf"(?<!\w)(?:{names})", body)
    assert first is not None and first.group(0) == SYNC, f"{kernel}: {first and first.group(0)} comes first"
