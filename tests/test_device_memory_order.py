"""Rules of memory order that a kernel's source has to keep and that no run can prove: a broken one
may give the right bits on every run of one machine.  Read from the source, so they run anywhere."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1308_0692_gb300", "csrc")


def _body(name: str, kernel: str) -> str:
    """The body of `kernel` in source file `name`, comments removed."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    at = src.index("{", re.search(rf"\b{kernel}\s*\(", src).end())
    depth, end = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(src[end], 0)
        end += 1
        if depth == 0:
            return src[at:end]


def test_column_kernel_waits_for_its_cluster_before_the_first_remote_store():
    """Shared memory of another block of the cluster may be written only once that block is known
    to run: a cluster barrier comes before the first publish() (whose own one comes after its stores)."""
    body = _body("step_column.cu", "column_kernel")
    first = re.search(r"^ {4}publish\(0\);", body, re.M).start()
    straight = re.sub(r"^ {4}auto \w+ = \[&\].*?^ {4}\};", "", body[:first], flags=re.M | re.S)   # less the lambdas' bodies
    arrive, wait = straight.find("cluster_arrive();"), straight.find("cluster_wait();")
    assert 0 <= arrive < wait


def test_training_kernels_take_no_read_only_loads():
    """The kernels of a training step are programmatic dependents of each other: the one that writes
    a parameter still runs when the one that reads it starts.  The read-only path is for data that
    nobody writes during a kernel."""
    for name in ("mlp_chain.cu", "mlp_grad.cu"):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        assert not re.search(r"__ldg|ld\.global\.nc|__restrict__", src), name


def test_batch_segment_kernel_takes_no_read_only_loads_of_the_state():
    """A launch takes many steps: what it reads in one it has written, from other multiprocessors,
    in the step before."""
    body = _body("batch.cu", "batch_group")
    loads = re.findall(r"__ldg\(([^;]*);", body)
    assert loads and all(re.match(r"p\)|p \+ 1\)|a\.src", x) for x in loads), loads
    src = open(os.path.join(CSRC, "batch.cu")).read()
    assert not re.search(r"const TS \*__restrict__ h\b", src)
