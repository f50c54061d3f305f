"""An mbarrier may be waited on only after its initialisation is visible: in
every kernel that initialises one by a single thread, a block barrier lies
between the initialisation and the first wait of the other threads (read from
the source, since a missing barrier need not show in a run)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_13811_gb300", "csrc")


def _body(src, name):
    """Source text of function `name` between its braces, comments removed."""
    src = re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)
    at = re.search(r"\b%s\s*\([^;{]*\)\s*\{" % name, src)
    assert at, name
    depth, i = 1, at.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        i += 1
    return src[at.end():i]


@pytest.mark.parametrize("path,kernel,init,wait", [
    ("adjoint2d.cu", "k_adj_smooth2d", r"mbar_init\(", r"mbar_wait\("),
    ("local2d.cu", "k_smooth2d", r"mbar_init\(", r"mbar_wait\("),
])
def test_block_barrier_between_init_and_wait(path, kernel, init, wait):
    with open(os.path.join(CSRC, path)) as f:
        body = _body(f.read(), kernel)
    last_init = [m.end() for m in re.finditer(init, body)][-1]
    first_wait = re.search(wait, body).start()
    assert last_init < first_wait
    assert "__syncthreads();" in body[last_init:first_wait], f"{kernel}: nothing orders the waits after the init"
