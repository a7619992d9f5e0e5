"""Properties of the device code that no run can show, because they matter only after a wait
has given up, or only under the memory model: read off the sources."""
import os
import re

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2111_12478_gb300", "csrc")


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def kernel(name, text):
    """The body of kernel `name`."""
    at = re.search(r"__global__[^;{]*?\b" + name + r"\s*\(", text).start()
    at = text.index("{", text.index(")", text.index(name + "(", at)))
    depth, i = 1, at + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[at:i]


def test_tile_walker_clears_the_members_tables_first():
    # after a wait that gave up a walker reads the tables and local times of members that have
    # not arrived: they are cleared before the walkers' first meeting
    head = kernel("k_prop_wide", source("gwcp_wide.cu")).split("__syncthreads()", 1)[0]
    layout = re.search(r"nbuf = tabs \+ apb \* (\d+);\s*uint32_t\* J = nbuf \+ (\d+);\s*uint32_t\* tcnt = J \+ (\d+)", head)
    clear = re.search(r"i < apb \* (\d+) \+ (\d+) \+ (\d+); i \+= blockDim\.x\)\s*tabs\[i\] = 0;", head)
    assert layout and clear and clear.groups() == layout.groups()


def test_a_sort_tile_always_scatters():
    # a tile that left without scattering would leave words of an earlier use in the output,
    # which the next passes and phases take for keys and indices: the only early exit is that
    # of a tile past the end, and the wait that gives up ends in a count of its own
    body = kernel("k_sweep", source("gwcp_prims.cu"))
    exits = re.findall(r"if \(([^;{]*)\)\s*return;", body)
    assert exits == ["size_t(tile) * TILE >= n"]
    assert re.search(r"if \(s_gone\) count_before<", body)


def test_barrier_rows_change_by_reductions_only():
    # several members add to one word of a barrier buffer between two barriers: a plain store
    # among their reductions is a race
    body = kernel("k_propagate", source("gwcp_propagate.cu"))
    assert "st.shared" not in body and "red_max(buf + own, N)" in body


def test_no_read_only_load_of_what_the_kernel_ahead_writes():
    # the Adam kernel's blocks are placed while the gradient kernel still writes the sums that
    # they read: not data for the read-only path, which may load it ahead of the wait
    assert "__ldg" not in kernel("k_adam", source("gwcp_rank.cu"))
