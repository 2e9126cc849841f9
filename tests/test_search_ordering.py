"""Memory ordering between the kernels of one search, read from the sources (a missing ordering
does not show in results, so no run can test for it)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_09996_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_rerank_orders_the_shortlist_after_the_walk_that_wrote_it():
    # The re-rank of an ordered search runs while walks still write.  One lane acquires the entry
    # of an ended walk; a shuffle hands the query to the others but orders no memory, so a warp
    # barrier has to stand between the acquire and the reads of the shortlist.
    body = source("lc_search.cu").split("refine_kernel(const RefineArgs a)")[1]
    acquire, read = body.index("ld.acquire.gpu"), body.index("a.shortlist")
    assert acquire < read
    last_shuffle = body.rindex("__shfl_sync(FULL, e, 0)", acquire, read)
    assert "__syncwarp()" in body[last_shuffle:read]


def test_read_only_loads_take_nothing_that_an_earlier_kernel_of_the_search_writes():
    # A kernel of a search may start while the one ahead still writes, and the read-only load path
    # is only for data that stays unwritten while the reading grid lives.
    written = r"\b(a\.(seed|seed_d|seed_up|order|yq|yq_in|shortlist|list|done_list)|key|yrot|sl)\b"
    for name in ("lc_walk.cuh", "lc_search.cu"):
        loads = re.findall(r"__ldg\(([^;]*)", source(name))
        assert loads
        assert not [x for x in loads if re.match(written, x.strip())], name


def test_a_team_is_told_of_no_empty_step():
    # The walk hands its helpers the number of nodes to score, and 0 says that the walk has ended: a
    # row without neighbours (the top level, mostly) must not be announced.
    body = source("lc_walk.cuh").split("walk_kernel(const WalkArgs a)")[1]
    announce = body.index("ctl[1] = ns")
    assert "ns > 0" in body[body.rindex("if", 0, body.rindex("{", 0, announce)):announce]
