"""The staged-row collide gives up a wait only with a bound, and its producer
then waits for the loads it has in flight, which write to the block's shared
memory.  No run can be made to get there (a wait of a sound kernel does not
run out), so the source is read for it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_05158_gb300", "csrc")


def test_a_producer_that_gives_up_waits_for_its_loads():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "lbm_rows.cuh")).read())
    wait = re.search(r"bool mbar_wait\(.*?\n}\n", src, re.S).group(0)
    assert re.search(r"for \(int i = 0; i < \(1 << \d+\); \+\+i\)", wait) and "return false" in wait
    producer = src[src.index("if (warp == cwarps) {"):src.index("} else {\n        for (int it = 0; it < mine; ++it) {")]
    # every load counted, and after a wait that ran out the ones from the unit at work on waited for
    assert producer.count("load(") == 3 and "load(it - 1 + nst);\n                loaded = it + nst;" in producer
    assert "int loaded = min(nst, mine), it = 0;" in producer and "for (int i = 0; i < loaded; ++i) load(i);" in producer
    gave_up = producer.index("if (!ok) rows_give_up(get(blockIdx.x).status, full0, it, loaded, nst, lane);")
    assert gave_up < producer.index("cp.async.bulk.wait_group 0")
    body = re.search(r"void rows_give_up\(.*?\n}\n", src, re.S).group(0)
    assert re.search(r"for \(; it < loaded; \+\+it\) mbar_wait\(full0 \+ 8 \* \(it % nst\), \(it / nst\) & 1\);", body)
