"""A kernel that may start before the one before it has finished must not
promise the compiler (``__restrict__``) that nobody else writes what it loads:
only data that was complete before it could start may carry the qualifier.
The sources of the kernels launched as programmatic dependents, and of the
bodies they share with other kernels, are read for it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_05158_gb300", "csrc")

# per function: what is complete before it can start (frames behind the marks, marks behind the collide, the
# channel's link lists)
COMPLETE = {"k_refill": {"fcur", "fprev"}, "refill_body": {"fcur", "fprev"},
            "k_links": {"fcur", "flag", "owner"}, "links_body": {"fcur", "flag", "owner"},
            "k_chan_flinks": {"list"}, "k_chan_rlinks": {"list", "sp"},
            # not loaded from at all: read by bulk copies in assembly, or only added to
            "k_collide_rows": {"f", "status"}}
BODIES = {"mark_body", "mark_corr_body", "refill_body", "links_body", "rows_body"}


def source():
    return "\n".join(re.sub(r"//[^\n]*", "", open(p).read()) for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))))


def parameters(src, name):
    """Parameter lists of the definitions of `name` (a kernel's launch bounds may come before its name)."""
    out = []
    for m in re.finditer(r"(?:void|__launch_bounds__\([^{;]*?\))\s+%s\(" % name, src):
        depth, at = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(src[at], 0)
            at += 1
        if src[at:].lstrip().startswith("{"):
            out.append(src[m.end():at - 1])
    return out


def test_no_restrict_on_what_the_kernel_before_may_still_write():
    src = source()
    started_early = set(re.findall(r"launch_step\((k_\w+)", src)) | set(re.findall(r"chan_launch\(c, (k_\w+)", src))
    started_early |= set(re.findall(r"const auto k = (k_collide_rows)<", src)) | {"k_dem_local"}
    assert {"k_mark", "k_refill", "k_stream_collide", "k_stream_collide2", "k_collide_rows", "k_links", "k_chan_step",
            "k_chan_adj", "k_chan_flinks", "k_chan_rlinks", "k_chan_gsum"} <= started_early
    for name in sorted(started_early | BODIES):
        lists = parameters(src, name)
        assert lists, name
        for params in lists:
            promised = set(re.findall(r"__restrict__ (\w+)", params))
            assert promised <= COMPLETE.get(name, set()), (name, promised)
