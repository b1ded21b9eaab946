"""Cluster barriers of the kernels that read another CTA's shared memory.  Only a
releasing arrival orders such a load before the owner's next store to the place
(PTX memory model: a relaxed arrival orders nothing, and a release restricted to
shared::cta covers a CTA's own memory alone); a missing one shows as a rare wrong
value on some compiler, so the order is checked in the source."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1807_11313_gb300", "csrc")
RELEASE = "cluster_arrive()"


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_every_arrival_releases():
    """No arrival without a release of its own or a release fence in the same statement."""
    found = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        for text in re.findall(r"asm volatile\((.*?)\);", _code(os.path.basename(path)), flags=re.S):
            if "barrier.cluster.arrive" not in text:
                continue
            found += 1
            assert "barrier.cluster.arrive.release" in text or re.search(r"fence\.(release|acq_rel).*barrier\.cluster\.arrive", text, re.S), (path, text)
    assert found >= 2


def _events(name, kernel):
    """The kernel's barriers, gathers of whole surfaces and reads of sums, in source order."""
    body = _code(name)
    body = body[re.search(kernel + r"\(const", body).start():]
    body = body[:body.index("\n}\n")]
    pat = r"cluster_arrive\w*\(\)|gather_lines\(|gather<0>\(|ld_cluster\(at|ld_cluster(?:_f)?\(map_to_rank|if \(bad\)|continue;"
    return [m.group(0) for m in re.finditer(pat, body)]


@pytest.mark.parametrize("name,kernel,gathers", [("k_search256.cu", "k_search256", 1), ("k_peak256.cu", "k_peak256", 1),
                                                 ("k_prep256.cu", "k_prep256", 2)])
def test_release_after_gathers(name, kernel, gathers):
    """The first barrier after a gather lets the owner overwrite what was read: it releases."""
    ev = _events(name, kernel)
    at = [i for i, e in enumerate(ev) if e.startswith("gather") or e == "ld_cluster(at"]
    after = [next(e for e in ev[i:] if e.startswith("cluster_arrive")) for i in at]
    assert len(at) >= gathers and after == [RELEASE] * len(at)


def test_release_after_sums():
    """Sums and maxima read from the other CTAs: a releasing arrival before their slots are written again."""
    ev = _events("k_peak256.cu", "k_peak256")
    last = max(i for i, e in enumerate(ev) if e.startswith("ld_cluster(map"))
    assert next(e for e in ev[last:] if e.startswith("cluster_arrive")) == RELEASE
    # pre-processing: the sums of an image are read before its gathers (which release); one without
    # signal has no gathers and releases before the next image starts
    ev = _events("k_prep256.cu", "k_prep256")
    first = next(i for i, e in enumerate(ev) if e.startswith("ld_cluster(map"))
    assert ev.index("ld_cluster(at") > first
    bad = ev[ev.index("if (bad)"):]
    assert RELEASE in bad[:bad.index("continue;")]
