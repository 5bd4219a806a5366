"""The end of the coarse-level cluster kernel: a CTA's shared memory stays until every
other CTA has read its part of the coarse iterate from it.  Shown on the source and on
the slabs' arithmetic, without a GPU."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_07732_gb300", "csrc",
                   "mg_cluster.cuh")


def kernel_body():
    s = re.sub(r"//[^\n]*", "", open(SRC).read())
    a = s.index("{", s.index("k_mg_cluster("))
    depth, e = 0, a
    while True:
        depth += {"{": 1, "}": -1}.get(s[e], 0)
        e += 1
        if depth == 0:
            return s[a:e]


def ends_in_cluster_barrier(body):
    """Whether every thread waits at a cluster barrier behind the loop over the levels,
    having arrived at it before the last pass (which stores to no other CTA) or there."""
    tail = re.search(r"if \(C > 1\) \{\s*const bool last_pass = ([^;]*);\s*if \(!last_pass\) cl_arrive\(\);\s*"
                     r"cl_depart\(\);", body)
    early = re.search(r"const bool fin = ([^;]*);\s*if \(fin && C > 1\) cl_arrive\(\);", body)
    if not tail or not early or body.count("cl_arrive(") != 2:
        return False
    # the two arrivals exclude one another: the last pass is the black one of the last of
    # nu2 sweeps of the first level, run by every CTA that the level has not left out
    assert early.group(1) == "!down && q == 0 && s == nu - 1 && col == 1"
    assert tail.group(1) == "last > 0 && nu2 > 0 && (M.v[0].nct > 1 || rank == 0)"
    assert "if (v.nct == 1 && rank > 0) continue;" in body
    # no access to another CTA behind the arrivals
    rest = body[early.end():]
    stores = rest.index("cl_store_async")
    assert "if (!fin) {" in rest[:stores]
    assert not re.search(r"remote\(|coarse\(|cl_store_async|cl_addr", body[tail.start():])
    return True


def slab(ns, C):
    t = -(-ns // C)
    t += t & 1
    return t, -(-ns // t)


# layers of the first level, CTAs; whether CTA 0 alone runs the next level
@pytest.mark.parametrize("ns,C,single", [(32, 16, False), (16, 8, False), (28, 16, False), (24, 16, False), (64, 16, False),
                                         (32, 16, True), (20, 16, False)])
@pytest.mark.parametrize("nu2", [0, 1, 2, 3, 4])
def test_no_cta_leaves_before_its_readers(ns, C, single, nu2):
    t, nct = slab(ns, C)
    tc, ncc = (ns // 2, 1) if single else slab(ns // 2, C)
    barrier = ends_in_cluster_barrier(kernel_body())
    for r in range(nct):
        for k in range(max(0, r * t - 1), min(ns, r * t + t + 1)):  # its own layers and the halo's
            owner = (k >> 1) // tc if ncc > 1 else 0
            # a pass's halo exchange orders neighbours; nu2 = 0 has a cluster barrier instead
            reach = C if nu2 == 0 else 2 * nu2 - 1
            assert barrier or abs(r - owner) <= reach, f"CTA {owner} may leave while CTA {r} reads layer {k >> 1}"
