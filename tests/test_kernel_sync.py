"""Waits that the kernels need although leaving one out may go unnoticed in every run, checked in
the source: none of them can be shown to be missing by a run without risk to the GPU."""

import os
import re

from paper_2411_14413_gb300 import _native as N


def _source(name):
    text = open(os.path.join(N.CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _bodies(text):
    """(name, head and body) of every function definition at namespace scope."""
    for m in re.finditer(r"^(?:template[^\n]*\n)?__(?:global|device)__[^;{]*\{", text, re.M):
        end = text.index("\n}\n", m.end())
        head = m.group(0)
        yield re.findall(r"(\w+)\s*\(", re.sub(r"__\w+__\s*\([^)]*\)", "", head))[0], text[m.start():end]


def test_clusters_have_started_before_remote_stores():
    """Another block's shared memory may be accessed only once every block of the cluster has started."""
    bodies = dict(_bodies(_source("sput_adjoint.cu")))
    remote = [n for n, b in bodies.items() if "map_shared_rank" in b]
    assert remote
    for name in remote:
        b = bodies[name]
        first = b.index("map_shared_rank")
        assert "cluster_wait()" in b[:first], name
        assert "cl.sync()" in b[first:], name
    kernels = [n for n, b in bodies.items() if "__cluster_dims__" in b]
    assert kernels
    for name in kernels:
        # arrived in program order before anything that could leave or diverge
        b = bodies[name]
        head = b[b.index("{"):b.index("cluster_started()")] if "cluster_started()" in b else None
        assert head is not None and not re.search(r"\b(if|for|while|return)\b", head), name


def test_warp_scratch_is_ordered_between_its_uses():
    """A warp's scratch in shared memory serves the surface test and the partner sampling in turn.
    Votes and shuffles do not order memory: after the last reads of each use there is a __syncwarp."""
    bodies = dict(_bodies(_source("sput_transport.cu")))
    surface = bodies["nearest_hit_masks"]
    reads = surface.rindex("list[at]")
    leave = surface.index("if (total < 32) return;")
    assert reads < surface.index("__syncwarp()", reads) < leave
    partner = bodies["partner_sample_warp"]
    reads = partner.rindex("ws->ask")
    again = partner.index("if (own)", reads)
    assert "if (!own) __syncwarp();" in partner[reads:again]
