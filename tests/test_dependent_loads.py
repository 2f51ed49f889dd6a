"""Kernels may be set up while their predecessor still runs, so what a predecessor writes is not read-only
for the kernel's lifetime: loads that assume so (``__ldg``, or pointers to const with ``__restrict__``) are
kept to what only the host writes. The compiler may move such a load above the wait for the predecessor,
which no test of results can rule out; the sources can."""
import glob
import os
import re

import pytest

from paper_2309_08068_gb300 import build as lbm_build

SOURCES = sorted(glob.glob(os.path.join(lbm_build.CSRC, "*.cu")) + glob.glob(os.path.join(lbm_build.CSRC, "*.cuh")))
# media, material table, a source cell's record (tile_source's r); p is read()'s, see the second test
HOST_WRITTEN = {"&m.id[i]", "&m.eps_r[i]", "&m.mu_r[i]", "&m.sigma[i]", "&t->c0", "&t->c1", "r", "r + 1", "p"}


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_read_only_loads_are_of_what_the_host_writes(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    loads = [m.strip() for m in re.findall(r"__ldg\(((?:[^()]|\([^()]*\))*)\)", text)]
    assert [x for x in loads if x not in HOST_WRITTEN] == []
    pointers = re.findall(r"const\s+([\w:<> ]+?)\s*\*\s*__restrict__", text)
    assert [x for x in pointers if x not in ("BatchLattice", "BatchTile")] == []  # uploaded before the launches


def test_read_only_pulls_are_for_kernels_that_are_launched_plainly():
    """read<true> is the one way to such a load of populations; the MM tiled pass and the MM backward step of
    large lattices take it, and are never launched that way while their predecessor runs."""
    text = {os.path.basename(p): open(p).read() for p in SOURCES}
    everything = "\n".join(text.values())
    assert everything.count("__ldg(p)") == 1 and everything.count("mm_pull<S, true>") == 1
    assert "load<true>" not in everything and "read<true>" not in everything
    assert not re.search(r"launch_after\(\s*mm_tile2_kernel", everything)
    assert len(re.findall(r"mm_tile2_kernel<[^>]*><<<", text["mm.cu"])) == 2
    assert re.findall(r"mm_adjoint_kernel<([^>]*)>", text["mm.cu"]) == ["M, true", "M, false"]
    assert re.search(r"mm_adjoint_kernel<M, true><<<", text["mm.cu"])
    assert re.search(r"launch_after\(mm_adjoint_kernel<M, false>", text["mm.cu"])
