"""Which pass of the moments writes a node's walk record, restated and checked on
trees cut at every level (node arrays too small for the deeper levels): the pass
over nodes without children and the pass over the internal nodes of the levels
above the last kept one together write every record exactly once, so that
nothing can follow a record that this call did not write.  CPU only."""
import numpy as np
import pytest

import oracle


@pytest.mark.parametrize("n,n_leaf", [(40, 1), (600, 8), (900, 16)])
def test_every_node_of_a_cut_tree_has_its_record(n, n_leaf):
    pos = np.random.default_rng(n).random((n, 3))
    nodes = oracle.Tree(pos, np.ones(n), np.full(n, 0.01), n_leaf=n_leaf, n_grp=64).nodes()
    level, nchild, first = nodes["level"], nodes["nchild"], nodes["child_first"]
    for last in range(int(level.max()) + 1):
        kept = level <= last
        # ids are breadth-first: the kept nodes are 0 .. nn - 1, and a node of
        # the last kept level has lost its children
        nn = int(kept.sum())
        assert kept[:nn].all()
        lv = level[:nn]
        nc = np.where(lv == last, 0, nchild[:nn])
        top = int(lv.max()) - 1  # the levels' pass starts one above the last kept level
        by_leaves = nc == 0
        by_levels = (nc > 0) & (lv <= top)
        assert (by_leaves ^ by_levels).all()
        # and what the records lead to are nodes of the tree
        inner = nc > 0
        assert (first[:nn][inner] + nc[inner] <= nn).all()


def test_the_passes_of_the_source_follow_this_rule():
    import os
    import re
    src = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                            "paper_1601_03138_gb300", "csrc", "build.cu")).read()
    leaves = src[src.index("k_moments_leaves(MomArgs"):src.index("k_moments_small(MomArgs")]
    assert re.search(r"meta_nchild\(A\.nd_meta\[i\]\) == 0u", leaves) and "meta_leaf(A.nd_meta" not in leaves
