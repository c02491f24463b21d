"""TreeSession's host side: what it hands to the binding, without a GPU."""
import dataclasses

import pytest

from workloads import CONFIGS


@pytest.fixture(scope="module")
def B():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2509_06040_b200 import binding
    return binding


def test_fusion_takes_the_settings_the_workload_has_when_it_is_called(B, monkeypatch):
    """Another beta, eps or clip tried on the same trees: the next call uses it (as pruning does with its settings)."""
    from paper_2509_06040_b200.session import TreeSession
    s = TreeSession(CONFIGS["toy"], device="cpu")
    seen = []
    monkeypatch.setattr(B, "tree_fuse_advantage", lambda tree, r, beta, scale, eps, clip: seen.append((beta, scale, eps, clip)))
    s.fuse_advantage()
    s.w = dataclasses.replace(s.w, beta=0.5, eps=1e-3, adv_clip=4.0)
    s.fuse_advantage()
    assert seen == [(CONFIGS["toy"].beta, 1.0, CONFIGS["toy"].eps, CONFIGS["toy"].adv_clip), (0.5, 1.0, 1e-3, 4.0)]
