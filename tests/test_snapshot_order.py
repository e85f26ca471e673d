"""Snapshots whose nodes are not in preorder: what is valid, and what is not, does not depend on the order of nodes."""
import numpy as np
import pytest

import paper_2606_17059_gb300 as g
from gpu_util import seqlist_from_lists


def _flat(order):
    snap = g.p2p_snapshot_build(seqlist_from_lists([[1, 2, 3], [1, 2, 4, 5], [1, 2, 4, 6, 7], [8], [8, 9]]))
    flat = {k: np.array(v) for k, v in g.p2p_snapshot_view(snap).items()}
    g.p2p_snapshot_free(snap)
    new = np.array(order, np.int32)  # old -> new
    old = np.argsort(new)
    for k in ("label_off", "label_len", "child_begin", "child_count", "term_count"):
        flat[k] = np.ascontiguousarray(flat[k][old])
    flat["child_idx"] = new[flat["child_idx"]]
    return flat


ORDERS = [[0, 1, 2, 3, 4, 5, 6, 7], [0, 7, 6, 5, 4, 3, 2, 1], [0, 3, 1, 2, 7, 5, 6, 4]]


@pytest.mark.parametrize("order", ORDERS)
def test_any_order_is_valid(order):
    assert len(_flat(order)["label_off"]) == 8
    assert g.p2p_flat_tree_validate(_flat(order)) == 0


@pytest.mark.parametrize("order", ORDERS)
@pytest.mark.parametrize("fault", ["orphan", "two parents", "cycle", "label out of range", "child out of range"])
def test_faults_are_found_in_any_order(order, fault):
    d = _flat(order)
    root_e = int(d["child_begin"][0])
    if fault == "orphan":  # the root lists one child less; that child's subtree has no path from it
        d["child_count"][0] -= 1
    elif fault == "two parents":
        d["child_idx"][-1] = d["child_idx"][root_e]
    elif fault == "cycle":  # node a lists itself where its child was
        a = int(d["child_idx"][root_e])
        d["child_idx"][int(d["child_begin"][a])] = a
    elif fault == "label out of range":
        d["label_off"][int(d["child_idx"][root_e])] = len(d["labels"])
    else:
        d["child_idx"][root_e] = 8
    assert g.p2p_flat_tree_validate(d) == g.P2P_E_FORMAT
