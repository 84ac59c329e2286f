"""Acceptance at the edges of its ranges, against the oracle: vocabularies around what the threads of a cluster hold in registers
(a cluster of c CTAs holds 2048 c entries per word, eight words at most; beyond that a pass loads batch after batch), more sequences than
clusters of 16 fit, deep and wide trees of 64 rows, and rejected children whose residual has no mass."""
import numpy as np
import pytest
import torch

import sv_inputs as si

pytestmark = pytest.mark.gpu


def _check(c):
    import paper_2512_21911_b200 as sv
    from test_gpu_parity import _check_accept, _gpu_accept, _settle_accept_case
    r = _settle_accept_case(c)
    got = _gpu_accept(sv, c)
    _check_accept(c, r, got)
    dev = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
    S, T, _ = c["p_target"].shape
    out = [torch.full(shape, -9, dtype=torch.int32, device="cuda") for shape in ((S, T), (S,), (S,))]
    sv.sv_accept(*(dev(c[k]) for k in ("p_target", "p_draft", "tokens", "parent", "u_accept", "u_next")), *out)
    for a, b in zip(out, got):   # without the probabilities the walk takes first children from a table
        np.testing.assert_array_equal(a.cpu().numpy(), b)


@pytest.mark.parametrize("S,V", [(1, 2048), (1, 2052), (1, 16384), (2, 65536), (2, 65540), (1, 131072), (1, 131076), (1, 262144), (1, 262148),
                                 (10, 65536), (10, 131076), (1, 524300)])
def test_accept_at_the_edges_of_what_a_cluster_holds(S, V):
    for rejecting in (False, True):
        c = si.make_accept_case(S, 4, V, seed=V + rejecting, tree=rejecting)
        if rejecting:   # three siblings: two residuals, the second of them drawn from or followed by a third
            c["parent"][:] = np.array([-1, 0, 0, 0], np.int32)
            c["u_accept"][:] = 0.9995
        _check(c)


@pytest.mark.parametrize("wide", [False, True])
def test_accept_64_rows(wide):
    c = si.make_accept_case(3, 64, 2048, seed=64 + wide, tree=True)
    c["parent"][:] = np.concatenate([[-1], np.arange(63) // 2 * (2 if wide else 1)]).astype(np.int32)
    c["u_accept"][1] = 0.0     # all the way down first children
    c["u_accept"][2] = 0.9995
    _check(c)


def test_accept_residual_without_mass():
    """p == q and a child rejected all the same (u = 1): p stays, also when nothing is left to try."""
    c = si.make_accept_case(2, 4, 4096, seed=5, tree=True)
    c["p_draft"][:] = c["p_target"]
    c["parent"][:] = np.array([[-1, 0, 0, 0], [-1, 0, 1, 2]], np.int32)
    c["u_accept"][:] = np.array([[0, 1, 1, 1], [0, 0, 1, 0]], np.float32)
    _check(c)
