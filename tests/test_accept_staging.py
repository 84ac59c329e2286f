"""Acceptance at vocabularies around the threads' and CTAs' shares of a row (4 entries a word; 65536 on eight CTAs are four words a thread;
151936 and 212992 also ones that a real model has, or that took another path when rows were staged in shared memory), against the
oracle and with every child of a row rejected in turn."""
import numpy as np
import pytest

import sv_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [4, 2044, 8188, 65532, 65540, 151936, 212992, 212996])
def test_accept_at_the_edges_of_segments(V):
    import paper_2512_21911_b200 as sv
    from test_gpu_parity import _check_accept, _gpu_accept, _settle_accept_case
    for rejecting in (False, True):
        c = si.make_accept_case(2, 4, V, seed=V + rejecting, tree=rejecting)
        if rejecting:
            c["parent"][:] = np.array([-1, 0, 0, 0], np.int32)
            c["u_accept"][:] = 0.9995
        r = _settle_accept_case(c)
        _check_accept(c, r, _gpu_accept(sv, c))
