"""A request server on either side of the line between products from planes and
without: max_requests x the largest plane ring against a quarter of the arena. With
them a request has the bits of the same matrix alone; without, every request is
within the precision's bound of the oracle (1e-12, 1e-5) all the same."""
import time

import numpy as np
import pytest

from oracle import oracle as O
from paper_2504_19171_gb300 import workloads as W
from tests.gpu_helpers import need_gpu, rel_err, run_gpu
from tests.host_build import plan_host

POOL = [(6, 128, 1, 16), (4, 100, 1, 20), (5, 40, 2, 3)]
SLOTS = 4


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("planes", [True, False])
def test_both_sides_of_the_line(precision, planes):
    S = need_gpu()
    import torch
    ring = max(plan_host().plane_bytes(*sh, precision) for sh in POOL[:2])
    arena = 4 * SLOTS * ring - (0 if planes else 8)
    srv = S.StilesServer(POOL, arena, max_requests=SLOTS, precision=precision)
    try:
        for m, lay in enumerate(srv.layouts):
            n = srv.shape_doubles(m)[1]
            srv.set_base(m, *[torch.zeros(k, dtype=torch.float64) for k in (lay.doubles, n, n)])
        srv.start(30.0)
        mats = [W.random_arrowhead(*sh, seed=60 + m) for m, sh in enumerate(POOL)]
        got, t0 = {}, time.time()
        for m, M in enumerate(mats):
            lay = srv.layouts[m]
            assert srv.submit_values(m, lay.pack(M.tiles, np.zeros(lay.doubles)), tag=m) is not None
        while len(got) < len(POOL):
            assert time.time() - t0 < 30.0
            for r, m in srv.poll():
                out = torch.empty(srv.layouts[m].doubles, dtype=torch.float64)
                assert srv.result(r)[0] == S.STILES_OK
                srv.sigma(r, out)
                got[m] = srv.layouts[m].unpack(out.numpy())
                srv.release(r)
        assert srv.stop() == S.STILES_OK
    finally:
        srv.close()
    for m, M in enumerate(mats):
        _, Sr, _ = O.selinv(M)
        assert rel_err(got[m], Sr) < {1: 1e-12, 2: 1e-5}[precision]
        if planes or m == 2:  # (the third shape takes no planes anywhere)
            _, Sg, _, status = run_gpu(M, "fused", precision=precision)
            assert status[0] == 0 and all(np.array_equal(got[m][k], Sg[k]) for k in Sg), m
