"""Chains of block products without a synchronisation between them: each reads
the rows of X that the launch before it packed from the result of the one before
that, while its CTAs start early.  Against the CPU oracle, single and batched."""
import numpy as np
import pytest

import gen
import oracle
from helpers import rand_block, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,nvec", [(65521, 16), (251, 5), (2**31 - 1, 7), (2**32 - 5, 16)])
@pytest.mark.parametrize("batched", [False, True])
def test_chain_of_products(lib, m, nvec, batched):
    import torch
    n, steps = 3001, 24
    rng = np.random.default_rng(m % 997)
    lengths = rng.integers(0, 12, n)
    lengths[5] = 1700
    A = gen.uniform_matrix(3, n, n, lengths, m, pm_fraction=0.2)
    M = lib.Matrix.from_csr(A, transpose_mode=lib.TRANSPOSE.NONE)
    M.launches(False, nvec)      # the layout is there
    x = rand_block(9, n, nvec, m)
    want = x
    for _ in range(steps):
        want = oracle.csr_spmv(A, want)
    for _ in range(3):
        bufs = [to_dev(x), torch.zeros((n, nvec), dtype=torch.int32, device="cuda")]
        for i in range(steps):
            if batched:
                lib.spmv_batch_apply([M.handle], [bufs[i & 1]], [bufs[~i & 1]], [nvec])
            else:
                M.apply(bufs[i & 1], bufs[~i & 1])
        assert np.array_equal(to_host(bufs[steps & 1]), want)
