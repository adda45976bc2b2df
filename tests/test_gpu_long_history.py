"""Recorded samples of a run whose history is longer than a 2D copy's pitch can span (2^28 samples of room)."""
import contextlib

import numpy as np
import pytest

from paper_2111_13072_gb300.inputs import WORKLOADS, workload_state

pytestmark = pytest.mark.gpu

W = WORKLOADS["fp64_n2e4_l8"]


def test_samples_of_a_long_history():
    import torch
    assert torch.cuda.is_available()
    from paper_2111_13072_gb300 import build, imrp
    build.build()
    with contextlib.ExitStack() as stack:
        a, b = (stack.enter_context(imrp.Sim(imrp.params_from_workload(W, N=2000, l_max=2))) for _ in range(2))
        for s in (a, b):
            s.load(*workload_state(W, N=2000))
        q, u = a.step(6)
        # room for this many steps fits once: the batch grows the first history, refuses the second and steps neither
        many = int(0.6 * torch.cuda.mem_get_info()[0] / 16)
        assert many >= 1 << 28
        batch = imrp.Batch([a, b])
        with pytest.raises(imrp.IMRPError):
            batch.step(many)
        assert batch.failed_index() == 1
        batch.close()
        with contextlib.suppress(imrp.IMRPError):  # CUDA's record of the refused allocation
            a.sync()
        for got, want in zip(a.qdiff(0, 6), (q, u)):
            np.testing.assert_array_equal(got, want)
        a.step(2)
        np.testing.assert_array_equal(a.qdiff(0, 6)[0], q)
