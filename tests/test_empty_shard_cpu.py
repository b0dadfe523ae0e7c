"""sbp_boxing_shard of a destination shard that holds nothing launches nothing: every thread of such a grid would leave
before it waits for the kernel ahead of it, and the kernel behind it would then read what that one is still writing.  The
local tensors here are host memory, so that anything launched or refused shows."""
import pytest
import torch

import paper_2110_15032_b200 as sbp

F32 = torch.float32
S0, S1, B, P, PM = sbp.S(0), sbp.S(1), sbp.B, sbp.P_SUM, sbp.P_MAX


class Stream:
    cuda_stream = 0


def _host(shape, sig, k):
    return sbp.SbpTensor(shape, F32, sig, [torch.zeros(sbp.sbp_local_shape(shape, sig, k, r, F32)) for r in range(k)])


@pytest.mark.parametrize("src", [S0, S1, B, P, PM])
@pytest.mark.parametrize("ks,kd", [(3, 3), (5, 5), (2, 3), (7, 4)])
@pytest.mark.parametrize("shape", [(2, 5), (1, 900001)])
def test_empty_destination_shard(src, ks, kd, shape):
    before = sbp.sbp_launch_count()
    sbp.sbp_boxing_shard(_host(shape, src, ks), _host(shape, S0, kd), kd - 1, Stream())
    assert sbp.sbp_launch_count() == before


def test_a_shard_outside_the_placement_is_still_refused():
    with pytest.raises(sbp.SbpError):
        sbp.sbp_boxing_shard(_host((2, 5), B, 3), _host((2, 5), S0, 3), 3, Stream())
