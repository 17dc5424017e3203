"""A batch call that fails leaves the batch as it was, and one that succeeds
keeps no memory that the batch does not read."""
import numpy as np
import pytest

from gpu_helpers import DEV, cost_matrix_gpu, torch
from paper_1706_04399_gb300 import dpso, inputs

pytestmark = pytest.mark.gpu


def _fill_device():
    """Tensors that leave less than a few MB of the device free."""
    held, size = [], torch.cuda.mem_get_info()[0]
    while size >= 1 << 20:
        try:
            held.append(torch.empty(size, dtype=torch.uint8, device=DEV))
        except torch.OutOfMemoryError:
            # (from 10 MB down the allocator asks for 20 MB, or 2 MB for 1 MB at most)
            size = size // 2 if size >= 20 << 20 else (1 << 20 if size > 1 << 20 else 0)
    return held


def test_failed_autotune_keeps_the_route():
    inst = inputs.random_instance(64, 2, 31)
    C = cost_matrix_gpu(inst)
    p = dpso.default_params(swarm=60000)
    solo = dpso.Swarm(C, inst.n, inst.tags, p, 8)
    solo.step(4)
    want = solo.state()
    solo.close()
    sw = dpso.Swarm(C, inst.n, inst.tags, p, 8)
    batch = dpso.Batch([sw])
    batch.set_two_opt_shape(32, 1, 1)  # the copies that the timing reads are there
    batch.step(1)
    torch.cuda.synchronize()
    held = _fill_device()
    try:
        with pytest.raises(dpso.DpsoError) as err:
            batch.autotune()  # no room for scratch copies of 7.7 MB of tours
    finally:
        del held
        torch.cuda.empty_cache()
    assert err.value.status == dpso.ERR_NO_MEMORY
    batch.step(3)
    got = sw.state()
    for key in ("X", "V", "P", "G", "F", "PF", "history"):
        assert np.array_equal(got[key], want[key]), key
    batch.close()
    sw.close()


def test_autotune_keeps_no_copies_for_the_list_kernel():
    inst = inputs.random_instance(900, 2, 32)  # row-shifted copies of 13 MB
    C = cost_matrix_gpu(inst)
    p = dpso.default_params(swarm=64)
    free = []
    for _ in range(2):  # (the first batch loads the kernels)
        sw = dpso.Swarm(C, inst.n, inst.tags, p, 8)
        batch = dpso.Batch([sw])
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
        rows, tpc, tg = batch.autotune()
        assert rows in (32, 30, 24, 16, 8) and tpc in (1, 2, 4) and tg in (1, 2)
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
        batch.set_two_opt_shape(rows, tpc, tg)  # (the copies are made again)
        batch.step(1)
        batch.close()
        sw.close()
    # random tours, 32 moves each: the list kernel is several times faster
    assert free[3] > free[2] - (8 << 20)
