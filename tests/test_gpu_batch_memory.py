"""Batches whose room for tensor-core operands is cut down because memory is short: the same states, and
the next calls keep the room and the captured graphs."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fails", [1, 3, 20])      # half the room, an eighth, one operand at a time
def test_a_smaller_room_is_kept(gpu, fails):
    import torch
    sv = gpu
    n, count = 13, 6
    fam = [W.hea(n, 3, seed=60 + i) for i in range(count)]
    circs = [sv.sv_fuse(sv.gates_from_specs(f), n, 5) for f in fam]
    ngates = sv.sv_circuit_size(circs[0])[0]
    states = []
    for short in (False, True):
        b = sv.sv_batch_alloc(n, 0, count, stream=torch.cuda.current_stream())
        if short:
            most = int(np.log2(count * ngates))   # the room for one operand has to be granted
            sv.sv_debug_fail_allocs(min(fails, most))
        reused = []
        for _ in range(3):
            sv.sv_batch_set_basis(b, 1)
            reused.append(sv.sv_batch_apply(b, circs)["graph_reused"])
        sv.sv_debug_fail_allocs(0)
        assert reused == [0, 1, 1]
        states.append([sv.sv_batch_get_state(b, i) for i in range(count)])
        b.free()
    assert all(np.array_equal(p, q) for p, q in zip(*states))
