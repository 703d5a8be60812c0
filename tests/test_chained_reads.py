"""A chained step kernel starts while the kernel that writes its input still
runs (griddepcontrol). The read-only path -- __ldg, const __restrict__ kernel
arguments -- is defined only for data that nobody writes during the kernel's
life, and the compiler may move such a load above the wait: the state is read
by ordinary loads. Checked in the sources here, and on the GPU by steps that
overlap against steps that are waited for."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1411_3133_gb300", "csrc")
# the chained kernels and what they inline to read the state
READERS = {"kernels.cuh": ["step_node", "k_step", "k_step_list"],
           "pair.cuh": ["ld16", "gather_pair_far", "gather_pair_table", "step_pair", "k_step_pair", "k_step_pair_list"],
           "lbm_device.cuh": ["for_each_source_far", "gather_table", "gather_step"]}


def _definition(text, name):
    """Signature and body of device function or kernel `name`."""
    m = re.search(r"(?:void|uint32_t)(?: __launch_bounds__\([^;{]*?\))?\s+%s\(" % name, text)
    assert m, name
    i = text.index("{", m.end())
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
    return text[m.start():i], text[i:j]


@pytest.mark.parametrize("file,name", [(f, n) for f, ns in READERS.items() for n in ns])
def test_state_is_read_by_ordinary_loads(file, name):
    with open(os.path.join(CSRC, file)) as f:
        sig, body = _definition(re.sub(r"//.*", "", f.read()), name)
    assert not re.search(r"\*\s*__restrict__\s+(fin|src)\b", sig)
    for arg in re.findall(r"__ldg\(([^;]*);", body):
        assert not re.search(r"\b(fin|src|p)\b", re.sub(r"d\.src|src_", "", arg)), arg


# contexts and a batch below the groups' size: one chained launch a step, from
# one block to a few waves of them
CASES = [("cylindrical", True, (8, 1, 16), 1, "fp32"), ("cylindrical", True, (16, 4, 32), 1, "fp32"),
         ("cylindrical", True, (16, 4, 32), 1, "fp16_shifted"), ("ellipsoidal", False, (16, 4, 33), 2, "fp32"),
         ("ellipsoidal", False, (16, 3, 33), 2, "bf16_shifted"), ("cylindrical", True, (17, 3, 41), 2, "fp64"),
         ("ellipsoidal_theta", False, (9, 8, 24), 1, "fp32"), ("cylindrical", True, (48, 4, 301), 1, "fp32"),
         ("ellipsoidal", True, (48, 4, 300), 1, "fp16_shifted")]


@pytest.mark.gpu
@pytest.mark.parametrize("call", CASES, ids=lambda c: f"{c[0]}-{'x'.join(map(str, c[2]))}-b{c[3]}-{c[4]}")
@pytest.mark.parametrize("batch", [False, True], ids=["context", "batch"])
def test_overlapping_steps_are_the_waited_for_steps(call, batch):
    """Bitwise: 60 steps issued without a wait, and 60 with one after each."""
    import torch

    from gpu_helpers import lib
    from test_gpu_calls import _context, _state
    if batch and call[0] == "ellipsoidal_theta":
        pytest.skip("batches refuse the theta-resolved ellipsoid")
    L = lib()
    st = torch.cuda.Stream()
    a, b = _context(L, *call, stream=st), _context(L, *call, stream=st)
    many = L.LBBatch([a]) if batch else None
    for _ in range(60):
        many.lb_batch_step(1) if batch else a.lb_step(1)
    got = _state(a)
    for _ in range(60):
        b.lb_step(1)
        st.synchronize()
    assert np.array_equal(got, _state(b))
    if batch:
        many.close()
    a.close()
    b.close()
