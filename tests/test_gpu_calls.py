"""What calls need around them and leave behind: device memory, other host threads' calls, stream capture."""
import threading
import time

import numpy as np
import pytest

import graphgen as gg
from oracle import deco_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2509_18612_gb300 as deco  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("precision", [deco.DECO_PREC_FP32, deco.DECO_PREC_BF16])
def test_batches_leave_no_device_memory_behind(precision):
    # the members' images of the row-vector form (some 0.6 MiB here) are kept with the batch and go with it
    members = [deco.graph_from(gg.ba_graph(900, 4, i)) for i in range(20)]
    pop = deco.population(candidates=2, rounds=1, t_lo=1, t_hi=2, e_lo=-2.5, e_hi=-1.5, lifts=(1,))

    def program(times):
        for _ in range(times):
            b = deco.deco_create_batch(members)
            deco.deco_solve_batch(b, 16, deco.params(init=deco.DECO_INIT_IDI, precision=precision), pop, 1)
            deco.deco_destroy_batch(b)
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    before = program(3)
    assert before - program(40) <= 8 << 20
