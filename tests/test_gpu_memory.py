"""Device memory a simulator holds."""
import pytest
import torch

import workloads as wl

pytestmark = pytest.mark.gpu


def test_floating_base_holds_one_tape_buffer():
    """The link-frame tape (119 words a link) and the pipelined adjoint's tapes (3 x 38 a link
    and 3 x 43 a system) share a buffer, beside 32 + 1 words of constants, 71 of the adjoint
    record, a mass gradient and the link map a link, four stacks of one 27-word entry and
    four words a system.  Counted as what destroying the simulator gives back."""
    from paper_2109_07719_gb300 import Simulator
    B, n = 40960, 13
    w = wl.quadruped(B=B, T=1, precision="fp32")
    sim = Simulator(w.model, precision="fp32")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    del sim
    held = torch.cuda.mem_get_info()[0] - before
    words = max(119 * n, 3 * (38 * n + 43)) + (33 + 71 + 1 + 1) * n + 4 * 27 + 4
    assert held < 4 * words * B + (32 << 20), (held, 4 * words * B)   # and 32 MiB for the allocator's rounding
