"""Slots of shared-out entries are given up only where a request would not
run beside them at all (no GPU)."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2503_09184_gb300.serving import Request, serve

CT, EXT = 100, 10


class Executor:
    reserved_bytes = 5000

    def whole_entries(self):
        self.reserved_bytes = 1000

    def admit(self, req):
        pass

    def release(self, req):
        pass

    def run_wave(self, blocks):
        return 1


# a dense 2 x 3 request of 4 columns: A takes 660 bytes, a column 530
@pytest.mark.parametrize("room,reserved,done", [(5000 + 660 + 530, 5000, 1), (5000 + 660 + 529, 1000, 1),
                                                (1000 + 660 + 530, 1000, 1), (1000 + 660 + 529, 1000, 0)])
def test_slots_are_given_up_for_a_request_that_would_be_rejected(room, reserved, done):
    req = Request(0, np.ones((2, 3), np.int64), np.ones((3, 4), np.int64))
    ex = Executor()
    out = serve([req], ex, room, wave_products=8, ct_bytes=CT, ext_bytes=EXT)
    assert out["done"] == done and ex.reserved_bytes == reserved
