"""A whole training update (every kernel with bounded waits: the segment projection, the
GEMMs, attention and its backward) after a wait of an earlier kernel gave up: its own
waits may give up, too, it ends by itself, and the next update is right again."""
import fixtures as F
import pytest
import torch

from paper_2609_35139_gb300 import cr
from test_gpu_train import _batch, _session, _step, lib  # noqa: F401

pytestmark = pytest.mark.gpu


def test_update_after_a_wait_gave_up():
    case = F.make_case("small_multi")
    a = _batch(case)

    def update(times=1):
        ts, dev, n = _session(case, a)
        for _ in range(times):
            _step(ts, dev, a, n, 1e-3)
        return ts.grads.clone()

    want = update()
    assert cr.cr_get_device_status()[0] == cr.CR_OK
    try:
        cr.cr_wait_selftest()
        update(3)
        assert cr.cr_get_device_status()[0] == cr.CR_ERR_TIMEOUT
    finally:
        cr.cr_clear_device_status()
    assert torch.equal(update(), want)
    assert cr.cr_get_device_status()[0] == cr.CR_OK
