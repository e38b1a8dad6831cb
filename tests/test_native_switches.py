"""The switch and the step size of the Python calls take whatever int() and float() take (no GPU, no library call)."""
import numpy as np
import pytest
import torch

from test_native_calls import calls  # noqa: F401  (a fixture)


@pytest.mark.parametrize("on", [True, 1, 1.0, np.bool_(True), np.int64(1), np.array(True), torch.tensor(True), torch.tensor(1.0)])
def test_per_block(calls, on):  # noqa: F811
    n, seen = calls
    g, t = torch.zeros(24), torch.zeros(8, dtype=torch.int32)
    n.amplitudes(g, 20, t, None, 2.0, 3.0, 10, on, t, None)
    n.encode_dev(g, 20, t, t, 1, 2, 0, 10, on, None, None)
    n.server_aggregate_dev(t, 20, g, t, 1, 2, None, 0, 3, t, 1, t, 10, on, None)
    n.downlink_decode_dev(t, 20, g, t, 1, 2, 1, 10, on, None)
    n.downlink_encode(g, 20, t, t, 1, 2, 1, 10, on, None)
    n.downlink_apply(t, 20, g, t, 1, 2, 0.5, 1, 10, on, None)
    place = {"fosgd_amplitudes": 8, "fosgd_encode_dev": 9, "fosgd_server_aggregate_dev": 9, "fosgd_downlink_decode_dev": 5,
             "fosgd_downlink_encode": 6, "fosgd_downlink_apply": 6}
    assert [name for name, _ in seen] == list(place)
    assert all(a[place[name]] == 1 for name, a in seen)


@pytest.mark.parametrize("step", [0.5, np.float32(0.5), np.array(0.5), torch.tensor(0.5), "0.5"])
def test_step_size(calls, step):  # noqa: F811
    n, seen = calls
    t = torch.zeros(8, dtype=torch.int32)
    n.downlink_apply(t, 20, t, 0.25, 1, 2, step, 1, 0, False, None)
    assert seen[-1][1][4] == 0.25 and seen[-1][1][9] == 0.5


def test_what_neither_takes_is_refused_before_the_call(calls):  # noqa: F811
    n, seen = calls
    t = torch.zeros(8, dtype=torch.int32)
    for step, on in ((None, False), (0.5, None), ("x", False), (0.5, "x")):
        with pytest.raises((TypeError, ValueError)):
            n.downlink_apply(t, 20, t, 0.25, 1, 2, step, 1, 0, on, None)
    assert not seen
