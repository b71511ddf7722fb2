"""The serving loop makes its calls with its own device current, whatever the caller's is.  Stand-ins for the loop's parts
and for torch's device calls: nothing is launched."""
import contextlib
import types

import pytest
import torch

from paper_2608_14205_b200 import serving as S


@pytest.mark.parametrize("callers", [0, 1, 2])
@pytest.mark.parametrize("entry", ["layer_step", "realised_loads"])
def test_entry_points_run_on_the_loops_device(monkeypatch, callers, entry):
    current = [callers]

    @contextlib.contextmanager
    def device(index):
        before, current[0] = current[0], index
        yield
        current[0] = before

    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: current[0], raising=False)
    monkeypatch.setattr(torch.cuda, "device", device)

    class Reached(Exception):
        pass

    class Parts:                                             # the first thing the loop touches tells where it runs
        def __getattr__(self, name):
            raise Reached(current[0])

    loop = S.ServingLoop.__new__(S.ServingLoop)
    loop.device, loop.dev, loop.out, loop.ctx, loop.wl = 1, torch.device("cuda", 1), {}, Parts(), Parts()
    loop.placement, loop._spare = {0: None}, None
    x = types.SimpleNamespace(shape=(4, 8))
    args = (0, None, x, x, None, True) if entry == "layer_step" else ({}, None)
    loop._q = {}
    with pytest.raises(Reached) as seen:
        getattr(loop, entry)(*args)
    assert seen.value.args == (1,)
