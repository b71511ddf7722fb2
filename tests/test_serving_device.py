"""The serving loop runs its calls with its own device current, whatever the caller's is.  A stand-in for the loop and for
torch's device calls: nothing is launched."""
import contextlib
import types

import pytest
import torch

from paper_2608_14205_b200 import serving as S


@pytest.mark.parametrize("callers", [0, 1, 2])
def test_methods_run_on_the_loops_device(monkeypatch, callers):
    current = [callers]

    @contextlib.contextmanager
    def device(d):
        before, current[0] = current[0], d.index
        yield
        current[0] = before

    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: current[0], raising=False)
    monkeypatch.setattr(torch.cuda, "device", device)
    seen = []
    loop = types.SimpleNamespace(dev=torch.device("cuda", 1))
    run = S._on_its_device(lambda self, a, b=0: seen.append((current[0], a, b)) or a + b)
    assert run(loop, 2, b=3) == 5
    assert seen == [(1, 2, 3)] and current == [callers]


def test_the_loops_entry_points_are_wrapped():
    for name in ("layer_step", "realised_loads"):
        assert hasattr(getattr(S.ServingLoop, name), "__wrapped__"), name
