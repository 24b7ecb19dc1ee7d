"""The training workspaces that a Refiner keeps are bounded over many batch sizes.
On the host, with stand-ins for the library's size query and for device memory."""
import pytest

from paper_2608_02438_gb300 import binding as X


class Torch:
    uint8 = None

    class empty:
        def __init__(self, size, dtype=None, device=None):
            self.size = size

        def data_ptr(self):
            return 768

        def numel(self):
            return self.size


def train_size(b):
    return (b << 20) + (b % 3 << 18)                             # not always growing with b


@pytest.fixture()
def refiner(monkeypatch):
    monkeypatch.setattr(X, "xpress_train_workspace_size", lambda handle, b, B: train_size(b))
    monkeypatch.setattr(X, "xpress_refine_workspace_size", lambda handle, b: b << 20)
    r = object.__new__(X.Refiner)
    r.handle, r.B, r._ws, r.torch = None, 16, {}, Torch
    return r


def test_training_workspaces_of_many_batch_sizes(refiner):
    for b in range(1, 513):
        _, size = refiner.workspace("train", b)
        assert train_size(b) <= size                             # every batch fits its workspace,
        assert size - 256 <= (b << 20) * 9 / 8 + (2 << 18)       # which is for an eighth more at most
    assert sum(buf.numel() for buf in refiner._ws.values()) < 13 * (512 << 20)


def test_powers_of_two_and_small_batches_have_their_own_size(refiner):
    for b in (*range(1, 17), 32, 64, 128, 256, 512):
        assert refiner.train_workspace_sizes(b)[-1] == b
    assert refiner.workspace("train", 16)[1] == train_size(16) + 256


def test_other_workspaces_are_per_batch_size(refiner):
    for b in (32, 33, 34):
        assert refiner.workspace("refine", b)[1] == (b << 20) + 256
    assert len(refiner._ws) == 3
