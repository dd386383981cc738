"""surrogate.train reports a training kernel that gave up a wait (CPU: a fake network)."""
import pytest
import torch

from paper_2303_11103_gb300 import rt
from paper_2303_11103_gb300 import surrogate as SG


class Net:
    def __init__(self, fail_at):
        self.steps, self.fail_at = 0, fail_at

    def train_step(self, x, t, lr, acc):
        self.steps += 1

    def status(self):
        return int(self.fail_at is not None and self.steps >= self.fail_at)


def test_a_step_that_timed_out_ends_the_training():
    x, t = torch.zeros(512, 6), torch.zeros(512, 2)
    net = Net(None)
    assert len(SG.train(net, x, t, epochs=3, batch=128)) == 3 and net.steps == 12
    net = Net(6)   # in the second epoch
    with pytest.raises(rt.RtError, match="RT_ERR_TIMEOUT"):
        SG.train(net, x, t, epochs=3, batch=128)
    assert net.steps == 8
