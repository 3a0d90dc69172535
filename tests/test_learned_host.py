"""Training sets that learned.train refuses before it touches the device (no GPU)."""
from types import SimpleNamespace

import pytest
import torch

NET = SimpleNamespace(cin=3, n=None)


@pytest.mark.parametrize("x,t,batch", [
    ((6, 3, 5), (6, 1, 3, 5), 2),              # no channel axis
    ((6, 1, 3, 4, 5), (6, 1, 4, 5), 2),        # an axis too many
    ((0, 3, 4, 5), (0, 1, 4, 5), 2),           # empty
    ((6, 3, 4, 5), (0, 1, 4, 5), 2),
    ((6, 3, 4, 5), (5, 1, 4, 5), 2),           # a target short
    ((6, 2, 4, 5), (6, 1, 4, 5), 2),           # another network's channels
    ((6, 3, 4, 5), (6, 1, 4, 5), -2),
    ((6, 3, 4, 5), (6, 1, 4, 5), 0),
])
def test_train_refuses(x, t, batch):
    from paper_1507_06767_gb300 import learned as LN

    with pytest.raises(ValueError):
        LN.train(NET, torch.zeros(x), torch.zeros(t), 1, batch, 1e-3, seed=0)


def test_train_refuses_other_types():
    from paper_1507_06767_gb300 import learned as LN

    x, t = torch.zeros((6, 3, 3, 5)), torch.zeros((6, 1, 3, 5))
    for a, b in ((x.bfloat16(), t), (x, t.bfloat16())):
        with pytest.raises(ValueError):
            LN.train(NET, a, b, 1, 2, 1e-3, seed=0)
