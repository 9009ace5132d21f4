"""Calls that end in an error leave none of their memory behind."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_a_refused_training_gives_its_memory_back():
    import paper_1404_0812_gb300 as R
    net = R.EpsNet(11)
    X, y = torch.zeros(5000, 33, device="cuda"), torch.zeros(5000, device="cuda")
    net.train(X[:64], y[:64], epochs=1, batch=64)
    torch.cuda.synchronize()
    used = R.memory_stats()["used"]
    for _ in range(3):
        with pytest.raises(R.RbffdError) as e:   # more than 4096 batches
            net.train(X, y, epochs=1, batch=1)
        assert e.value.status == 1
    torch.cuda.synchronize()
    assert R.memory_stats()["used"] == used
