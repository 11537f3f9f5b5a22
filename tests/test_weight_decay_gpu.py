"""Weight decay of the cost model's training: one rule for train() and for a
loop of Trainer.epoch calls, none unless it is asked for."""
import numpy as np
import pytest

from paper_1706_10086_gb300 import inputs, tuning

pytestmark = pytest.mark.gpu


def small_set(n=60, C=11):
    sh = inputs.shapes(47, n, 64, 16384)
    return {"M": sh[:, 0], "N": sh[:, 1], "K": sh[:, 2], "path": np.arange(n, dtype=np.int32) % 2,
            "T": np.abs(inputs.uniform(48, 0, (n, C))).astype(np.float32),
            "Mask": (inputs.uniform(49, 0, (n, C)) > -0.5).astype(np.float32), "C": C}


@pytest.mark.parametrize("decay", [0.0, 0.5, 3.0])
def test_epoch_decays_after_adam(alp, decay):
    plain, decayed = tuning.Trainer(small_set()), tuning.Trainer(small_set())
    lr = 3e-3
    plain.epoch(lr)
    decayed.epoch(lr, decay)
    want = plain.params * (1.0 - lr * decay) if decay else plain.params
    assert np.array_equal(decayed.params.cpu().numpy(), want.cpu().numpy())
    assert np.array_equal(decayed.m.cpu().numpy(), plain.m.cpu().numpy())


def test_train_is_the_loop_of_epochs(alp):
    (params, mean, std), _ = tuning.train(small_set(), epochs=20, lr=3e-3)
    tr = tuning.Trainer(small_set())
    for e in range(20):
        tr.epoch(3e-3 if e < 14 else 3e-4, tuning.WEIGHT_DECAY)
    for got, want in zip((params, mean, std), tr.model()):
        assert np.array_equal(got, want)
