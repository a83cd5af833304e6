"""The training kernel's waits (needs a GB300)."""
import numpy as np
import pytest

from tests.test_gpu_guide import _random_inputs, feat_tensor, pack, rounded_weights

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2511_13894_gb300.pdhgc")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ROWS = 3000


def _data():
    F, lab = _random_inputs(ROWS, 11)
    return feat_tensor(F)[0], torch.as_tensor(np.asarray(lab).astype(np.uint8)).cuda()


@pytest.mark.parametrize("batch", [4096])
def test_training_wait_that_gives_up_reports_device_error(batch):
    """The grid waits give up at once: DEVICE, and with the weights set again a run gives its usual bits."""
    feat, lab = _data()
    g = P.Guide(seed=0)
    w = pack(rounded_weights(2))

    def train():
        g.set_weights(w)
        return g.train(feat, lab, rows=ROWS, batch=batch, steps=20, lr=1e-3, seed=5), g.get_weights()
    losses, trained = train()
    g.set_wait_limit(0)
    with pytest.raises(P.PdhgcError) as e:
        train()
    assert e.value.code == -10
    g.set_wait_limit(1 << 24)
    again, trained_again = train()
    assert np.array_equal(again, losses) and np.array_equal(trained_again, trained)
    g.close()
