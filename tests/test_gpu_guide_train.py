"""The training kernel at the edges of its grid, and its waits (needs a GB300)."""
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


def _drawn(seed, first, count, rows):
    """SplitMix64(seed) outputs first + 1 .. first + count, mod rows."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(first + 1, first + count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z % np.uint64(rows)).astype(np.int32)


# one chunk of 64 rows, its edges, two chunks; 42 to 44 chunks (43 CTAs give each parameter a thread); more
@pytest.mark.parametrize("batch", [1, 63, 64, 65, 128, 2688, 2689, 2752, 2753, 2816])
def test_steps_are_gradient_and_adam_of_the_drawn_rows(batch):
    """Three steps against pdhgc_guide_grad (the same partial sums, so the loss bit for bit) and Adam in FP32: the
    update is at most lr / sqrt(1 - 0.999) in all, its few operations round to 2^-24 each, and so does the weight."""
    feat, lab = _data()
    lr, seed = 1e-3, 5
    net, ref = P.Guide(seed=0), P.Guide(seed=0)
    w = pack(rounded_weights(2)).astype(np.float32)
    now, m1, m2 = w, np.zeros_like(w), np.zeros_like(w)
    for k in range(3):
        net.set_weights(w)  # the run from its start: steps 0 .. k
        losses = net.train(feat, lab, rows=ROWS, batch=batch, steps=k + 1, lr=lr, seed=seed)
        ref.set_weights(now)
        grad, loss = ref.grad(feat, lab, _drawn(seed, k * batch, batch, ROWS))
        assert losses[k] == np.float32(loss)
        m1 = np.float32(0.9) * m1 + np.float32(0.1) * grad
        m2 = np.float32(0.999) * m2 + np.float32(0.001) * grad * grad
        c1, c2 = np.float32(1 / (1 - 0.9 ** (k + 1))), np.float32(1 / (1 - 0.999 ** (k + 1)))
        step = np.float32(lr) * (m1 * c1) / (np.sqrt(m2 * c2) + np.float32(1e-8))
        want, now = now - step, net.get_weights()
        tol = 2.0 ** -23 * np.abs(want).max() + 16 * 2.0 ** -24 * np.abs(step).max()
        assert np.abs(now - want).max() <= tol
    net.close()
    ref.close()


@pytest.mark.parametrize("batch", [64, 4096])
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
