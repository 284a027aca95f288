"""The MLP kernels at the edges of the batch and of the alignment (16-byte
loads against single ones), against the numpy reference with the tolerance
of the other MLP tests, and the two load forms against each other bit for
bit (the same arithmetic in the same order)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp  # noqa: E402
from paper_2303_10581_gb300 import learned  # noqa: E402

pytestmark = pytest.mark.gpu


def at_offset(a, shift):
    """A contiguous device copy starting `shift` floats past a 256-byte boundary."""
    buf = torch.zeros(a.size + shift, dtype=torch.float32, device="cuda")
    buf[shift:] = torch.from_numpy(a.ravel()).cuda()
    return buf[shift:].view(a.shape)


def step(B, shift):
    rng = np.random.default_rng(B)
    prop = learned.Proposal(seed=B)
    X = (rng.uniform(0, 1, (B, 1024)) / 30).astype(np.float32)
    label = rng.integers(0, 4, B).astype(np.int32)
    off = rng.uniform(-0.4, 0.4, (B, 64)).astype(np.float32)
    mask = (rng.uniform(0, 1, B) > 0.25).astype(np.float32)
    p0 = prop.params.float().cpu().numpy()
    Xd = at_offset(X, shift)
    out = prop.forward(Xd).cpu().numpy()
    loss = prop.train_step(Xd, torch.from_numpy(label).cuda(), torch.from_numpy(off).cuda(),
                           torch.from_numpy(mask).cuda(), lam=0.5, lr=1e-3).cpu().numpy()
    ref_loss, g = mlp.grads(X, p0, label, off, mask, 0.5)
    assert np.allclose(out, mlp.forward(X, p0)[2], rtol=1e-4, atol=1e-5)
    assert np.allclose(loss, ref_loss, rtol=1e-4, atol=1e-5)
    m = prop.m.cpu().numpy()   # a first step's first moment is 0.1 of the gradient
    assert np.allclose(m, 0.1 * g, rtol=1e-4, atol=1e-7)
    return out, loss, m, prop.master.cpu().numpy()


@pytest.mark.parametrize("B", [1, 2, 31, 64, 65])
def test_batch_and_alignment(B):
    for a, b in zip(step(B, 0), step(B, 1)):
        assert np.array_equal(a, b)
