"""The planner's training kernels at batch sizes around their splits (16 samples
a block, 512 lanes over the batch) and with buffers off 16-byte alignment,
against float64.

Bounds: a float32 sum of n products errs by at most (n + 2) 2^-24 of the sum of
the products' magnitudes A; the longest here are 64 products a unit, two layers
deep, and for the gradients the lanes' sums of B / 512 products and 21 more
additions, with factors that carry the layers' errors: 1e-5 A covers all."""
import numpy as np
import pytest

from oracle import planner as PL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2609_03613_gb300 import tilegs as G  # noqa: E402


def off_alignment(a):
    """A device copy starting 4 bytes past a 16-byte boundary."""
    buf = torch.empty(a.size + 1, dtype=torch.float32, device="cuda")
    v = buf[1:].view(a.shape)
    v.copy_(torch.from_numpy(a))
    return v


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("B", [1, 15, 16, 17, 511, 512, 513, 4099])
def test_mlp_batch_sizes_match_float64(B, aligned):
    rng = np.random.default_rng(B)
    F, H, C = G.PLAN_FEATURES, G.PLAN_HIDDEN, G.PLAN_CLASSES
    X = rng.normal(0.0, 1.5, (B, F)).astype(np.float32)
    P = rng.normal(0.0, 0.25, G.PLAN_PARAMS).astype(np.float32)
    dz = (rng.normal(0.0, 1.0, (B, C)) / B).astype(np.float32)
    put = (lambda a: torch.from_numpy(a).cuda()) if aligned else off_alignment
    Xd, Pd, dzd = put(X), put(P), put(dz)
    acts, logits = G.mlp_forward(Pd, Xd)
    grads = G.mlp_backward(Pd, Xd, acts if aligned else put(acts.cpu().numpy()), dzd,
                           deltas=put(np.zeros((B, 2 * H), np.float32)))
    h1, h2, z = PL.forward(P.astype(np.float64), X.astype(np.float64))
    np.testing.assert_allclose(acts.cpu().numpy(), np.concatenate([h1, h2], 1), rtol=1e-5, atol=1e-5)
    np.testing.assert_allclose(logits.cpu().numpy(), z, rtol=1e-5, atol=1e-5)
    # the deltas from the kernel's own activations: a unit within rounding of
    # its ReLU's corner may be on either side in float64
    a = acts.cpu().numpy().astype(np.float64)
    h1, h2, Pd64, X64, dz64 = a[:, :H], a[:, H:], P.astype(np.float64), X.astype(np.float64), dz.astype(np.float64)
    ref = PL.backward(Pd64, X64, h1, h2, dz64)
    A = PL.backward(np.abs(Pd64), np.abs(X64), h1, h2, np.abs(dz64))
    g = grads.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - ref) <= 1e-5 * A + 1e-12)
    again = G.mlp_backward(Pd, Xd, acts if aligned else put(acts.cpu().numpy()), dzd)
    assert torch.equal(grads, again)  # the sums meet in a fixed order
