"""The weight-gradient kernel where its blocks run several tiles one after the other and reuse their buffers:
the same gradient as with one tile per block, and the same bits every time."""
import numpy as np
import pytest

from oracle import surrogate_ref as S
from paper_2108_02419_gb300 import workloads as W
from tests.test_gpu_surrogate import assert_gradient_close, dirichlet_targets, ref_inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PER_TILE = 16  # races of 8: 128 rows, one tile


def gradient(s, rb, target, repeats=1):
    from paper_2108_02419_gb300 import bbe

    out = []
    with bbe.Batch(rb) as b:
        t = torch.from_numpy(np.ascontiguousarray(target)).cuda()
        for _ in range(repeats):
            grad = torch.empty(S.N_PARAMS, dtype=torch.float32, device="cuda")
            loss = torch.empty(1, dtype=torch.float32, device="cuda")
            bbe.bbe_surrogate_grad(s, b.handle, t, grad, loss)
            bbe.bbe_surrogate_status(s)
            out.append(grad.cpu().numpy())
    return out


@pytest.fixture()
def net():
    from paper_2108_02419_gb300 import bbe

    s = bbe.bbe_surrogate_create(0)
    bbe.bbe_surrogate_set_params(s, S.init_params(6).astype(np.float32))
    yield s
    bbe.bbe_surrogate_destroy(s)


@pytest.mark.parametrize("tiles", [75, 76, 77, 151, 152, 153, 430])
def test_gradient_of_several_tiles_a_block(net, tiles):
    rb = W.uniform_batch(seed=tiles, n_races=PER_TILE * tiles, n=8, rollouts=10)
    target = dirichlet_targets(rb, tiles)
    grads = gradient(net, rb, target, repeats=20)
    for g in grads[1:]:
        assert np.array_equal(g.view(np.uint32), grads[0].view(np.uint32))
    want = S.backward(S.init_params(6).astype(np.float32).astype(np.float64), ref_inputs(rb), rb.race_off,
                      target.astype(np.float64), bf16=True)
    assert_gradient_close(grads[0].astype(np.float64), want)


@pytest.mark.parametrize("parts", [2, 4])
def test_gradient_is_the_mean_of_one_tile_a_block(net, parts):
    """A batch of `parts` x 76 tiles against its parts of 76 tiles, which reuse no buffer on 152 SMs.  A power of
    two scales every rounding alike, so only the order of the 32-bit additions differs: an addition's
    rounding of 2^-22 of the partial sum, 32 of them a block, partial sums up to 100 times the result."""
    m = PER_TILE * 76
    rb = W.uniform_batch(seed=parts, n_races=parts * m, n=8, rollouts=10)
    target = dirichlet_targets(rb, parts)
    whole = S.unpack(gradient(net, rb, target)[0])
    each = [S.unpack(gradient(net, rb.slice(i * m, (i + 1) * m), target[8 * i * m:8 * (i + 1) * m])[0])
            for i in range(parts)]
    for name, _ in S.SHAPES[:-1]:
        mean = sum(e[name] for e in each) / parts
        assert np.abs(whole[name] - mean).max() <= 1e-3 * np.abs(mean).max(), name
