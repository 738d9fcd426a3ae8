"""The far field's device buffers come as one allocation: a fit is refused whole, with nothing
left allocated, or granted whole; a refit takes over the former far field's allocation (while a map
of that one is still queued on another stream), or gives it back where it is far too large."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

import workloads as W  # noqa: E402
from gpu_util import make_ctx  # noqa: E402
from paper_1703_09707_gb300 import mlens as M  # noqa: E402

RAYS = W.Grid(-4.0, 4.0, -2.0, 2.0, 512, 256)


@pytest.mark.parametrize("net,batch", [(0, 128), (1, 1000), (1, 1 << 20)])
def test_fit_is_refused_or_granted_whole(net, batch):
    f = W.config("tiny").fields[0]
    par = M.fit_params(cells_x=8, order=10, use_network=net, train_samples=3000, epochs=1, batch=batch, tolerance=1.0)
    ctx, other = make_ctx(f), make_ctx(f)
    try:
        before = M.mlens_device_memory_in_use()
        M.mlens_fit_far_field(ctx, RAYS, par)
        need = M.mlens_device_memory_in_use() - before
        M.mlens_set_device_memory_limit(before + need)
        M.mlens_fit_far_field(ctx, RAYS, par)
        assert M.mlens_device_memory_in_use() == before + need
        ctx.close()
        before = M.mlens_device_memory_in_use()
        M.mlens_set_device_memory_limit(before + need - 1)
        with pytest.raises(M.MlensError) as ei:
            M.mlens_fit_far_field(other, RAYS, par)
        assert ei.value.code == M.MLENS_ERR_NOMEM
        assert M.mlens_device_memory_in_use() == before
    finally:
        M.mlens_set_device_memory_limit(0)
        ctx.close()
        other.close()


def test_refit_takes_over_the_allocation():
    f = W.random_field(5, 4000, 0.4, 0.1, 0.2, 0.0)
    big, small = W.Grid(-4.0, 4.0, -2.0, 2.0, 4096, 2048), W.Grid(-4.0, 4.0, -2.0, 2.0, 512, 256)
    src = W.Grid(-2.0, 2.0, -2.0, 2.0, 64, 64)
    par = [M.fit_params(cells_x=8, order=o, use_network=0, tolerance=1.0) for o in (10, 6)]

    def shot(c, stream=None):
        out = torch.empty(src.n, dtype=torch.int32, device="cuda")
        M.mlens_shoot_learned(c, big, src, out, stream=stream)
        return out

    fresh = []
    for p in par:
        ctx = make_ctx(f)
        M.mlens_fit_far_field(ctx, big, p)
        fresh.append(shot(ctx))
        torch.cuda.synchronize()
        used = M.mlens_device_memory_in_use()
        ctx.close()
    empty = M.mlens_device_memory_in_use()
    ctx, s = make_ctx(f), torch.cuda.Stream()
    M.mlens_fit_far_field(ctx, big, par[0])
    with torch.cuda.stream(s):
        maps = [shot(ctx, s) for _ in range(8)]
    M.mlens_fit_far_field(ctx, big, par[1])  # on the current stream
    assert M.mlens_device_memory_in_use() == used
    last = shot(ctx)
    torch.cuda.synchronize()
    assert all(torch.equal(m, fresh[0]) for m in maps) and torch.equal(last, fresh[1])
    M.mlens_fit_far_field(ctx, small, par[0])
    assert M.mlens_device_memory_in_use() - empty < (used - empty) // 2
    with pytest.raises(M.MlensError):
        M.mlens_fit_far_field(ctx, W.Grid(-4.0, 4.0, -2.0, 2.0, 500, 256), par[0])  # no whole tiles per cell
    ctx.close()
    assert M.mlens_device_memory_in_use() == empty
