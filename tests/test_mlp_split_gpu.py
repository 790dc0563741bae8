"""The network's backward pass where its split over the rows can go wrong:
one chunk and fewer, chunk edges, more chunks than a cluster has CTAs, ragged
tiles, single columns, FP32 and BF16 inputs, each output alone, and dx in
the place of x; and the Adam step on several tensors at once.

The references take the operands as the kernels do (dz and x rounded to
BF16), so the products are exact and only FP32 accumulation is left: 1e-4
relative L2, the suite's bar for FP32 outputs of exact BF16 products.  dz is
elementwise (1e-5) and db an FP32 sum of at most 4096 terms (1e-5)."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from test_mlp_gpu import dev, env, rel  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (2, 6, 256), (63, 64, 64), (64, 65, 129), (127, 256, 32), (128, 6, 31), (129, 33, 130),
          (255, 70, 1), (256, 256, 256), (257, 256, 512), (1024, 4, 128), (1025, 64, 65), (4096, 256, 256)]


def layer(torch, rows, k, n, xt, seed=0):
    rng = np.random.default_rng([rows, k, n, seed])
    x = rng.standard_normal((rows, k))
    W = M.bf16(rng.standard_normal((n, k)) / np.sqrt(k))
    z = rng.standard_normal((rows, n)).astype(np.float32)
    dy = rng.standard_normal((rows, n)).astype(np.float32)
    t = dict(x=dev(torch, x, xt), W=dev(torch, W, torch.bfloat16), z=dev(torch, z, torch.float32),
             dy=dev(torch, dy, torch.float32))
    f32 = dict(dtype=torch.float32, device="cuda")
    t.update(dz=torch.empty((rows, n), **f32), dw=torch.empty((n, k), **f32), db=torch.empty(n, **f32),
             dx=torch.empty((rows, k), **f32))
    dz, _, db, _ = M.layer_backward(M.bf16(x), z.astype(np.float64), dy.astype(np.float64), W, "gelu")
    dzb = M.bf16(dz.astype(np.float32).astype(np.float64))
    return t, dz, db, dzb.T @ M.bf16(x.astype(np.float32).astype(np.float64)), dzb @ W


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("rows,k,n", SHAPES)
def test_backward_split(env, rows, k, n, bf16):  # noqa: F811
    torch, mlp = env
    t, dz, db, dw, dx = layer(torch, rows, k, n, torch.bfloat16 if bf16 else torch.float32)
    mlp.backward(t["x"], t["z"], t["dy"], t["W"], 1, t["dz"], t["dw"], t["db"], t["dx"])
    mlp.check()
    got = {q: t[q].cpu().numpy() for q in ("dz", "db", "dw", "dx")}
    assert rel(got["dz"], dz) <= 1e-5
    assert rel(got["db"], db) <= 1e-5
    assert rel(got["dw"], dw) <= 1e-4
    assert rel(got["dx"], dx) <= 1e-4
    # each output alone, and a repeated run: the same bits
    for only in ("db", "dw", "dx"):
        for q in ("dw", "db", "dx"):
            t[q].fill_(float("nan"))
        mlp.backward(t["x"], t["z"], t["dy"], t["W"], 1, t["dz"], *[t[q] if q == only else None
                                                                    for q in ("dw", "db", "dx")])
        mlp.check()
        assert np.array_equal(t[only].cpu().numpy(), got[only])


def test_dx_in_the_place_of_x(env):  # noqa: F811
    torch, mlp = env
    t, _, _, dw, dx = layer(torch, 300, 64, 96, torch.float32)
    mlp.backward(t["x"], t["z"], t["dy"], t["W"], 1, t["dz"], t["dw"], None, t["x"])
    mlp.check()
    assert rel(t["dw"].cpu().numpy(), dw) <= 1e-4
    assert rel(t["x"].cpu().numpy(), dx) <= 1e-4


@pytest.mark.parametrize("n", [1, 8, 16, 19])
def test_adam_on_several_tensors(env, n):  # noqa: F811
    """the same bits as one tensor at a time, empty tensors among them"""
    torch, mlp = env
    rng = np.random.default_rng(n)
    sizes = [int(s) for s in rng.integers(1, 70000, n)]
    if n > 2:
        sizes[1] = 0
    f = lambda s: dev(torch, rng.standard_normal(s), torch.float32)
    w, m, v, g = ([f(s) for s in sizes] for _ in range(4))
    v = [a.abs() for a in v]
    wb = [torch.empty(s, dtype=torch.bfloat16, device="cuda") if q % 2 == 0 else None for q, s in enumerate(sizes)]
    wd = [1e-4 * (q % 3) for q in range(n)]
    one = [[a.clone() if a is not None else None for a in ts] for ts in (w, m, v, wb)]
    mlp.adam_multi(w, m, v, g, wb, 1e-3, 3, weight_decays=wd)
    for q in range(n):
        if sizes[q]:
            mlp.adam(one[0][q], one[1][q], one[2][q], g[q], one[3][q], 1e-3, 3, weight_decay=wd[q])
    torch.cuda.synchronize()
    for a, b in zip((w, m, v, wb), one):
        for x, y in zip(a, b):
            assert x is None or torch.equal(x, y)
