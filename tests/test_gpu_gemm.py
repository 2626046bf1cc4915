"""The standalone linear and lm_head at the edges of their kernels' tiles and dispatch: one row to
several token tiles, K of one 64-wide atom to many slices, every kind of adapter rank, operands that
no tensor map can describe, ties and infinities in the read-out.  References in float64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_12422_gb300 import pbd
    pbd.load()
    return torch


def _rand(torch, g, shape, std):
    return (torch.randn(shape, generator=g, device="cuda") * std).to(torch.bfloat16)


def _linear_ref(x, W, A, B, scale):
    """(y in float64, bound): one bf16 rounding of y, fp32 sums of K products, and a rounding of each
    u to bf16 that may fall the other way."""
    y = x.double() @ W.double().T
    tol = 2e-6 * (x.double().abs() @ W.double().abs().T)
    if A is not None:
        u = (x.double() @ A.double().T).bfloat16().double()
        y = y + scale * (u @ B.double().T)
        tol = tol + abs(scale) * 2.0 ** -8 * (u.abs() @ B.double().abs().T)
    return y, tol + 2.0 ** -8 * y.abs() + 1e-7


LINEARS = [(1, 64, 128, 0), (2, 64, 128, 1), (31, 320, 256, 3), (32, 256, 128, 32), (33, 3072, 1024, 16),
           (64, 256, 128, 32), (65, 64, 128, 0), (65, 192, 256, 5), (129, 1024, 384, 8), (257, 512, 6272, 3),
           (300, 2048, 1024, 24), (1000, 320, 128, 16), (4096, 64, 128, 16), (3, 4096, 128, 16), (3, 4352, 128, 16)]


@pytest.mark.parametrize("M,K,N,r", LINEARS)
def test_linear_tile_edges(torch, M, K, N, r):
    from paper_2607_12422_gb300 import pbd
    g = torch.Generator(device="cuda").manual_seed(M + K + N + r)
    x, W = _rand(torch, g, (M, K), 1.0), _rand(torch, g, (N, K), 0.02)
    A, B = (_rand(torch, g, (r, K), 0.02), _rand(torch, g, (N, r), 0.02)) if r else (None, None)
    ref, tol = _linear_ref(x, W, A, B, 2.0)
    y = pbd.pbd_op_linear(x, W, A, B, 2.0)
    assert ((y.double() - ref).abs() <= tol).all()
    if M <= 36 or (M <= 300 and N <= 1024 and K <= 512):  # the static scratch holds these
        assert torch.equal(pbd.pbd_op_linear_static(x, W, A, B, 2.0), y)


@pytest.mark.parametrize("M", [17, 200])
def test_linear_unaligned_adapter_and_output(torch, M):
    """B and y start on odd element offsets: B has no tensor map, y takes no 32-bit stores."""
    from paper_2607_12422_gb300 import pbd
    g = torch.Generator(device="cuda").manual_seed(M)
    K, N, r = 256, 256, 16
    x, W, A = _rand(torch, g, (M, K), 1.0), _rand(torch, g, (N, K), 0.02), _rand(torch, g, (r, K), 0.02)
    B = _rand(torch, g, (N * r + 1,), 0.02)[1:].view(N, r)
    y = torch.zeros(M * N + 1, dtype=torch.bfloat16, device="cuda")
    got = pbd.pbd_op_linear_static(x, W, A, B, 2.0, y=y[1:].view(M, N))
    ref, tol = _linear_ref(x, W, A, B, 2.0)
    assert ((got.double() - ref).abs() <= tol).all() and float(y[0]) == 0.0


def test_linear_rows_do_not_depend_on_the_row_count(torch):
    from paper_2607_12422_gb300 import pbd
    g = torch.Generator(device="cuda").manual_seed(9)
    for K in (1024, 3072, 320):
        x, W = _rand(torch, g, (700, K), 1.0), _rand(torch, g, (512, K), 0.02)
        y = pbd.pbd_op_linear(x, W)
        for M in (1, 17, 64, 65, 300):
            assert torch.equal(pbd.pbd_op_linear(x[:M].contiguous(), W), y[:M]), (K, M)


@pytest.mark.parametrize("M,H,V", [(1, 64, 128), (32, 1024, 128 * 155), (33, 256, 128 * 153), (64, 1024, 2048),
                                   (65, 1024, 128 * 160), (144, 512, 4096), (256, 256, 128 * 3), (7, 2048, 1024)])
def test_lm_head_edges(torch, M, H, V):
    from paper_2607_12422_gb300 import pbd
    g = torch.Generator(device="cuda").manual_seed(M + H + V)
    x, E = _rand(torch, g, (M, H), 1.0), _rand(torch, g, (V, H), 0.02)
    # every row of E again at the far end: each maximum occurs twice, the lower id wins
    E[V // 2:] = E[:V - V // 2]
    x[0, 3] = float("inf")  # infinite logits of both signs in one row
    ids, lg = pbd.pbd_op_lm_head_argmax(x, E, want_logits=True)
    ref = x[1:].double() @ E.double().T
    assert ((lg[1:].double() - ref).abs() <= 2e-6 * (x[1:].double().abs() @ E.double().abs().T)).all()
    want = np.argmax(lg.cpu().numpy(), axis=1)  # lowest index among equal maxima
    assert not torch.isnan(lg).any() and np.array_equal(ids.cpu().numpy(), want)
    assert (want < max(V // 2, 1)).all()
    plain, none = pbd.pbd_op_lm_head_argmax(x, E)
    assert none is None and torch.equal(plain, ids)
