"""Forward passes of a handful of tokens (the thin kernels): token counts around
the multiples of 16 the MMA rounds up to and around the largest count, ragged
weight tiles and k-blocks, one to three projections, the gated product, every
mode, and both sides of the lines above which Y and the gated product take the
token-major GEMMs.  Against plain fp32 products of the same bf16 inputs and stored H.
"""
import pytest
import torch

from paper_2502_10940_gb300 import inputs as I

pytestmark = pytest.mark.gpu
CLUSTER = 128   # launch-trace flag: K splits reduced inside a cluster


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_10940_gb300 import build
    build.build()


def _wide(n, cols):
    ld = I.padded_ld(cols)
    return torch.full((n, ld), float("nan"), dtype=torch.bfloat16, device="cuda")[:, :cols]


def _padding_intact(t):
    ld = t.stride(0)
    return bool(torch.as_strided(t, (t.shape[0], ld), (ld, 1))[:, t.shape[1]:].isnan().all())


def _close(got, ref):
    # one bf16 rounding as a whole (2^-9 / sqrt(3) = 1.1e-3), and per element
    # half an ulp of the value plus the noise of the fp32 sums
    got = got.float()
    assert torch.isfinite(got).all()
    assert (got - ref).norm() / ref.norm() < 3e-3
    assert bool(((got - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-3).all())


def _sigma(name, z):
    z = z.float()
    return {"silu": torch.nn.functional.silu, "gelu": torch.nn.functional.gelu, "identity": lambda t: t}[name](z)


def _y_is_thin(n, r):
    return n <= 32 or r >= (512 if n <= 48 else 1024)


# n, d_in, d_out, r, projections (3008 wide: 15 tiles of Z, more than the clusters of 16 that run at once)
SHAPES = [(1, 64, 64, 192, 1), (1, 4096, 4096, 1024, 3), (2, 72, 100, 64, 2), (15, 333, 91, 192, 1), (16, 520, 130, 320, 1),
          (17, 1000, 3000, 192, 3), (32, 136, 520, 64, 3), (33, 2048, 5461, 512, 2), (63, 5461, 2048, 512, 1), (64, 1027, 257, 256, 3),
          (64, 4096, 11008, 1024, 1), (20, 3008, 200, 640, 3), (48, 640, 390, 384, 2), (48, 640, 390, 512, 2), (49, 640, 390, 960, 2)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("sigma", ["silu", "gelu", "identity"])
def test_thin_forward(shape, sigma):
    from paper_2502_10940_gb300 import cola
    n, d_in, d_out, r, c = shape
    X = I.normal_bf16(n, d_in, 1.0, 1, "cuda", ld=I.padded_ld(d_in))
    A = I.normal_bf16(c * r, d_in, d_in ** -0.5, 2, "cuda", ld=I.padded_ld(d_in))
    B = [I.normal_bf16(d_out, r, r ** -0.5, 3 + j, "cuda") for j in range(c)]
    outs = {}
    for mode in ("cola", "cola_m", "infer"):
        d = cola.desc(n, d_in, d_out, r, ld_x=cola.ld_of(X), ld_y=I.padded_ld(d_out), ld_a=cola.ld_of(A), sigma=sigma, mode=mode)
        ws = cola.workspace(d, c)
        Y = [_wide(n, d_out) for _ in range(c)]
        Z = _wide(n, c * r) if mode != "infer" else None
        H = _wide(n, c * r) if mode == "cola" else None
        with cola.Trace(8) as tr:
            if c == 1:
                cola.cola_fwd(d, X, A, B[0], Y[0], Z, H, ws)
            else:
                cola.cola_fwd_shared_x(d, X, A, B, Y, Z, H, ws)
        rec = [(t[0], t[3] & CLUSTER) for t in tr.records()]
        assert rec == [("fwd_zh", CLUSTER), ("fwd_y", CLUSTER if _y_is_thin(n, r) else 0)], tr.records()
        assert c * r <= 14 * 128 or tr.records()[0][2] <= 13
        assert cola.cola_check_status(ws) == (0, 0)
        assert all(_padding_intact(y) for y in Y)
        outs[mode] = (Y, Z, H)
        if mode == "cola_m":   # the recompute gives the forward's Y bit for bit
            Yr = [_wide(n, d_out) for _ in range(c)]
            cola.cola_recompute_up(d, Z, B, Yr, ws)
            assert all(torch.equal(a, b) for a, b in zip(Y, Yr))
    Y, Z, H = outs["cola"]
    _close(Z, X.float() @ A.float().T)
    assert ((H.float() - _sigma(sigma, Z)).norm() / H.float().norm()) < 3e-3
    for j in range(c):
        _close(Y[j], H[:, j * r:(j + 1) * r].float() @ B[j].float().T)
        assert torch.equal(Y[j], outs["cola_m"][0][j]) and torch.equal(Y[j], outs["infer"][0][j])
    assert torch.equal(Z, outs["cola_m"][1])


@pytest.mark.parametrize("n,d,d_ff,r", [(1, 64, 65, 64), (5, 200, 328, 128), (16, 333, 91, 192), (32, 2048, 5461, 512),
                                        (64, 1000, 2999, 256), (64, 4096, 11008, 1024), (31, 496, 1034, 128),
                                        (48, 256, 4096, 512), (48, 256, 4100, 512), (33, 256, 9215, 640), (64, 256, 6143, 1024),
                                        (50, 256, 6145, 1024)])
def test_thin_gated_product(n, d, d_ff, r):
    from paper_2502_10940_gb300 import cola
    X = I.normal_bf16(n, d, 1.0, 1, "cuda", ld=I.padded_ld(d))
    A = I.normal_bf16(2 * r, d, d ** -0.5, 2, "cuda", ld=I.padded_ld(d))
    B = [I.normal_bf16(d_ff, r, r ** -0.5, 3 + j, "cuda") for j in range(2)]
    M, Mi, Yg, Yu = (_wide(n, d_ff) for _ in range(4))
    Z, H = _wide(n, 2 * r), _wide(n, 2 * r)
    dd = cola.desc(n, d, d_ff, r, ld_x=cola.ld_of(X), ld_y=I.padded_ld(d_ff), ld_a=cola.ld_of(A), mode="cola")
    ws = cola.workspace(dd, 2)
    with cola.Trace(8) as tr:
        cola.cola_fwd_gate_up(dd, X, A, B[0], B[1], M, Yg, Yu, Z, H, ws)
    tiles = (d_ff + 127) // 128
    thin = n <= 32 or (r >= 1024 and tiles <= 48 if n > 48 else tiles <= (72 if r >= 640 else 32 if r >= 320 else 0))
    assert [(t[0], t[3] & CLUSTER) for t in tr.records()] == [("fwd_zh", CLUSTER), ("fwd_glu", CLUSTER if thin else 0)], tr.records()
    assert cola.cola_check_status(ws) == (0, 0)
    for j, Y in enumerate((Yg, Yu)):
        _close(Y, H[:, j * r:(j + 1) * r].float() @ B[j].float().T)
    assert torch.equal(M, (Yg.float() * Yu.float()).to(torch.bfloat16))
    di = cola.desc(n, d, d_ff, r, ld_x=cola.ld_of(X), ld_y=I.padded_ld(d_ff), ld_a=cola.ld_of(A), mode="infer")
    wi = cola.workspace(di, 2)
    cola.cola_fwd_gate_up(di, X, A, B[0], B[1], Mi, None, None, None, None, wi)
    assert torch.equal(M, Mi) and all(_padding_intact(t) for t in (M, Mi, Yg, Yu))
