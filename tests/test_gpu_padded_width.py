"""Compute-heavy GEMMs of widths that 256-column tiles pad: on CTA pairs or on
128-column tiles as the waves of both and the length of the walk have it.  Against
plain fp32 products of the same bf16 inputs and stored Z and H.
"""
import pytest
import torch

from paper_2502_10940_gb300 import inputs as I

pytestmark = pytest.mark.gpu
PAIR, MSUB2 = 4, 8   # launch-trace flags: CTA pairs; two 128-row sub-tiles on one CTA


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_10940_gb300 import build
    build.build()


def _rel(got, ref):
    assert torch.isfinite(got.float()).all()
    return float((got.float() - ref).norm() / ref.norm())


# n, d_in, d_out, r, tiles of Z, Y, dZ, dX (None: not compute-heavy) and the weight gradients.  Of 76
# pairs and 152 SMs: 384 wide 2 waves to 1, then 2 to 2; 832 wide below and from K = 1024 on; 2600 wide
# 6 to 6.  Weight gradients: 142 k-block steps to 103, else less than 5/4
@pytest.mark.parametrize("n,d_in,d_out,r,zh,y,dz,dx,wgrad", [
    (12715, 2048, 2048, 384, MSUB2, None, MSUB2, None, PAIR),
    (16954, 2048, 2048, 384, PAIR, None, PAIR, None, PAIR),
    (10172, 2560, 2560, 384, MSUB2, None, MSUB2, None, MSUB2),
    (26112, 832, 1027, 832, MSUB2, PAIR, PAIR, PAIR, PAIR),
    (12019, 2600, 2600, 640, PAIR, PAIR, PAIR, PAIR, PAIR),
])
def test_tiles_of_padded_widths(n, d_in, d_out, r, zh, y, dz, dx, wgrad):
    from paper_2502_10940_gb300 import cola
    lx, ly = I.padded_ld(d_in), I.padded_ld(d_out)
    X, dY = I.normal_bf16(n, d_in, 1.0, 1, "cuda", ld=lx), I.normal_bf16(n, d_out, 1.0, 2, "cuda", ld=ly)
    A, B = I.normal_bf16(r, d_in, d_in ** -0.5, 3, "cuda", ld=lx), I.normal_bf16(d_out, r, r ** -0.5, 4, "cuda")

    def new(rows, cols):
        return torch.full((rows, I.padded_ld(cols)), float("nan"), dtype=torch.bfloat16, device="cuda")[:, :cols]

    d = cola.desc(n, d_in, d_out, r, ld_x=lx, ld_y=ly, ld_a=lx, mode="cola")
    ws = cola.workspace(d)
    Y, Z, H, dX, dA, dB = new(n, d_out), new(n, r), new(n, r), new(n, d_in), new(r, d_in), new(d_out, r)
    with cola.Trace(16) as tr:
        cola.cola_fwd(d, X, A, B, Y, Z, H, ws)
        cola.cola_bwd(d, X, A, B, dY, Z, H, dX, dA, dB, ws)
    assert cola.cola_check_status(ws) == (0, 0)
    tiles = {t[0]: t[3] & (PAIR | MSUB2) for t in tr.records()}
    for kind, want in (("fwd_zh", zh), ("fwd_y", y), ("bwd_dz", dz), ("bwd_dx", dx), ("wgrad", wgrad)):
        assert want is None or tiles[kind] == want, (kind, tr.records())
    f = torch.Tensor.float
    # one bf16 rounding (1.1e-3 as a whole) for Z and Y, two to three chained ones for the others
    assert _rel(Z, f(X) @ f(A).T) < 3e-3
    assert _rel(Y, f(H) @ f(B).T) < 3e-3
    s = torch.sigmoid(f(Z))
    dZ = (f(dY) @ f(B)) * (s * (1 + f(Z) * (1 - s)))
    assert _rel(dX, dZ @ f(A)) < 5e-3
    assert _rel(dA, dZ.T @ f(X)) < 5e-3
    assert _rel(dB, f(dY).T @ f(H)) < 5e-3
    for t in (Y, dX):
        assert torch.as_strided(t, (n, t.stride(0)), (t.stride(0), 1))[:, t.shape[1]:].isnan().all()


# 128-column tiles would run unsplit in one wave (71 k-block steps), 256-column ones split three ways take 47
def test_weight_gradients_split_where_wide_tiles_take_far_fewer_steps():
    from paper_2502_10940_gb300 import cola
    n, d_in, d_out, r = 4500, 456, 4584, 192
    X, dY = I.normal_bf16(n, d_in, 1.0, 1, "cuda"), I.normal_bf16(n, d_out, 1.0, 2, "cuda")
    A, B = I.normal_bf16(r, d_in, d_in ** -0.5, 3, "cuda"), I.normal_bf16(d_out, r, r ** -0.5, 4, "cuda")
    Z, H = I.normal_bf16(n, r, 1.0, 5, "cuda"), I.normal_bf16(n, r, 1.0, 6, "cuda")
    d = cola.desc(n, d_in, d_out, r, sigma="identity", mode="cola")
    ws = cola.workspace(d)
    dX, dA, dB = torch.empty_like(X), torch.empty_like(A), torch.empty_like(B)
    with cola.Trace(16) as tr:
        cola.cola_bwd(d, X, A, B, dY, Z, H, dX, dA, dB, ws)
    assert [t[2] for t in tr.records() if t[0] == "wgrad"] == [3], tr.records()
    f = torch.Tensor.float
    assert _rel(dB, f(dY).T @ f(H)) < 3e-3                     # one bf16 rounding
    assert _rel(dA, (f(dY) @ f(B)).T @ f(X)) < 5e-3            # and dZ's
