"""The product epilogue at the edges of its 64-column chunks, on single CTAs and
on CTA pairs with either ring length: Y_gate, Y_up against a plain fp32 product
of the same stored H, M bit for bit bf16(Y_gate * Y_up), the inference M equal.
"""
import pytest
import torch

from paper_2502_10940_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_10940_gb300 import build
    build.build()


@pytest.mark.parametrize("n,d_ff,r,pair", [
    (1, 65, 64, False), (129, 64, 128, False), (300, 127, 128, False), (257, 328, 64, False),
    (4360, 4033, 512, True), (4231, 4096, 512, True), (4360, 4095, 960, True),
    (2184, 4033, 1024, True), (2177, 4160, 1024, True),
])
def test_product_chunk_edges(n, d_ff, r, pair):
    from paper_2502_10940_gb300 import cola
    d, ld = 136, I.padded_ld(d_ff)

    def wide():
        return torch.full((n, ld), float("nan"), dtype=torch.bfloat16, device="cuda")[:, :d_ff]

    X, A = I.normal_bf16(n, d, 1.0, 1, "cuda"), I.normal_bf16(2 * r, d, d ** -0.5, 2, "cuda")
    B = [I.normal_bf16(d_ff, r, r ** -0.5, 3 + j, "cuda") for j in range(2)]
    M, Mi, Yg, Yu = (wide() for _ in range(4))
    Z, H = (torch.empty((n, 2 * r), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    dd = cola.desc(n, d, d_ff, r, ld_y=ld, mode="cola")
    ws = cola.workspace(dd, 2)
    with cola.Trace(8) as tr:
        cola.cola_fwd_gate_up(dd, X, A, B[0], B[1], M, Yg, Yu, Z, H, ws)
    rec = tr.records()[-1]
    assert rec[0] == "fwd_glu" and bool(rec[3] & 4) == pair, rec
    for j, Y in enumerate((Yg, Yu)):
        ref = H[:, j * r:(j + 1) * r].float() @ B[j].float().T
        # one bf16 rounding of the result: 2^-9 / sqrt(3) = 1.1e-3 as a whole,
        # half an ulp (2^-9 of the value) plus fp32 summation noise per element
        assert (Y.float() - ref).norm() / ref.norm() < 3e-3
        assert bool(((Y.float() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-4).all())
    assert torch.equal(M, (Yg.float() * Yu.float()).to(torch.bfloat16))
    di = cola.desc(n, d, d_ff, r, ld_y=ld, mode="infer")
    wi = cola.workspace(di, 2)
    cola.cola_fwd_gate_up(di, X, A, B[0], B[1], Mi, None, None, None, None, wi)
    assert torch.equal(M, Mi)
    for t in (M, Mi, Yg, Yu):
        assert torch.as_strided(t, (n, ld), (ld, 1))[:, d_ff:].isnan().all()
    assert cola.cola_check_status(ws)[0] == 0 and cola.cola_check_status(wi)[0] == 0
