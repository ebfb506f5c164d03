"""Right edges inside a 64-column box and inside a 16-byte group, and rows that
begin and end inside a 32-byte sector: the plain output GEMM on single CTAs and on
CTA pairs and the gated forward, whose last box is stored with clipped rows.
Against a plain fp32 product of the same stored bf16 H; the row padding stays as it
was.
"""
import pytest
import torch

from paper_2502_10940_gb300 import inputs as I

pytestmark = pytest.mark.gpu
PAIR = 4   # launch-trace flag: CTA pairs


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_10940_gb300 import build
    build.build()


# n, d_out, row pitch, r: one column past a box, one short of it, inside a 16-byte
# group, a 16-byte group that ends a row inside a sector; one row past a warp's 32
@pytest.mark.parametrize("n,d_out,ld,r,pair",
                         [(161, 65, 72, 64, False), (300, 191, 192, 128, False), (129, 333, 344, 192, False),
                          (2049, 1000, 1000, 256, False), (16500, 1003, 1016, 512, True), (16417, 1033, 1040, 512, True)])
def test_right_edges(n, d_out, ld, r, pair):
    from paper_2502_10940_gb300 import cola
    d_in = 256

    def new(cols, pitch=None):
        return torch.full((n, pitch or cols), 7.0, dtype=torch.bfloat16, device="cuda")[:, :cols]

    X, A = I.normal_bf16(n, d_in, 1.0, 1, "cuda"), I.normal_bf16(2 * r, d_in, d_in ** -0.5, 2, "cuda")
    B = [I.normal_bf16(d_out, r, r ** -0.5, 3 + j, "cuda") for j in range(2)]
    Y, M, Yg, Yu = [new(d_out, ld) for _ in range(2)], new(d_out, ld), new(d_out, ld), new(d_out, ld)
    Z, H = new(2 * r), new(2 * r)
    d = cola.desc(n, d_in, d_out, r, ld_y=ld, mode="cola")
    ws = cola.workspace(d, 2)
    with cola.Trace(8) as tr:
        cola.cola_fwd_shared_x(d, X, A, B, Y, Z, H, ws)
        ref = [H[:, j * r:(j + 1) * r].float() @ B[j].float().T for j in range(2)]
        cola.cola_fwd_gate_up(d, X, A, B[0], B[1], M, Yg, Yu, Z, H, ws)
    assert cola.cola_check_status(ws) == (0, 0)
    assert all(bool(t[3] & PAIR) == pair for t in tr.records() if t[0] in ("fwd_y", "fwd_glu")), tr.records()

    def close(got, want):
        # one bf16 rounding of each entry, and fp32 sums of up to 512 products: 2^-8
        # of the entry with 2^-14 of the largest
        assert ((got.float() - want).abs() <= want.abs() * 2 ** -8 + want.abs().max() * 2 ** -14).all()

    for got, want in zip(Y + [Yg, Yu], ref + ref):
        close(got, want)
    assert torch.equal(M, (Yg.float() * Yu.float()).bfloat16())
    for t in Y + [M, Yg, Yu]:
        assert (torch.as_strided(t, (n, ld), (ld, 1))[:, d_out:] == 7.0).all()
