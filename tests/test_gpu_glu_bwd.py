"""The gated dX epilogue at the edges of its 64-column chunks, on single CTAs,
on CTA pairs and in its long-K form, with gradients written apart from and
over the saved outputs: bit for bit bf16(dM * Y) of the plain backward's dM,
which the other tests check against the oracle.
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
    (4360, 4033, 512, True), (4231, 4096, 512, True), (4360, 4095, 512, True),
    (2184, 4033, 1024, True), (2200, 4088, 1024, True), (2177, 4160, 1024, True),
])
def test_gated_dx_chunk_edges(n, d_ff, r, pair):
    from paper_2502_10940_gb300 import cola
    d, ld = 128, I.padded_ld(d_ff)

    def wide(seed, fill=float("nan")):
        buf = torch.full((n, ld), fill, dtype=torch.bfloat16, device="cuda")
        if seed is not None:
            buf[:, :d_ff] = I.normal_bf16(n, d_ff, 1.0, seed, "cuda")
        return buf[:, :d_ff]

    M, Yg, Yu = wide(1), wide(2), wide(3)
    A, B = I.normal_bf16(r, d_ff, d_ff ** -0.5, 4, "cuda", ld=ld), I.normal_bf16(d, r, r ** -0.5, 5, "cuda")
    dY = I.normal_bf16(n, d, 1.0, 6, "cuda")
    Z = I.normal_bf16(n, r, 1.0, 7, "cuda")
    dd = cola.desc(n, d_ff, d, r, ld_x=ld, ld_a=ld, mode="cola_m")
    ws = cola.workspace(dd)
    dA, dB = torch.empty((r, ld), dtype=torch.bfloat16, device="cuda")[:, :d_ff], torch.empty_like(B)
    dM = wide(None)
    cola.cola_bwd(dd, M, A, B, dY, Z, None, dM, dA, dB, ws)
    want_g = (dM.float() * Yu.float()).to(torch.bfloat16)
    want_u = (dM.float() * Yg.float()).to(torch.bfloat16)

    def check(dYg, dYu):
        with cola.Trace(8) as tr:
            cola.cola_bwd_down_gated(dd, M, A, B, dY, Z, None, Yg, Yu, dYg, dYu, dA, dB, ws)
        rec = [x for x in tr.records() if x[0] == "bwd_dx"]
        assert len(rec) == 1 and bool(rec[0][3] & 4) == pair, rec
        assert torch.equal(dYg, want_g) and torch.equal(dYu, want_u)
        for t in (dYg, dYu):
            assert torch.as_strided(t, (n, ld), (ld, 1))[:, d_ff:].isnan().all()

    check(wide(None), wide(None))
    check(Yg, Yu)       # in place: dY_gate over Y_gate, dY_up over Y_up
    assert cola.cola_check_status(ws)[0] == 0


# d_ff mod 64 = 1, 33, 63: the last chunk of a row is stored directly, not from its box
@pytest.mark.parametrize("swap", [False, True], ids=["over", "crossed"])
@pytest.mark.parametrize("n,d_ff,r", [(4360, 4033, 1024), (4330, 4065, 768), (2177, 4095, 1024), (4360, 4095, 512)])
def test_gated_dx_in_place_at_a_ragged_edge(n, d_ff, r, swap):
    """Gradients over the saved outputs equal those written apart, bit for bit, run after run."""
    from paper_2502_10940_gb300 import cola
    d, ld = 128, I.padded_ld(d_ff)
    M, Yg, Yu = (I.normal_bf16(n, d_ff, 1.0, s, "cuda", ld=ld) for s in (1, 2, 3))
    A, B = I.normal_bf16(r, d_ff, d_ff ** -0.5, 4, "cuda", ld=ld), I.normal_bf16(d, r, r ** -0.5, 5, "cuda")
    dY, Z = I.normal_bf16(n, d, 1.0, 6, "cuda"), I.normal_bf16(n, r, 1.0, 7, "cuda")
    dd = cola.desc(n, d_ff, d, r, ld_x=ld, ld_a=ld, mode="cola_m")
    ws = cola.workspace(dd)
    dA, dB = torch.empty((r, ld), dtype=torch.bfloat16, device="cuda")[:, :d_ff], torch.empty_like(B)

    def run(yg, yu, dyg, dyu):
        with cola.Trace(8) as tr:
            cola.cola_bwd_down_gated(dd, M, A, B, dY, Z, None, yg, yu, dyg, dyu, dA, dB, ws)
        assert [x[3] & 4 for x in tr.records() if x[0] == "bwd_dx"] == [4], tr.records()   # CTA pairs
        return dyg, dyu

    def fresh(t):
        return torch.empty((n, ld), dtype=torch.bfloat16, device="cuda")[:, :d_ff].copy_(t)

    want = run(Yg, Yu, fresh(Yg), fresh(Yu))
    for _ in range(8):
        yg, yu = fresh(Yg), fresh(Yu)
        got = run(yg, yu, *((yu, yg) if swap else (yg, yu)))
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert cola.cola_check_status(ws)[0] == 0
