"""Large GEMMs whose weight A has rows that do not begin on 32-byte sectors run on
a copy of it at an aligned pitch: bit for bit the results of a call whose A has an
aligned pitch already, the weight's own padding unread, and neither the weight nor
what the workspace keeps between the launches disturbed.
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


# n, d_in, r, projections (0: the down layer of a gated MLP, forward only): d_in inside and at the
# end of a 16-byte group; token splits of the weight gradients that leave room for
# the copy; a token count whose dZ has none; single CTAs
@pytest.mark.parametrize("n,d_in,r,c", [(16385, 4101, 512, 1), (9000, 4104, 512, 2), (16400, 4099, 512, 0),
                                        (65536, 1000, 512, 1), (2048, 33000, 512, 1), (30001, 1000, 256, 1),
                                        (24000, 997, 128, 3)])
@pytest.mark.parametrize("mode", ["cola", "cola_m"])
def test_misaligned_weight(n, d_in, r, c, mode):
    from paper_2502_10940_gb300 import cola
    glu, c, d_out = c == 0, max(c, 1), 256
    lx, la = I.padded_ld(d_in), (d_in + 63) // 64 * 64
    X = I.normal_bf16(n, d_in, 1.0, 1, "cuda", ld=lx)
    A0 = I.normal_bf16(c * r, d_in, d_in ** -0.5, 2, "cuda", ld=lx)
    A1 = torch.empty((c * r, la), dtype=torch.bfloat16, device="cuda")[:, :d_in].copy_(A0)
    A0_bits = torch.as_strided(A0, (c * r, lx), (lx, 1)).clone()
    B = [I.normal_bf16(d_out, r, r ** -0.5, 3 + j, "cuda") for j in range(c)]
    dY = [I.normal_bf16(n, d_out, 1.0, 6 + j, "cuda") for j in range(c)]
    Yg, Yu = (I.normal_bf16(n, d_in, 1.0, 10 + j, "cuda", ld=lx) for j in range(2))
    assert lx % 16 == 8

    def run(A):
        def new(rows, cols, ld=None):
            return torch.zeros((rows, ld or cols), dtype=torch.bfloat16, device="cuda")[:, :cols]

        lda = A.stride(0)
        d = cola.desc(n, d_in, d_out, r, ld_x=lx, ld_a=lda, mode=mode)
        ws = cola.workspace(d, c)
        Y, Z, H = [new(n, d_out) for _ in range(c)], new(n, c * r), new(n, c * r) if mode == "cola" else None
        dX, dX2, dA, dB = new(n, d_in, lx), new(n, d_in, lx), new(c * r, d_in, lda), [new(d_out, r) for _ in range(c)]
        with cola.Trace(32) as tr:
            if c > 1:
                cola.cola_fwd_shared_x(d, X, A, B, Y, Z, H, ws)
                cola.cola_bwd_shared_x(d, X, A, B, dY, Z, H, dX, dA, dB, ws)
            else:
                cola.cola_fwd(d, X, A, B[0], Y[0], Z, H, ws)
                if glu:
                    cola.cola_bwd_down_gated(d, X, A, B[0], dY[0], Z, H, Yg, Yu, dX, dX2, dA, dB[0], ws)
                else:
                    cola.cola_bwd(d, X, A, B[0], dY[0], Z, H, dX, dA, dB[0], ws)
        assert cola.cola_check_status(ws) == (0, 0)
        # the forward's copy lies in dZ, the backward's behind it
        need, dz = c * r * la * 2, (n * c * r * 2 + 255) // 256 * 256
        fits = (need <= dz) + (not glu and need <= cola.cola_workspace_size(d, c) - 256 - dz)
        return fits, [t[0] for t in tr.records()].count("repack"), Y + [Z, dX, dX2, dA] + dB

    (fits, k0, got), (_, k1, want) = run(A0), run(A1)
    assert (k0, k1) == (fits, 0)
    assert all(torch.equal(g, w) for g, w in zip(got, want))
    assert float(want[c].float().norm()) > 0
    assert torch.equal(torch.as_strided(A0, (c * r, lx), (lx, 1)), A0_bits)
    dA = got[c + 3]
    assert (torch.as_strided(dA, (c * r, lx), (lx, 1))[:, d_in:] == 0).all()


# single CTAs and CTA pairs; a workspace with and without the room for the copy
@pytest.mark.parametrize("n,d_in,r,c", [(30001, 1000, 256, 1), (9000, 4101, 512, 2)])
def test_misaligned_weight_inference(n, d_in, r, c):
    from paper_2502_10940_gb300 import cola
    lx, la, d_out = I.padded_ld(d_in), (d_in + 63) // 64 * 64, 256
    X = I.normal_bf16(n, d_in, 1.0, 1, "cuda", ld=lx)
    A0 = I.normal_bf16(c * r, d_in, d_in ** -0.5, 2, "cuda", ld=lx)
    A1 = torch.empty((c * r, la), dtype=torch.bfloat16, device="cuda")[:, :d_in].copy_(A0)
    B = [I.normal_bf16(d_out, r, r ** -0.5, 3 + j, "cuda") for j in range(c)]

    def run(A, less=0):
        Y = [torch.zeros((n, d_out), dtype=torch.bfloat16, device="cuda") for _ in range(c)]
        d = cola.desc(n, d_in, d_out, r, ld_x=lx, ld_a=A.stride(0), mode="infer")
        ws = cola.workspace(d, c)
        with cola.Trace(8) as tr:
            if c > 1:
                cola.cola_fwd_shared_x(d, X, A, B, Y, None, None, ws[:ws.numel() - less])
            else:
                cola.cola_fwd(d, X, A, B[0], Y[0], None, None, ws[:ws.numel() - less])
        assert cola.cola_check_status(ws) == (0, 0)
        return [t[0] for t in tr.records()].count("repack"), Y, ws.numel()

    k1, want, b1 = run(A1)
    k0, got, b0 = run(A0)
    k2, low, _ = run(A0, less=b0 - b1)
    assert (k0, k1, k2) == (1, 0, 0) and b0 - b1 == (c * r * la * 2 + 255) // 256 * 256
    assert all(torch.equal(g, w) and torch.equal(x, w) for g, x, w in zip(got, low, want))
    assert float(want[0].float().norm()) > 0
