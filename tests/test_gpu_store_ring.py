"""The plain store epilogues at widths whose last column tile gives a warp an odd
number of chunks, so that a staged box is written again while the stores of the
last full tile are on their way: 64-column boxes, one per warp, on CTA pairs, and
the ring of two 32-column boxes of single CTAs.  Against a plain fp32 product of the
same stored bf16 H, box by box.
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


def _box_errors(got, ref, cols):
    """Largest relative error of a 32-row box of `cols` columns."""
    n, w = (ref.shape[0] + 31) // 32 * 32, (ref.shape[1] + cols - 1) // cols * cols
    d, r = (torch.zeros((n, w), device="cuda") for _ in range(2))
    d[:ref.shape[0], :ref.shape[1]] = got.float() - ref
    r[:ref.shape[0], :ref.shape[1]] = ref
    norm = lambda t: t.view(n // 32, 32, w // cols, cols).square().sum((1, 3)).sqrt()
    return float((norm(d) / norm(r)).max())


# d_out mod 256: 192 (3 boxes of 64, 6 of 32 columns), 136 (the last one partial), 91 (ragged right edge:
# 64-column boxes on single CTAs too)
@pytest.mark.parametrize("n,d_in,r,box,pair", [(4313, 1536, 512, 64, True), (4313, 512, 128, 32, False)],
                         ids=["pairs", "single"])
@pytest.mark.parametrize("d_out", [3776, 3720, 3675])
def test_pair_store_of_an_odd_chunk_count(d_out, n, d_in, r, box, pair):
    from paper_2502_10940_gb300 import cola
    ld = (d_out + 15) // 16 * 16   # rows on 32-byte sectors: single CTAs keep the ring
    X, A = I.normal_bf16(n, d_in, 1.0, 1, "cuda"), I.normal_bf16(2 * r, d_in, d_in ** -0.5, 2, "cuda")
    B = [I.normal_bf16(d_out, r, r ** -0.5, 3 + j, "cuda") for j in range(2)]
    Y = [torch.empty((n, ld), dtype=torch.bfloat16, device="cuda")[:, :d_out] for _ in range(2)]
    Z, H = (torch.empty((n, 2 * r), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    d = cola.desc(n, d_in, d_out, r, ld_y=ld, mode="cola")
    ws = cola.workspace(d, 2)
    ref = None
    for _ in range(4):
        for y in Y:
            y.zero_()
        with cola.Trace(4) as tr:
            cola.cola_fwd_shared_x(d, X, A, B, Y, Z, H, ws)
        assert tr.records()[-1][0] == "fwd_y" and bool(tr.records()[-1][3] & 4) == pair, tr.records()
        if ref is None:
            ref = [H[:, j * r:(j + 1) * r].float() @ B[j].float().T for j in range(2)]
        for j in range(2):
            # one bf16 rounding of the result: 2^-9 / sqrt(3) = 1.1e-3 over a box of some thousand
            # values, 2^-8 at most of each; a box that is misplaced or overwritten is off by > 1
            err = _box_errors(Y[j], ref[j], box)
            assert err < 3e-3, (j, err)
    assert cola.cola_check_status(ws)[0] == 0
