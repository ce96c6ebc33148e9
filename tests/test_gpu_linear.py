"""GPU parity of the dense projection (dm_linear) against the oracle's in_proj / out_proj rows: sizes that
span several tiles of every kernel with ragged tails in every dimension, the row-scale and addend epilogue, and
in-place accumulation into an fp32 output."""
import numpy as np
import pytest
import torch

from oracle import bimamba_oracle as O
from paper_2511_15927_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dm():
    from paper_2511_15927_b200 import build
    build.build()
    from paper_2511_15927_b200 import binding
    return binding


def _rand(shape, seed, dtype, scale=1.0):
    a = (scale * np.random.default_rng(seed).standard_normal(shape)).astype(np.float32)
    return I.round_to_bf16(a) if dtype == I.BF16 else a


@pytest.mark.parametrize("dtype", [I.BF16, I.F32])
@pytest.mark.parametrize("M,N,K", [(1, 8, 8), (300, 520, 200), (129, 257, 72), (1000, 1288, 256), (2048, 2048, 1024), (77, 100, 64),
                                   (512, 50304 // 16, 128),
                                   # few rows, many columns (ragged rows and columns)
                                   (300, 13000, 192), (512, 17024, 256), (130, 18000, 64),
                                   # up to 128 rows: K cut over clusters of 2, 4 and 8 CTAs and not at all, one and two CTAs per SM, uneven K shares
                                   (16, 4200, 2048), (17, 5000, 1096), (48, 300, 4096), (64, 130, 2056), (65, 9000, 1032), (112, 2000, 3000), (128, 1001, 2048),
                                   # the two-CTA kernel around its tiles of 256 rows x 256 or 128 columns: one row or column more, one CTA of a
                                   # pair without rows, K of a single and of one more k-block than the ring of stages holds, several rounds
                                   (257, 128, 64), (256, 129, 72), (384, 250, 456), (385, 40000, 512), (2304, 9480, 136)])
def test_linear_parity(dm, dtype, M, N, K):
    from paper_2511_15927_b200.torch_io import dev, dm_dtype, tdtype
    x = _rand((M, K), 1, dtype); w = _rand((N, K), 2, dtype, 0.05)
    xd, wd = dev(x, dtype), dev(w, dtype)
    want = O.in_proj(x, w)
    for y_dtype in ([I.BF16, I.F32] if dtype == I.BF16 else [I.F32]):
        yd = torch.empty((M, N), device="cuda", dtype=tdtype(y_dtype))
        dm.dm_linear(dm_dtype(dtype), xd.data_ptr(), wd.data_ptr(), yd.data_ptr(), dm_dtype(y_dtype), M, K, N, 0, 0,
                     torch.cuda.current_stream().cuda_stream)
        dm.dm_check(0)
        got = yd.float().cpu().numpy().astype(np.float64)
        rel = np.linalg.norm(got - want) / np.linalg.norm(want)
        assert rel <= (3e-3 if y_dtype == I.BF16 else 1e-5), rel       # bf16 output rounding alone is ~2e-3
        if y_dtype == I.F32:
            np.testing.assert_allclose(got, want, rtol=0, atol=2e-5 * np.sqrt(K) * 0.05 * 4 + 1e-6)


@pytest.mark.parametrize("dtype", [I.BF16, I.F32])
@pytest.mark.parametrize("shape", [(333, 300, 136), (300, 13000, 136), (100, 300, 136)])
def test_linear_epilogue_scale_addend_inplace(dm, dtype, shape):
    from paper_2511_15927_b200.torch_io import dev, dm_dtype
    M, N, K = shape                                         # tensor-core path: narrow and wide tiles of the two-CTA kernel, the kernel for up to 128 rows
    x = _rand((M, K), 3, dtype); w = _rand((N, K), 4, dtype, 0.05)
    sc = np.random.default_rng(5).uniform(0.5, 2.0, M).astype(np.float32)
    add = np.random.default_rng(6).standard_normal((M, N)).astype(np.float32)
    xd, wd, scd = dev(x, dtype), dev(w, dtype), dev(sc)
    yd = dev(add.copy())                                    # accumulate in place: y <- sc * (x W^T) + y
    dm.dm_linear(dm_dtype(dtype), xd.data_ptr(), wd.data_ptr(), yd.data_ptr(), dm.DM_F32, M, K, N, scd.data_ptr(), yd.data_ptr(),
                 torch.cuda.current_stream().cuda_stream)
    dm.dm_check(0)
    want = sc[:, None].astype(np.float64) * O.out_proj(x, w) + add
    np.testing.assert_allclose(yd.cpu().numpy().astype(np.float64), want, rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("y_dtype", [I.BF16, I.F32])
@pytest.mark.parametrize("M,N", [(100, 300), (128, 64), (129, 32), (129, 64), (129, 100), (300, 300), (256, 520), (333, 40), (2304, 1096)])
def test_linear_separate_addend(dm, y_dtype, M, N):
    """An addend that is not the output, both output types: every epilogue of the tensor-core kernels (up to 128 rows; rows of 16-byte pieces, whole and cut short
    inside a group of 64 columns and of 32; rows that are not)."""
    from paper_2511_15927_b200.torch_io import dev, dm_dtype, tdtype
    K = 136
    x = _rand((M, K), 7, I.BF16); w = _rand((N, K), 8, I.BF16, 0.05)
    sc = np.random.default_rng(9).uniform(0.5, 2.0, M).astype(np.float32)
    add = np.random.default_rng(10).standard_normal((M, N)).astype(np.float32)
    xd, wd, scd, addd = dev(x, I.BF16), dev(w, I.BF16), dev(sc), dev(add)
    yd = torch.full((M, N), float("nan"), device="cuda", dtype=tdtype(y_dtype))
    dm.dm_linear(dm.DM_BF16, xd.data_ptr(), wd.data_ptr(), yd.data_ptr(), dm_dtype(y_dtype), M, K, N, scd.data_ptr(), addd.data_ptr(), torch.cuda.current_stream().cuda_stream)
    dm.dm_check(0)
    want = sc[:, None].astype(np.float64) * O.out_proj(x, w) + add
    # bf16: half a unit in the last place (2^-9 of the value) beside the fp32 sums' error
    np.testing.assert_allclose(yd.double().cpu().numpy(), want, rtol=2.0 ** -8 if y_dtype == I.BF16 else 1e-5, atol=1e-5)


@pytest.mark.parametrize("M,N,K", [(6400, 768, 72), (6300, 840, 136), (9728, 2048, 64), (2048, 9728, 456), (600, 24960, 64)])
def test_linear_mixed_tile_widths(dm, M, N, K):
    """The two-CTA kernel with tiles of two widths: an incomplete last round cut into halves (rows or columns first in the tile order), a last column tile of 72 columns,
    both, with ragged rows; a column strip whose tiles start in the last round of wide ones."""
    test_linear_parity(dm, I.BF16, M, N, K)


@pytest.mark.parametrize("M,N,K", [(32, 11264, 520), (33, 11392, 520), (128, 18900, 200), (100, 25000, 136), (5, 25000, 136)])
def test_linear_few_rows_uncut_tiles(dm, M, N, K):
    """Up to 128 rows around the line where K is no longer cut (88 and 89 tiles), one tile per SM, and more tiles than SMs with one and two CTAs on each."""
    test_linear_parity(dm, I.BF16, M, N, K)


@pytest.mark.parametrize("M,N,K", [(5, 38016, 72), (64, 38016, 520), (80, 40000, 1032), (81, 37889, 72), (128, 38100, 456)])
def test_linear_few_rows_tiles_in_turn(dm, M, N, K):
    """Up to 128 rows and more tiles than two to an SM: each CTA takes several, in two accumulator buffers; three rounds for some CTAs; rows that are not 16-byte pieces."""
    test_linear_parity(dm, I.BF16, M, N, K)


@pytest.mark.parametrize("M,N,K", [(96, 300, 768), (97, 300, 768), (97, 300, 776), (128, 20000, 776), (97, 19000, 72)])
def test_linear_few_rows_kernel_choice(dm, M, N, K):
    """The lines between the few-row kernel and the two-CTA one: 96 rows, K of 768; more tiles than SMs with more than 80 rows (three stages to a CTA)."""
    test_linear_parity(dm, I.BF16, M, N, K)
