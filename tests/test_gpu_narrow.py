"""The scan of narrow states (bf16, d_state 16, more than 64 tokens) against the CPU oracle: lengths around its sub-chunks of 32 tokens and around one round of a chain's warps, both head
widths, odd head counts, carried state in and out, flags, single directions; and its error beside that of the 128-token kernel on the same inputs."""
import numpy as np
import pytest

from oracle import bimamba_oracle as O
from paper_2511_15927_b200 import inputs as I

pytestmark = pytest.mark.gpu
BF16_REL, BF16_ABS = 1e-2, 5e-2


@pytest.fixture(scope="module")
def G():
    from paper_2511_15927_b200 import build
    build.build()
    import tests.gpu_util as g
    return g


def _check(G, got, want):
    assert np.all(np.isfinite(got))
    assert G.rel_l2(got, want) <= BF16_REL, G.rel_l2(got, want)
    assert G.max_abs(got, want) <= BF16_ABS, G.max_abs(got, want)


# (batch, heads, headdim, length, conv width, flags, directions).  A chain's tile warps take 32 tokens each in turn: 19 warps (608 tokens a round) for up to 148 chains, 9 (288), 5 (160) and 4 (128) from
# 149, 297 and 445.  Heads of 64 are chains of half a head each for up to 74 heads of all sequences and directions, and without the D skip (flag 4), and one chain elsewhere.  (40, 16): more chains
# than are resident
@pytest.mark.parametrize("B,H,P,L,k,flags,dirs", [
    (1, 2, 64, 65, 4, 7, 3), (2, 8, 64, 96, 4, 7, 3), (2, 8, 32, 97, 4, 7, 3), (1, 8, 64, 128, 4, 7, 3), (3, 8, 32, 129, 3, 7, 3), (1, 16, 32, 159, 2, 6, 3),
    (2, 8, 64, 161, 4, 5, 1), (2, 8, 64, 255, 4, 3, 2), (1, 8, 64, 640, 4, 7, 3), (1, 8, 64, 641, 4, 7, 3), (2, 24, 64, 513, 4, 7, 3), (4, 24, 64, 225, 4, 7, 3), (10, 16, 64, 161, 3, 7, 3),
    (40, 16, 64, 130, 4, 7, 3), (1, 4, 64, 1301, 4, 0, 3), (2, 72, 64, 100, 4, 7, 3),
    (1, 8, 64, 608, 4, 7, 3), (1, 8, 64, 609, 4, 7, 3), (5, 8, 64, 608, 4, 7, 3), (5, 8, 64, 609, 4, 7, 3), (5, 8, 64, 641, 2, 6, 3), (4, 24, 64, 288, 4, 7, 3), (4, 24, 64, 289, 4, 7, 3),
    (4, 24, 64, 321, 3, 7, 3), (10, 16, 64, 160, 4, 7, 3), (6, 16, 32, 289, 4, 7, 3), (2, 24, 64, 321, 4, 3, 3), (2, 3, 64, 100, 4, 7, 3), (3, 5, 64, 193, 4, 7, 3), (2, 3, 32, 97, 4, 7, 3),
    (1, 5, 32, 66, 3, 5, 3), (26, 3, 64, 72, 4, 7, 3)])
def test_forward_and_state(G, B, H, P, L, k, flags, dirs):
    shape = I.MixerShape(B, L, P * H // 2, 2, 16, k, H)
    wf, wr = I.make_mixer_weights(shape, 80 + L, I.BF16, perturb=True)
    x = I.make_activations(shape, 80 + L, I.BF16)
    kw = G.oracle_kwargs(shape, flags)
    want = O.bimamba_forward(x, wf, wr, dir_mask=dirs, **kw)
    got = G.run_forward(shape, I.BF16, wf, wr, x, flags=flags, dir_mask=dirs)
    _check(G, got, want)
    np.testing.assert_array_equal(got, G.run_forward(shape, I.BF16, wf, wr, x, flags=flags, dir_mask=dirs))          # run to run
    if not dirs & 1:
        return
    ssm_in, conv_in = I.make_states(shape, 80 + L, I.BF16)
    y_o, s_o, c_o = O.bimamba_block_step(x, wf, wr, ssm_state_in=ssm_in, conv_state_in=conv_in, dir_mask=dirs, **kw)
    y_g, s_g, c_g = G.run_block_step(shape, I.BF16, wf, wr, x, ssm_in, conv_in, flags=flags, dir_mask=dirs)
    _check(G, y_g, y_o)
    _check(G, s_g, s_o)
    _check(G, c_g, c_o)


@pytest.mark.parametrize("d,P,L,flags", [(512, 64, 300, 7), (512, 32, 300, 7), (512, 64, 500, 3), (1024, 64, 1000, 3), (512, 32, 300, 2), (768, 64, 96, 7)])
def test_error_is_no_larger_than_that_of_the_128_token_kernel(G, d, P, L, flags):
    """From a carried state, with and without the D skip and the norm, mean of three seeds.  The output: not larger.  The state: both kernels round B' and one factor of each term beside it once (x' here,
    w x' there) and sum in fp32, so that their errors are two samples of one distribution; 6 % between them (they came out 0.93 to 1.03 apart; rounding w B' a second time gave 1.11 to 1.14)."""
    e = []
    for seed in range(3):
        shape = I.MixerShape(1, L, d, 2, 16, 4, 2 * d // P)
        wf, wr = I.make_mixer_weights(shape, seed, I.BF16, perturb=True)
        x = I.make_activations(shape, seed, I.BF16)
        ssm_in, conv_in = I.make_states(shape, seed, I.BF16)
        y_o, s_o, _ = O.bimamba_block_step(x, wf, wr, ssm_state_in=ssm_in, conv_state_in=conv_in, **G.oracle_kwargs(shape, flags))
        for c in (0, 128):
            y, s, _ = G.run_block_step(shape, I.BF16, wf, wr, x, ssm_in, conv_in, flags=flags, chunk=c)
            e.append((G.rel_l2(y, y_o), G.rel_l2(s, s_o)))
    narrow, wide = np.mean(e[0::2], axis=0), np.mean(e[1::2], axis=0)
    assert narrow[0] <= wide[0] and narrow[1] <= 1.06 * wide[1], (narrow, wide)


def test_causality(G):
    shape = I.MixerShape(2, 300, 256, 2, 16, 4, 8)
    wf, wr = I.make_mixer_weights(shape, 4, I.BF16, perturb=True)
    x = I.make_activations(shape, 4, I.BF16)
    x2 = x.copy(); x2[0, 150] += 1.0
    for dirs in (1, 2):
        d = G.run_forward(shape, I.BF16, wf, wr, x2, dir_mask=dirs) - G.run_forward(shape, I.BF16, wf, wr, x, dir_mask=dirs)
        before, after = (d[0, :150], d[0, 150:]) if dirs == 1 else (d[0, 151:], d[0, :151])
        assert np.all(before == 0) and np.any(after != 0) and np.all(d[1] == 0)


def test_a_row_does_not_depend_on_the_rows_beside_it(G):
    """Few heads are split into halves, many are not: the sums of squares, and with them every bit of a row, are the same either way.  20 rows of 4 heads are 160 chains, 3 rows 24 (d_model 128: the
    products' tiles are the same for both); the host-buffer call cuts its batch into pieces of 3 rows."""
    shape = I.MixerShape(20, 2100, 128, 2, 16, 4, 4)
    wf, wr = I.make_mixer_weights(shape, 6, I.BF16, perturb=True)
    x = I.make_activations(shape, 6, I.BF16)
    whole = G.run_forward(shape, I.BF16, wf, wr, x)
    few = I.MixerShape(3, 2100, 128, 2, 16, 4, 4)
    np.testing.assert_array_equal(G.run_forward(few, I.BF16, wf, wr, np.ascontiguousarray(x[7:10])), whole[7:10])
    np.testing.assert_array_equal(G.run_forward_host(shape, I.BF16, wf, wr, x), whole)


@pytest.mark.parametrize("B,flags", [(2, 7), (3, 7), (3, 3)])
def test_no_room_for_sums_of_half_heads(G, B, flags):
    """expand 32: the sums of squares of 32 channels each have no place in the workspace, so heads of 64 stay whole at any batch (64 and 96 chains) and leave one sum each."""
    shape = I.MixerShape(B, 200, 32, 32, 16, 4, 16)
    assert shape.headdim == 64
    wf, wr = I.make_mixer_weights(shape, 7, I.BF16, perturb=True)
    x = I.make_activations(shape, 7, I.BF16)
    _check(G, G.run_forward(shape, I.BF16, wf, wr, x, flags=flags), O.bimamba_forward(x, wf, wr, **G.oracle_kwargs(shape, flags)))
