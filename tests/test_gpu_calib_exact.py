"""The calibration's float64 products on inputs whose exact result is known.

One token (its softmax weight is 1), identity rotations and values below 2^-26
(every level of Q2 is then fp16 zero) leave Vt - V = -V, so the value loss is
the mean over query rows and heads of |W_O[j] V|^2 / d_model: one product of
depth 128 whose operands a test chooses freely, compared with exact rational
arithmetic.  The tolerance is what a float64 FMA chain guarantees for terms of
one sign: 128 roundings per product (twice in the square), plus the roundings of
the sums of squares and of the mean (at most one per 32 channels, 256 rows and
a few more).
"""
from fractions import Fraction

import pytest
import torch

from paper_2608_02691_gb300 import optr

pytestmark = pytest.mark.gpu

F64 = torch.float64
D = 128
U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_02691_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _value_loss(v, W, nt):
    """(loss, tolerance) of one token with value v [128] under W [g][d_model][128]."""
    g, dm, _ = W.shape
    cfg = optr.calib_config(g, dm, 1, nt)
    I = torch.eye(D, dtype=F64)
    zeros = torch.zeros(1, D, dtype=F64)
    loss, _ = optr.optr_calib_loss_grad(
        cfg, 1, *[x.cuda() for x in (torch.zeros(nt, g, D, dtype=F64), zeros, v.view(1, D),
                                     torch.zeros(nt, dtype=torch.int32), W, zeros[0], I,
                                     torch.zeros(D, D, dtype=F64))], R_K=I.cuda(), grad=False)
    return float(loss.item()), (2 * D + dm / 32 + g * nt / 256 + 32) * U


def _exact(v, W):
    vs = [Fraction(x) for x in v.tolist()]
    sq = {}
    for w in W.flatten(0, 1).tolist():
        key = tuple(w)
        if key not in sq:
            sq[key] = [sum(a * Fraction(b) for a, b in zip(vs, w)) ** 2, 0]
        sq[key][1] += 1
    return sum(x * n for x, n in sq.values()) / (W.shape[0] * W.shape[1])


# (query rows, output channels): both tile shapes of the product, whole and
# ragged
SHAPES = [(1, 1), (65, 1249)]


def _const(c, last=1.0):
    x = torch.full((D,), c, dtype=F64)
    x[-1] *= last
    return x


@pytest.mark.parametrize("nt,dm", SHAPES)
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("x", [
    _const(15 / 17), _const(41 / 51), _const(259 / 510), _const(float.fromhex("0x1.fc04040404040p0")),
    _const(1 / 17, 8.0), _const(9 / 17, 64.0),
], ids=["15/17", "41/51", "259/510", "1.984", "8/17", "64*9/17"])
def test_constant_rows(x, sign, nt, dm):
    """Digits that repeat over the whole depth: the largest sums per weight."""
    v, W = x * 2.0 ** -36, (sign * x).expand(1, dm, D).contiguous()
    loss, rel = _value_loss(v, W, nt)
    ref = _exact(v, W)
    assert abs(Fraction(loss) - ref) <= rel * ref


def _spread(seed, lo, hi):
    """Positive values with exponents uniform in [lo, hi)."""
    gen = torch.Generator().manual_seed(seed)
    m = 1.0 + torch.rand(D, generator=gen, dtype=F64)
    return m * 2.0 ** torch.randint(lo, hi, (D,), generator=gen).to(F64)


def _outlier(seed, k, e):
    x = _spread(seed, 0, 2)
    x[k] = 2.0 ** e
    return x


WIDE = {
    # the row's largest element meets a zero, or the column's smallest
    "outlier x zero": (_outlier(1, 5, 60), _outlier(2, 5, -2000)),
    "outlier x small": (_outlier(1, 5, 40), _outlier(2, 5, -50)),
    "both outliers": (_outlier(1, 5, 50), _outlier(2, 6, 50)),
    "one element x zeros": (_outlier(1, 0, 200), torch.cat([torch.zeros(1), torch.ones(127)]).double()),
    "spread 10": (_spread(3, 0, 10), _spread(4, 0, 10)),
    "spread 80": (_spread(3, 0, 80), _spread(4, 0, 80)),
    "spread 600": (_spread(3, -600, 0), _spread(4, -400, 0)),
    "softmax": (torch.exp(10 * torch.randn(D, generator=torch.Generator().manual_seed(5), dtype=F64) - 40),
                _spread(6, 0, 12)),
}


@pytest.mark.parametrize("nt,dm", SHAPES)
@pytest.mark.parametrize("name", WIDE)
def test_wide_range_inside_a_row(name, nt, dm):
    """Elements far below their row's or column's largest keep their own precision."""
    v, w = WIDE[name]
    v = v / v.max() * 2.0 ** -36
    W = w.expand(1, dm, D).contiguous()
    loss, rel = _value_loss(v, W, nt)
    ref = _exact(v, W)
    assert ref > 0
    assert abs(Fraction(loss) - ref) <= rel * ref


@pytest.mark.parametrize("nt,dm", SHAPES)
def test_infinite_weight_gives_an_infinite_loss(nt, dm):
    W = _spread(7, 0, 4).expand(1, dm, D).contiguous()
    W[0, dm // 2, 17] = float("inf")
    assert _value_loss(_spread(8, -40, -36), W, nt)[0] == float("inf")
    W[0, dm // 2, 17] = float("nan")
    loss = _value_loss(_spread(8, -40, -36), W, nt)[0]
    assert loss != loss


@pytest.mark.parametrize("lo", [0, -8, -80])
def test_gradient_elements_keep_their_own_precision(lo):
    """With one token, one output channel and identity rotations the generator's
    gradient is V_i u_j - V_j u_i with u = -2 (w V) w, through every product of
    the backward pass; each element against the size of its own two terms.  Four
    products of depth 128 are on the way (and a few single roundings)."""
    v, w = _spread(11, lo, 1) * 2.0 ** -36, _spread(12, lo, 1)
    cfg = optr.calib_config(1, 1, 1, 1)
    I, zero = torch.eye(D, dtype=F64), torch.zeros(1, D, dtype=F64)
    _, dA = optr.optr_calib_loss_grad(
        cfg, 1, *[x.cuda() for x in (zero.view(1, 1, D), zero, v.view(1, D),
                                     torch.zeros(1, dtype=torch.int32), w.view(1, 1, D), zero[0], I,
                                     torch.zeros(D, D, dtype=F64))], R_K=I.cuda())
    vs, ws = [[Fraction(x) for x in t.tolist()] for t in (v, w)]
    e = -sum(a * b for a, b in zip(vs, ws))
    for i, row in enumerate(dA.cpu().tolist()):
        for j, got in enumerate(row):
            a, b = vs[i] * 2 * e * ws[j], vs[j] * 2 * e * ws[i]
            assert abs(Fraction(got) - (a - b)) <= (4 * D + 16) * U * (abs(a) + abs(b))


@pytest.mark.parametrize("size", [1e3, 1e6])
def test_output_error_in_the_weak_directions_of_W(size):
    """hist_v[0] of a calibration whose value lies where a badly conditioned W_O is
    weak: the rows are size s_m (1, 1, 0, ..) + b_m and V = (x, -x, 0, ..), so that
    W V = x (W_m0 - W_m1), a difference that float64 forms exactly while the squares
    of W round at size^2."""
    nt, dm = 64, 1024
    gen = torch.Generator().manual_seed(21)
    W = torch.rand(1, dm, D, generator=gen, dtype=F64)
    W[..., :2] += size * torch.randn(1, dm, 1, generator=gen, dtype=F64)
    v = torch.zeros(D, dtype=F64)
    v[0], v[1] = 2.0 ** -36, -2.0 ** -36
    zeros, I = torch.zeros(1, D, dtype=F64), torch.eye(D, dtype=F64)
    cfg = optr.calib_config(1, dm, 1, nt, steps=1, select_every=1)
    *_, hist_v = optr.optr_calibrate_head(
        cfg, *[x.cuda() for x in (torch.zeros(nt, 1, D, dtype=F64), zeros, v.view(1, D),
                                  torch.zeros(nt, dtype=torch.int32), W)], R0_K=I.cuda(), R0_V=I.cuda())
    ref = _exact(v, W)
    # a term has the roundings of its two products, the square and the sums theirs
    assert abs(Fraction(hist_v[0].item()) - ref) <= (dm / 32 + nt / 256 + 32) * U * ref


@pytest.mark.parametrize("rows", [1, D])
def test_generator_with_nan(rows):
    """NaN in some rows of A - A^T gives a NaN loss; a generator without a finite
    row is out of the exponential's range."""
    A = torch.zeros(D, D, dtype=F64)
    A[:rows, 7] = float("nan")
    if rows == D:
        A[:] = float("nan")
    I, zeros = torch.eye(D, dtype=F64), torch.zeros(2, D, dtype=F64)
    args = [x.cuda() for x in (torch.ones(1, 1, D, dtype=F64), zeros, zeros + 0.5,
                               torch.ones(1, dtype=torch.int32), torch.ones(1, 3, D, dtype=F64),
                               zeros[0], I, A)]
    call = lambda: optr.optr_calib_loss_grad(optr.calib_config(1, 3, 2, 1), 1, *args, R_K=I.cuda())
    if rows == D:
        with pytest.raises(optr.OptrError):
            call()
    else:
        loss, _ = call()
        assert loss.isnan().all()
