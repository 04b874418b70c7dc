"""The kernel for three to eight activation vectors where its arithmetic and its division of work can go wrong: every vector's result is bit for
bit what llvq_gemv writes for it alone (which the parity tests hold against the oracle)."""
import numpy as np
import pytest
import torch

from helpers import GAIN, make_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2609_02652_b200 import binding

    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.create(0)
    yield c
    c.close()


def one_by_one(B, ctx, case, buf, X):
    return torch.stack([B.gemv(ctx, 0, buf, case.d_scale, GAIN, x.contiguous(), case.rows, 24 * case.nb) for x in X])


# rows and blocks at the edges of a row group, a tile and a panel; shares cut at row groups and shares that cross them; one unit a warp and many
@pytest.mark.parametrize("rows,nb", [(1, 1), (31, 2), (33, 3), (64, 5), (65, 67), (500, 342), (1024, 107), (4096, 171), (3000, 33), (40, 1500), (20000, 70)])
@pytest.mark.parametrize("batch", [3, 4, 5, 8])
def test_every_vector_as_alone(B, ctx, rows, nb, batch):
    case = make_case(rows, 24 * nb, seed=rows + nb)
    buf = B.expand(ctx, 0, case.d_codes, rows, nb)
    X = torch.stack([torch.roll(case.d_x, 7 * j) * (0.25 * 3.0**j) for j in range(batch)]).half().contiguous()
    want = one_by_one(B, ctx, case, buf, X)
    for _ in range(2):                               # the second launch finds the accumulators clean
        assert torch.equal(B.gemv_batch(ctx, buf, case.d_scale, GAIN, X, rows, 24 * nb), want)
    B.status(ctx)


# the builds for six and for eight, filled and with a vector to spare: one launch whose rows end in a tile of one, two and three blocks
@pytest.mark.parametrize("rows,nb", [(33, 7), (500, 341), (4096, 170), (20000, 70)])
@pytest.mark.parametrize("batch", [2, 6, 7])
def test_every_vector_of_the_other_builds(B, ctx, rows, nb, batch):
    test_every_vector_as_alone(B, ctx, rows, nb, batch)


# Twice the fixed-point activation, given a largest |x| in [2, 4): x = units / 2^28.  The halves of 32656, 32688, 32720 and 32752 are kept in another
# form; 32640 and 32768 are the numbers beside them; 32624 everywhere is the largest sum of low halves, -32896 the least
@pytest.mark.parametrize("units", [(32656, 32688, 32720, 32752), (32640, 32656, 32768, -32656), (32624,), (32640,), (65536 + 32640, 98304 - 64, 131072 - 64)])
@pytest.mark.parametrize("nb", [9, 70, 171])
@pytest.mark.parametrize("batch", [3, 8])
def test_halves_of_activations(B, ctx, oracle, units, nb, batch):
    rows = 96
    case = make_case(rows, 24 * nb, seed=nb)
    buf = B.expand(ctx, 0, case.d_codes, rows, nb)
    rng = np.random.default_rng(len(units) + nb)
    special = np.float16(np.array(units, np.float64) / 2.0**28)
    assert (special.astype(np.float64) * 2.0**28 == np.array(units)).all()
    xs = np.stack([case.x] * batch)
    xs[0] = rng.choice(special, 24 * nb)             # all of the vector but its largest
    xs[0][5] = 3.0
    at = rng.integers(0, 24 * nb, max(1, nb // 8))   # a few among ordinary ones
    xs[batch - 1] = np.clip(xs[batch - 1], -2, 2)
    xs[batch - 1][at] = rng.choice(special, at.size)
    xs[batch - 1][0] = 3.0
    X = torch.from_numpy(xs).cuda()
    got = B.gemv_batch(ctx, buf, case.d_scale, GAIN, X, rows, 24 * nb)
    assert torch.equal(got, one_by_one(B, ctx, case, buf, X))
    # f32 constants, sums of at most four blocks and result: a few 2^-24 of a row's sum of magnitudes; activations rounded to 2^-27
    W = oracle.dequant(case.codes, rows, nb, case.row_scale, GAIN)
    for j in (0, batch - 1):
        x = xs[j].astype(np.float64)
        assert (np.abs(got[j].cpu().numpy() - W @ x) <= 2.0**-22 * (np.abs(W) @ np.abs(x)) + 2.0**-28 * np.abs(W).sum(1)).all()
    B.status(ctx)


@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("batch", [4, 7])
def test_one_vector_that_is_not_finite(B, ctx, bad, batch):
    """Its rows are NaN, the others' are theirs, and the next launch finds the accumulators clean."""
    case = make_case(200, 24 * 53, seed=9)
    buf = B.expand(ctx, 0, case.d_codes, case.rows, case.nb)
    X = torch.stack([torch.roll(case.d_x, j) for j in range(batch)]).contiguous()
    want = one_by_one(B, ctx, case, buf, X)
    broken = X.clone()
    broken[1, 17] = bad
    y = B.gemv_batch(ctx, buf, case.d_scale, GAIN, broken, case.rows, 24 * case.nb)
    assert y[1].isnan().all() and torch.equal(y[[0, 2, batch - 1]], want[[0, 2, batch - 1]])
    assert torch.equal(B.gemv_batch(ctx, buf, case.d_scale, GAIN, X, case.rows, 24 * case.nb), want)
    B.status(ctx)


@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("batch", [2, 3, 5, 6, 8])
def test_not_finite_in_every_build(B, ctx, bad, batch):
    """What is true of a vector that is not finite does not depend on how many go with it, nor on where among them it is."""
    case = make_case(500, 24 * 53, seed=10)
    buf = B.expand(ctx, 0, case.d_codes, case.rows, case.nb)
    X = torch.stack([torch.roll(case.d_x, j) for j in range(batch)]).contiguous()
    want = one_by_one(B, ctx, case, buf, X)
    for at in (0, batch - 1):
        broken = X.clone()
        broken[at, 24 * 53 - 1 - at] = bad
        y = B.gemv_batch(ctx, buf, case.d_scale, GAIN, broken, case.rows, 24 * case.nb)
        others = [j for j in range(batch) if j != at]
        assert y[at].isnan().all() and torch.equal(y[others], want[others])
    assert torch.equal(B.gemv_batch(ctx, buf, case.d_scale, GAIN, X, case.rows, 24 * case.nb), want)
    B.status(ctx)


@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("layout", ["PLANES", "ONEHOT", "PLANES13", "PLANES10X"])
def test_not_finite_in_every_layout(B, ctx, bad, layout):
    """One vector alone: y is NaN, and the next launch finds the accumulators clean."""
    case = make_case(200, 24 * 53, seed=11)
    buf = B.expand(ctx, getattr(B, layout), case.d_codes, case.rows, case.nb)
    call = lambda x: B.gemv(ctx, getattr(B, layout), buf, case.d_scale, GAIN, x, case.rows, 24 * case.nb)  # noqa: E731
    want = call(case.d_x)
    for at in (0, 700, 24 * 53 - 1):
        broken = case.d_x.clone()
        broken[at] = bad
        assert call(broken).isnan().all()
    assert want.isfinite().all() and torch.equal(call(case.d_x), want)
    B.status(ctx)
