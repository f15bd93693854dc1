"""GPU parity of the RoPElite search kernels (Algorithm 1 of the paper) against the float64
oracle.  Distances are fp32 sums over up to tens of thousands of causal pairs: relative tolerance
2e-4 (inputs are bf16 on both sides; the kernel's table is fp32).  The chosen chunk is an integer
decided by floating point: it must equal the oracle's choice whenever the oracle's best and
second-best distances differ by more than that tolerance, and must in any case be a chunk whose
oracle distance is within the tolerance of the minimum."""
import numpy as np
import pytest
import torch

from oracle import ropelite_oracle as R

pytestmark = pytest.mark.gpu

TOL = 2e-4


@pytest.fixture(scope="module")
def ek():
    from paper_2503_01586_b200 import binding
    binding.lib()
    return binding


def _acts(H, n, d_h, seed, graded=False):
    g = torch.Generator(device="cpu").manual_seed(seed)
    Q = torch.randn((H, n, d_h), generator=g)
    K = torch.randn((H, n, d_h), generator=g)
    if graded:       # per-head chunk energies in a scrambled, well separated order
        for h in range(H):
            order = torch.randperm(d_h // 2, generator=g)
            for rank, i in enumerate(order.tolist()):
                Q[h, :, 2 * i:2 * i + 2] *= 0.8 ** rank
    return Q.to(torch.bfloat16), K.to(torch.bfloat16)


@pytest.mark.parametrize("d_h,n", [(128, 150), (64, 203), (128, 1), (128, 4), (64, 65)])
def test_distances(ek, d_h, n):
    """Rows that end inside a thread's rows, key tiles with a ragged end, one token (all zero)."""
    H = 3
    Q, K = _acts(H, n, d_h, 100 + n)
    half = d_h // 2
    masks = [0, (1 << 3) | (1 << (half - 1)), (1 << half) - 1 - (1 << 5)]      # none, two, all but chunk 5
    got = ek.elitekv_ropelite_distances(Q.cuda(), K.cuda(), 10000.0,
                                        torch.from_numpy(np.array(masks, dtype=np.uint64).view(np.int64)).cuda()).cpu().double().numpy()
    for h in range(H):
        elite = [i for i in range(half) if (masks[h] >> i) & 1]
        want = R.distances(Q[h].double().numpy(), K[h].double().numpy(), elite, d_h)
        assert np.array_equal(np.isinf(got[h]), np.isinf(want))
        fin = np.isfinite(want)
        scale = max(float(np.max(want[fin])), 1e-30)
        assert np.all(np.abs(got[h][fin] - want[fin]) <= TOL * scale + 1e-6), (h, got[h][fin], want[fin])
    # no mask argument = nothing chosen yet
    got0 = ek.elitekv_ropelite_distances(Q.cuda(), K.cuda()).cpu().double().numpy()
    want0 = R.distances(Q[1].double().numpy(), K[1].double().numpy(), [], d_h)
    assert np.allclose(got0[1], want0, rtol=TOL, atol=1e-6)


@pytest.mark.parametrize("graded", [True, False])
def test_search(ek, graded):
    H, n, d_h, r = 4, 96, 128, 6
    Q, K = _acts(H, n, d_h, 7 + graded, graded)
    idx, trace = ek.elitekv_ropelite_search(Q.cuda(), K.cuda(), r, trace=True)
    torch.cuda.synchronize()
    idx, trace = idx.cpu().numpy(), trace.cpu().double().numpy()
    exact = 0
    for h in range(H):
        q, k = Q[h].double().numpy(), K[h].double().numpy()
        elite = []
        for rnd in range(r):
            want = R.distances(q, k, elite, d_h)           # the oracle's round on the GPU's own list so far
            fin = np.isfinite(want)
            assert np.array_equal(np.isinf(trace[rnd, h]), ~fin)
            assert np.allclose(trace[rnd, h][fin], want[fin], rtol=TOL, atol=1e-6)
            j = int(idx[h, rnd])
            assert j not in elite
            best = np.sort(want[fin])
            assert want[j] <= best[0] * (1 + TOL) + 1e-6      # a minimiser within the tolerance
            if best[1] > best[0] * (1 + 4 * TOL):
                assert j == int(np.argmin(want))              # a clear winner must be the oracle's
                exact += 1
            elite.append(j)
        if graded:
            assert elite == R.search(q, k, r, d_h)[0]
    assert exact >= H * r // 2
    # same inputs, same bits (fixed summation order)
    idx2, trace2 = ek.elitekv_ropelite_search(Q.cuda(), K.cuda(), r, trace=True)
    assert torch.equal(idx2.cpu(), torch.from_numpy(idx)) and torch.equal(trace2.cpu().double(), torch.from_numpy(trace))


@pytest.mark.parametrize("H,n,d_h,r,graded", [(2, 260, 128, 9, False), (2, 129, 64, 31, True), (40, 193, 64, 3, False)])
def test_search_with_kept_sums(ek, H, n, d_h, r, graded):
    """Calls beyond the small form keep R between rounds: tiles that end inside a block's rows and keys, both
    thread tiles, graded energies, whose norm falls so fast that R is summed afresh every few rounds, and all
    rounds but the last one.  Every round against the oracle on the GPU's own list so far."""
    Q, K = _acts(H, n, d_h, 31 + n, graded)
    idx, trace = ek.elitekv_ropelite_search(Q.cuda(), K.cuda(), r, trace=True)
    torch.cuda.synchronize()
    idx, trace = idx.cpu().numpy(), trace.cpu().double().numpy()
    for h in {0, H - 1}:
        q, k = Q[h].double().numpy(), K[h].double().numpy()
        elite = []
        for rnd in range(r):
            want = R.distances(q, k, elite, d_h)
            fin = np.isfinite(want)
            assert np.array_equal(np.isinf(trace[rnd, h]), ~fin)
            assert np.allclose(trace[rnd, h][fin], want[fin], rtol=TOL, atol=1e-6)
            assert want[idx[h, rnd]] <= want[fin].min() * (1 + TOL) + 1e-6
            elite.append(int(idx[h, rnd]))
        assert len(set(elite)) == r


@pytest.mark.parametrize("H,n,d_h,r", [(24, 450, 128, 2), (32, 400, 128, 1), (5, 161, 128, 3), (160, 193, 64, 2), (20, 400, 64, 1),
                                       (3, 130, 64, 2), (33, 300, 128, 1), (64, 521, 128, 4), (64, 300, 64, 5)])
def test_search_by_every_form(ek, H, n, d_h, r):
    """Few rounds run on resident operands (16, 8 and 4 rows per thread at both head dims) or staged ones that keep
    nothing; the last two calls keep R over several key tiles of an item and rounds that are neither the first nor the last.
    Distances against the float64 oracle on the GPU's own list so far, to the 1e-5 of the single rounds (fp32 sums of
    up to n (n + 1) / 2 terms of relative rounding 2^-24 each, through chains of at most ~200 terms)."""
    Q, K = _acts(H, n, d_h, 77 + n)
    idx, trace = ek.elitekv_ropelite_search(Q.cuda(), K.cuda(), r, trace=True)
    idx, trace = idx.cpu().numpy(), trace.cpu().double().numpy()
    for h in {0, H - 1}:
        q, k = Q[h].double().numpy(), K[h].double().numpy()
        for rnd in range(r):
            want = R.distances(q, k, idx[h, :rnd].tolist(), d_h)
            fin = np.isfinite(want)
            assert np.array_equal(np.isinf(trace[rnd, h]), ~fin)
            assert np.allclose(trace[rnd, h][fin], want[fin], rtol=1e-5, atol=1e-6)
            # (2-norm of the errors: 5e-8 on every form, whether R is summed or kept)
            assert np.linalg.norm(trace[rnd, h][fin] - want[fin]) <= 2e-7 * np.linalg.norm(want[fin])
            assert want[idx[h, rnd]] <= want[fin].min() * (1 + 1e-5)


@pytest.mark.parametrize("d_h", [64, 128])
def test_search_of_values_that_are_not_finite(ek, d_h):
    """An infinity, a NaN and large finite values: a search that keeps R gives what one gives that sums it in every round (which
    the least workspace makes it do), place by place."""
    H, n, r = 4, 300, 9
    Q, K = (x.cuda() for x in _acts(H, n, d_h, 21))
    Q[0, 200, 5] = float("inf")
    K[1, 17, 2] = float("nan")
    Q[2] *= 1e30
    big = ek.elitekv_ropelite_workspace_size(H, n, d_h)
    least = ek.elitekv_ropelite_workspace_size_rounds(H, n, d_h, 0)
    assert least < ek.elitekv_ropelite_workspace_size_rounds(H, n, d_h, r) <= big
    (i, t), (i0, t0) = (ek.elitekv_ropelite_search(Q, K, r, trace=True, workspace=torch.empty(size, dtype=torch.uint8, device="cuda"))
                        for size in (big, least))
    assert torch.equal(i, i0) and torch.allclose(t, t0, rtol=1e-6, equal_nan=True)
    assert torch.isnan(t[:, 1]).any() and torch.isfinite(t[0, 2:]).all()


def test_search_of_a_head_too_long_to_keep(ek):
    """A head of 23000 tokens needs more than the scratch for its sums: every round sums R, and is the single round for the
    chunks chosen so far."""
    n, d_h, r = 23000, 64, 3
    g = torch.Generator(device="cuda").manual_seed(8)
    Q, K = (torch.randn((1, n, d_h), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    assert ek.elitekv_ropelite_workspace_size(1, n, d_h) < 1 << 28
    idx, trace = ek.elitekv_ropelite_search(Q, K, r, trace=True)
    mask = 0
    for rnd in range(r):
        dist = ek.elitekv_ropelite_distances(Q, K, elite_mask=torch.tensor([mask], dtype=torch.int64, device="cuda"))
        assert torch.allclose(trace[rnd], dist, rtol=1e-6)
        mask |= 1 << int(idx[0, rnd])


@pytest.mark.parametrize("H,n,d_h,r", [(3, 300, 128, 5), (40, 260, 64, 4), (2, 90, 64, 3)])
def test_search_in_any_workspace(ek, H, n, d_h, r):
    """From the least workspace on a call runs the fastest way that fits, with the same distances (sums in another order:
    fp32, 1e-6); less is refused."""
    Q, K = (x.cuda() for x in _acts(H, n, d_h, 5 + n))
    least = ek.elitekv_ropelite_workspace_size_rounds(H, n, d_h, 0)
    sizes = [least] + [ek.elitekv_ropelite_workspace_size_rounds(H, n, d_h, k) for k in (1, r)] + [ek.elitekv_ropelite_workspace_size(H, n, d_h)]
    idx, trace = ek.elitekv_ropelite_search(Q, K, r, trace=True)
    dist = ek.elitekv_ropelite_distances(Q, K)
    for size in sizes + [(sizes[0] + sizes[2]) // 2]:
        ws = torch.full((size + 256,), 0x5a, dtype=torch.uint8, device="cuda")
        i, t = ek.elitekv_ropelite_search(Q, K, r, trace=True, workspace=ws[:size])
        assert torch.equal(i, idx) and torch.allclose(t, trace, rtol=1e-6, atol=1e-6)
        assert torch.allclose(ek.elitekv_ropelite_distances(Q, K, workspace=ws[:size]), dist, rtol=1e-6, atol=1e-6)
        assert torch.all(ws[size:] == 0x5a)
    with pytest.raises(ek.ElitekvError) as e:
        ek.elitekv_ropelite_search(Q, K, r, workspace=ws[:least - 1])
    assert e.value.code == ek.ERR_WORKSPACE_TOO_SMALL


def test_search_energy_in_one_chunk(ek):
    """R is that chunk's D alone: it goes first, and what is left of R is nothing, not a rounding error."""
    Q, K = _acts(1, 200, 128, 5)
    Q[:, :, :14] = 0
    Q[:, :, 16:] = 0
    idx, trace = ek.elitekv_ropelite_search(Q.cuda(), K.cuda(), 4, trace=True)
    assert idx[0].tolist() == [7, 0, 1, 2]
    assert torch.all(trace[1:][torch.isfinite(trace[1:])] == 0)


def test_search_in_groups_of_heads(ek):
    """More heads than the scratch holds at a time (1 GiB; what one head more takes, from the sizes of small calls, counts
    item results too, so that the seam lies within a head of it): the heads on both sides of the seam and the last one as
    in calls of their own (sums in another order where the call's form differs: fp32, 1e-6)."""
    H, n, d_h, r = 100, 2048, 128, 2
    size = lambda heads: ek.elitekv_ropelite_workspace_size_rounds(heads, n, d_h, r)
    seam = (1 << 30) // (size(41) - size(40))
    assert seam + 2 < H and size(H) < (1 << 30) + (1 << 25)
    g = torch.Generator(device="cuda").manual_seed(3)
    Q, K = (torch.randn((H, n, d_h), generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    idx, trace = ek.elitekv_ropelite_search(Q, K, r, trace=True)
    dist = ek.elitekv_ropelite_distances(Q, K)
    for h in (0, seam - 2, seam - 1, seam, seam + 1, seam + 2, H - 1):
        one, t = ek.elitekv_ropelite_search(Q[h:h + 1].contiguous(), K[h:h + 1].contiguous(), r, trace=True)
        assert torch.equal(one[0], idx[h])
        assert torch.allclose(t[:, 0], trace[:, h], rtol=1e-6) and torch.allclose(dist[h], trace[0, h], rtol=1e-6)


def test_waits_that_run_out_are_reported(ek):
    """Kernels that wait for copies which are never made: no index is made up, every round of both heads ends, and the
    context stays usable."""
    Q, K = (x.cuda() for x in _acts(2, 130, 64, 9))
    good = ek.elitekv_ropelite_search(Q, K, 2, trace=True)
    idx, trace = ek.elitekv_selftest_search_timeout(Q, K)
    assert torch.all(idx == -1) and torch.all(torch.isnan(trace))
    again = ek.elitekv_ropelite_search(Q, K, 2, trace=True)
    assert all(torch.equal(a, b) for a, b in zip(good, again)) and torch.all(again[0] >= 0)


def test_argument_checks(ek):
    Q, K = _acts(1, 8, 32, 1)
    with pytest.raises(ek.ElitekvError) as e:        # d_h = 32 is not covered
        ek.elitekv_ropelite_distances(Q.cuda(), K.cuda())
    assert e.value.code == ek.ERR_UNSUPPORTED_SHAPE
    Q, K = _acts(1, 8, 64, 1)
    with pytest.raises(ek.ElitekvError) as e:        # more rounds than chunks
        ek.elitekv_ropelite_search(Q.cuda(), K.cuda(), 33)
    assert e.value.code == ek.ERR_INVALID_ARG
