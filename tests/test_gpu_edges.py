"""GPU parity at the sizes where a kernel's tiles, remainders and dispatch lines lie, against the
float64 oracle on the same bytes (tolerances: tests/harness.py)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import elitekv_oracle as O
from paper_2503_01586_b200 import inputs as gen

from . import harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ek():
    from paper_2503_01586_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("n_items", [1, 4, 5, 16, 17, 33])
def test_combine_items_per_sequence(ek, n_items):
    """The combine holds 16 items' statistics in half a warp and 4 partial results in flight: one
    sequence of n_items one-tile items (the two-pass kernel's tile is 128 tokens), and a second row
    in the same warp with fewer."""
    w = gen.shrink(gen.LLAMA7B_75, B=2, ctx=128 * n_items)
    st = H.setup(w, lens=[128 * n_items, 65], decode_kernel=2)
    _, tile, n_workers, max_items, overhead = ek.elitekv_decode_plan_info(st.layer, st.cache, 2)
    _, first, _ = ek.elitekv_plan_workers(st.lens_dev, tile, n_workers, max_items, overhead)
    assert first.tolist() == [0, n_items, n_items + 1]
    H.check_parity(st, H.run_decode(st), H.sample_units(st, 24, seed=n_items))


# ------------------------------------------------------------------ RoPElite search
@pytest.mark.parametrize("heads,n,d_h", [(2, 127, 64), (2, 128, 128), (2, 129, 128), (2, 257, 64), (2, 520, 128),
                                         (300, 257, 64)])
def test_ropelite_distances_tile_edges(ek, heads, n, d_h):
    """Rows and keys around the 128 x 128 tile, key tiles in items of their own and (many heads) several
    per item, no mask / some chunks / all but one chosen.  fp32 sums of up to n (n + 1) / 2 terms of
    relative rounding 2^-24 each, added through chains of at most ~200 terms: 1e-5 is ample."""
    from oracle import ropelite_oracle as R
    g = torch.Generator().manual_seed(heads + n)
    Q, K = (torch.randn((heads, n, d_h), generator=g).to(torch.bfloat16) for _ in range(2))
    half = d_h // 2
    full = (1 << half) - 1
    masks = [0, 5 | (1 << (half - 1))] + [full & ~2] * (heads - 2)
    dev = torch.from_numpy(np.array(masks, dtype=np.uint64).view(np.int64)).cuda()
    got = ek.elitekv_ropelite_distances(Q.cuda(), K.cuda(), elite_mask=dev).cpu().double().numpy()
    for h in (0, 1, heads - 1):
        elite = [i for i in range(half) if (masks[h] >> i) & 1]
        want = R.distances(Q[h].double().numpy(), K[h].double().numpy(), elite, d_h)
        fin = np.isfinite(want)
        assert np.array_equal(np.isinf(got[h]), ~fin)
        assert np.allclose(got[h][fin], want[fin], rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("heads,n,d_h", [(1, 1, 64), (2, 16, 128), (3, 17, 64), (37, 64, 128), (75, 64, 64), (2, 65, 128), (18, 128, 128),
                                         (19, 128, 64), (75, 63, 128), (6, 152, 64), (5, 161, 128), (40, 152, 128), (48, 193, 64),
                                         (33, 300, 128), (64, 128, 64)])
def test_ropelite_distances_of_every_form(ek, heads, n, d_h):
    """The form for small calls (16 rows a block, 64 keys at a time) up to its lines at 64 and 128 tokens,
    and 4 and 8 rows per thread with ragged row tiles and key tiles; every chunk free, some chosen,
    two left.  Tolerance as above."""
    from oracle import ropelite_oracle as R
    g = torch.Generator().manual_seed(heads + n)
    Q, K = (torch.randn((heads, n, d_h), generator=g).to(torch.bfloat16) for _ in range(2))
    half = d_h // 2
    full = (1 << half) - 1
    masks = [(0, 9 | (1 << (half - 2)), full & ~(2 | (1 << (half - 1))))[h % 3] for h in range(heads)]
    dev = torch.from_numpy(np.array(masks, dtype=np.uint64).view(np.int64)).cuda()
    got = ek.elitekv_ropelite_distances(Q.cuda(), K.cuda(), elite_mask=dev).cpu().double().numpy()
    for h in {0, heads // 2, heads - 1}:
        want = R.distances(Q[h].double().numpy(), K[h].double().numpy(), [i for i in range(half) if (masks[h] >> i) & 1], d_h)
        fin = np.isfinite(want)
        assert np.array_equal(np.isinf(got[h]), ~fin)
        assert np.allclose(got[h][fin], want[fin], rtol=1e-5, atol=1e-6)

def test_ropelite_search_down_to_the_last_chunk(ek):
    """All d_h / 2 rounds: every chunk is chosen once and the last free one costs nothing."""
    g = torch.Generator().manual_seed(3)
    Q, K = (torch.randn((2, 140, 64), generator=g).to(torch.bfloat16).cuda() for _ in range(2))
    idx, trace = ek.elitekv_ropelite_search(Q, K, 32, trace=True)
    assert sorted(idx[0].tolist()) == list(range(32)) and sorted(idx[1].tolist()) == list(range(32))
    assert trace[31][torch.isfinite(trace[31])].abs().max().item() == 0.0


# ------------------------------------------------------------------ query preparation and the step's front end
@pytest.mark.parametrize("B", [1, 16, 17, 32, 33, 64, 65])
@pytest.mark.parametrize("shape", [dict(), dict(n_h=3, d_h=44, r=5, d_c=136, d=128), dict(n_h=4, d_h=64, r=32, d_c=128, d=256)],
                         ids=["7b", "odd", "all-elite"])
def test_absorb_row_tiles(ek, B, shape):
    """1, 2 and 4 row tiles per block, several groups; a head dim that is no multiple of 8 and a latent
    that ends inside a 128-wide slab; no un-rotated dim at all."""
    w = replace(gen.LLAMA7B_75, B=B, seed=900 + B, **shape)
    idx = gen.elite_index_sets(w)
    W_uk, W_uv = gen.up_projections(w, "cuda")
    layer = ek.Layer(w.n_h, w.d_h, w.r, w.d_c, idx, W_uk, W_uv, 300)
    q = gen.queries(w, "cuda")
    q_pos = (torch.arange(B, dtype=torch.int32) * 37 % 300).cuda()
    q_rope, q_abs = ek.elitekv_absorb_query(layer, q, q_pos)
    assert ek.elitekv_check_status(layer) == 0
    for b in {0, B // 2, B - 1}:
        want_rope, want_abs = O.absorb_query(H.f64(q[b]), int(q_pos[b]), idx.numpy().astype(np.int64), H.f64(W_uk), w.d_h, w.rope_base)
        # bf16 results of exact products with fp32 sums: half a unit of 2^-8 relative to the row's largest entry
        assert np.max(np.abs(H.f64(q_rope[b]) - want_rope)) <= 2.0 ** -8 * np.max(np.abs(want_rope))
        assert np.max(np.abs(H.f64(q_abs[b]) - want_abs)) <= 2.0 ** -8 * np.max(np.abs(want_abs)) + 1e-30


@pytest.mark.parametrize("B,pair_mode,d_h", [(3, 0, 128), (40, 1, 128), (5, 1, 44)])
def test_absorb_takes_nothing_from_elite_dims(ek, B, pair_mode, d_h):
    """q_abs sums over the un-rotated dims only: infinities and NaN in the elite dims (pairs of neighbours
    or half a head apart) leave it as it is with zeros there, bit for bit."""
    w = replace(gen.LLAMA7B_75, B=B, n_h=3, d_h=d_h, r=5, seed=70 + B)
    idx = gen.elite_index_sets(w)
    layer = ek.Layer(w.n_h, d_h, w.r, w.d_c, idx, *gen.up_projections(w, "cuda"), 300, pair_mode=pair_mode)
    q = gen.queries(w, "cuda")
    q_pos = (torch.arange(B, dtype=torch.int32) % 300).cuda()
    at = idx.long().cuda()
    dims = torch.cat([2 * at, 2 * at + 1] if pair_mode == 0 else [at, at + d_h // 2], dim=1).expand(B, -1, -1)
    got = []
    for v in (0.0, float("inf"), float("-inf"), float("nan")):
        got.append(ek.elitekv_absorb_query(layer, q.scatter(2, dims, v), q_pos)[1])
    assert torch.isfinite(got[0]).all() and got[0].any()
    assert all(torch.equal(got[0], x) for x in got[1:])

@pytest.mark.parametrize("B", [1, 33, 200])
def test_step_front_end_equals_the_three_calls(ek, B):
    """One launch for append, plan and query preparation: more tokens than append blocks (200), and
    batches of one and of several row tiles, bit for bit as the separate calls."""
    w = gen.shrink(gen.SWEEP_875, B=B, ctx=70)
    lens = [1 + 17 * b % 70 for b in range(B)]
    out = []
    for single in (False, True):
        st = H.setup(w, lens=lens, fill=False)
        st.rope_plane.normal_(generator=torch.Generator(device="cuda").manual_seed(1))
        st.latent_plane.normal_(generator=torch.Generator(device="cuda").manual_seed(2))
        last = torch.from_numpy(st.starts[1:] - 1).cuda()
        k_e, c, seq, pos = (x[last].contiguous() for x in (st.k_e, st.c, st.seq_id, st.pos))
        q_rope = torch.zeros((B, w.n_h, 2 * w.r), dtype=torch.bfloat16, device="cuda")
        q_abs = torch.zeros((B, w.n_h, w.d_c), dtype=torch.bfloat16, device="cuda")
        o = torch.zeros((B, w.n_h, w.d_h), dtype=torch.bfloat16, device="cuda")
        if single:
            ek.elitekv_decode_step(st.layer, st.cache, k_e, c, seq, pos, st.q, st.lens_dev, q_rope, q_abs, st.workspace, o)
        else:
            ek.elitekv_append(st.layer, st.cache, k_e, c, seq, pos)
            ek.elitekv_absorb_query(st.layer, st.q, pos, q_rope, q_abs)
            ek.elitekv_decode(st.layer, st.cache, q_rope, q_abs, st.lens_dev, st.workspace, o)
        assert ek.elitekv_check_status(st.layer) == 0
        out.append((st.rope_plane, st.latent_plane, q_rope, q_abs, o))
    for a, b in zip(*out):
        assert torch.equal(a, b)


# ------------------------------------------------------------------ cluster kernel (decode_kernel = 4)
CLUSTER_SHAPES = {"c2": gen.SWEEP_875, "c4": gen.LLAMA7B_75, "c5": gen.LLAMA13B_75, "c8": gen.SWEEP_50,
                  "c4-slrd": gen.SWEEP_75_SLRD}


@pytest.mark.parametrize("paged", [False, True])
@pytest.mark.parametrize("shape", CLUSTER_SHAPES)
def test_cluster_kernel_tile_edges(ek, shape, paged):
    """One tile (one stream only), two and three tiles, the 16-token steps of a ragged last tile, an
    empty sequence, and every cluster size."""
    lens = [64, 1, 15, 17, 63, 65, 128, 129, 200, 0, 413]
    w = gen.shrink(CLUSTER_SHAPES[shape], B=len(lens), ctx=413)
    if paged:
        w = replace(w, paged=True, page_size=64)
    st = H.setup(w, lens=lens, decode_kernel=4)
    assert ek.elitekv_decode_plan_info(st.layer, st.cache, len(lens))[0] == 4
    out = H.run_decode(st)
    assert not out[9].any()
    H.check_parity(st, out, [u for u in H.sample_units(st, 120, seed=4) if u[0] != 9] + [(0, 0), (1, w.n_h - 1), (10, w.n_h // 2)])


@pytest.mark.parametrize("shape", ["c4", "c5"])
def test_cluster_kernel_many_items_per_worker(ek, shape):
    """Workers walk many short items: queries replaced, accumulators merged and reused, statistics
    slots coming round; and one sequence cut over all workers."""
    w = gen.shrink(CLUSTER_SHAPES[shape], B=301, ctx=300)
    lens = [1 + (37 * i) % 300 for i in range(301)]
    st = H.setup(w, lens=lens, decode_kernel=4)
    H.check_parity(st, H.run_decode(st), H.sample_units(st, 64))
    st = H.setup(gen.shrink(CLUSTER_SHAPES[shape], B=1, ctx=15000), lens=[15000], decode_kernel=4)
    H.check_parity(st, H.run_decode(st), H.sample_units(st, 3))


@pytest.mark.parametrize("page_size", [64, 256])
def test_cluster_kernel_pages_and_bad_page(ek, page_size):
    """Several tiles per page, more than 32 tiles (rows are looked up 32 at a time), and a page id outside
    the pool: recorded, and the other sequences' results untouched."""
    w = replace(gen.shrink(gen.LLAMA7B_75, B=3, ctx=9000), paged=True, page_size=page_size)
    st = H.setup(w, lens=[9000, 2500, 64], decode_kernel=4)
    good = H.run_decode(st).clone()
    H.check_parity(st, good, H.sample_units(st, 8))
    st.page_table[1, 2] = st.cache.num_pages + 5
    q_rope, q_abs = ek.elitekv_absorb_query(st.layer, st.q, st.q_pos)
    out = ek.elitekv_decode(st.layer, st.cache, q_rope, q_abs, st.lens_dev, st.workspace)
    assert ek.elitekv_check_status(st.layer) == ek.ERR_BAD_PAGE
    assert ek.elitekv_last_status_detail(st.layer)[:2] == (1, st.cache.num_pages + 5)
    assert torch.equal(out[0], good[0]) and torch.equal(out[2], good[2])


@pytest.mark.parametrize("mode", ["scaled", "planted"])
def test_cluster_kernel_peaked(ek, mode):
    """The reference maximum moves inside items, in one stream and not in the other."""
    from .test_gpu_peaked import _run
    assert _run(ek, "7b", mode, 4) == 4


@pytest.mark.parametrize("shape", CLUSTER_SHAPES)
def test_cluster_kernel_tiles_without_a_finite_score(ek, shape):
    """Keys that give one head scores of -inf in whole 64-token tiles (finite bf16 rope dims whose fp32
    products overflow) weigh nothing, wherever the tile lies in its item: the head's output is that of
    the other tokens.  The plan makes items of one, two and three tiles."""
    B, h = 220, 3
    w = gen.shrink(CLUSTER_SHAPES[shape], B=B, ctx=192)
    idx = gen.elite_index_sets(w)
    tab = torch.zeros((194, w.d_h // 2, 2), device="cuda")
    tab[..., 0] = 1.0                                      # no rotation: signs below are those of the scores
    dead = [(), (0,), (1,), (2,), (0, 1), (1, 2)]          # tiles without a finite score, by sequence

    def edit(st):
        q = st.q[:, h].float()
        at = idx[h].long().cuda()
        qe = torch.stack([q[:, 2 * at], q[:, 2 * at + 1]], dim=2)              # [B][r][2]
        qe = torch.where(qe < 0, -2.0, 2.0)
        st.q[:, h, 2 * at], st.q[:, h, 2 * at + 1] = qe[..., 0].to(torch.bfloat16), qe[..., 1].to(torch.bfloat16)
        for b in range(B):
            for t in dead[b % len(dead)]:
                lo = int(st.starts[b]) + 64 * t
                st.k_e[lo:lo + 64, h] = (-3e38 * torch.sign(qe[b])).to(torch.bfloat16)

    st = H.setup(w, lens=[192] * B, decode_kernel=4, cos_sin=tab, edit_tokens=edit)
    out = H.run_decode(st)
    _, tile, n_workers, max_items, overhead = ek.elitekv_decode_plan_info(st.layer, st.cache, B)
    first = ek.elitekv_plan_workers(st.lens_dev, tile, n_workers, max_items, overhead)[1]
    assert first.diff().min().item() == 1                  # some sequences are one item of three tiles
    assert torch.isfinite(out).all()
    W_uk, W_uv, dn = H.f64(st.W_uk), H.f64(st.W_uv), w.d_h - 2 * w.r
    at = idx[h].numpy().astype(np.int64)
    el = np.stack([2 * at, 2 * at + 1], axis=1).reshape(-1)
    rest = np.setdiff1d(np.arange(w.d_h), el)
    for b in range(0, 24):
        lo = int(st.starts[b])
        keep = np.concatenate([np.arange(64 * t, 64 * t + 64) for t in range(3) if t not in dead[b % len(dead)]])
        q, c, k = H.f64(st.q[b, h]), H.f64(st.c[lo:lo + 192])[keep], H.f64(st.k_e[lo:lo + 192, h])[keep].reshape(len(keep), -1)
        ck, cv = (c[:, :st.d_ck], c[:, st.d_ck:]) if st.d_ck else (c, c)
        s = (k @ q[el] + ck @ (W_uk[:, h * dn:(h + 1) * dn] @ q[rest])) / w.d_h ** 0.5
        p = np.exp(s - s.max())
        want = (p / p.sum()) @ cv @ W_uv[:, h * w.d_h:(h + 1) * w.d_h]
        assert np.linalg.norm(H.f64(out[b, h]) - want) <= H.REL_L2_TOL * np.linalg.norm(want)

def test_cluster_kernel_refuses_uncovered_shapes(ek):
    w = replace(gen.LLAMA7B_75, B=2, ctx=64, n_h=24)          # 384 rope dims: clusters of three are not built
    with pytest.raises(ek.ElitekvError) as e:
        H.setup(w, lens=[5, 5], decode_kernel=4)
    assert e.value.code == ek.ERR_UNSUPPORTED_SHAPE


@pytest.mark.parametrize("lens", [[16], [17], [1000], [15, 16, 9000]])
def test_generic_kernel_item_edges(ek, lens):
    """Items of 16 tokens, a ragged last one, more items than a warp has lanes in the combine, and
    contexts long enough for larger pieces."""
    w = gen.shrink(gen.TINY, B=len(lens), ctx=max(lens))
    st = H.setup(w, lens=lens)
    assert ek.elitekv_decode_plan_info(st.layer, st.cache, len(lens))[:2] == (1, 16)
    H.check_parity(st, H.run_decode(st), H.all_units(st))


# ------------------------------------------------------------------ projection, paired forms
# one small layer per property: 256 columns of rope and latent side by side in a tile (128 + 128), table
# rows as long as a buffer holds (half = 64) and longer (half = 96, read directly), the smallest depth
PAIR_SHAPES = {
    "7b": (gen.LLAMA7B_75, 4096),
    "split-tile": (replace(gen.LLAMA7B_75, n_h=16, r=4, d_c=128), 448),
    "wide-heads": (replace(gen.LLAMA7B_75, n_h=16, d_h=192, r=8, d_c=256), 512),
}


@pytest.mark.parametrize("shape,T", [("7b", 1153), ("7b", 2304), ("7b", 2305), ("split-tile", 9473), ("split-tile", 18945),
                                     ("wide-heads", 4737), ("wide-heads", 9473)])
@pytest.mark.parametrize("paged", [False, True])
def test_project_append_paired_forms(ek, shape, T, paged):
    """Calls on both sides of the lines between the forms (one tile of 128 x 128 per block; pairs of
    blocks with 256 or 512 tokens x 256 columns), with ragged last token tiles."""
    from .test_gpu_parity import _projection_case
    w, d = PAIR_SHAPES[shape]
    lens = [T - 200, 137, 63]
    _projection_case(ek, gen.shrink(w, B=3, ctx=max(lens)), d, lens, paged, T)


@pytest.mark.parametrize("n", [1, 15, 16, 17, 4096, 16 * 256 * 512 * 4 + 16 * 300 + 5])
def test_copy_both_ways(ek, n):
    """Bytes below, at and above one 16-byte request, and more than one round of the largest grid;
    neighbouring bytes stay as they are."""
    host = torch.randint(0, 256, (n,), dtype=torch.uint8).pin_memory()
    dev = torch.full((n + 16,), 7, dtype=torch.uint8, device="cuda")
    back = torch.full((n + 16,), 9, dtype=torch.uint8).pin_memory()
    ek.elitekv_copy(dev[:n], host)
    ek.elitekv_copy(back[:n], dev[:n])
    torch.cuda.synchronize()
    assert torch.equal(dev[:n].cpu(), host) and torch.equal(back[:n], host)
    assert (dev[n:] == 7).all() and (back[n:] == 9).all()


@pytest.mark.parametrize("graph", [False, True])
def test_step_runner_keeps_its_pinned_buffers_until_the_step_is_through(ek, graph):
    """A runner that goes away with a step under way (behind 50 ms of other work) gives its pinned buffers
    back when the step has read and written them, not before."""
    w = gen.shrink(gen.TINY, B=2, ctx=20)
    st = H.setup(w, lens=[20, 7])
    run = ek.DecodeStepRunner(st.layer, st.cache, 2, "cuda", graph=graph)
    for k, v in (("q", st.q), ("seq_id", torch.arange(2, dtype=torch.int32)), ("pos", st.lens - 1), ("lens", st.lens)):
        run.host[k].copy_(v.cpu().view(run.host[k].shape))
    for _ in range(3):
        run.run()
    torch.cuda._sleep(100_000_000)
    run.run(wait=False)
    stream = torch.cuda.current_stream()
    assert not stream.query()
    del run
    assert stream.query()

def test_copy_refuses_what_the_device_cannot_address(ek):
    dev = torch.zeros(64, dtype=torch.uint8, device="cuda")
    for dst, src in ((dev[:32], torch.zeros(32, dtype=torch.uint8)), (dev[1:33], dev[32:])):
        with pytest.raises((ek.ElitekvError, ValueError)):
            ek.elitekv_copy(dst, src)


@pytest.mark.parametrize("B", [1, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("n_items", [3, 33, 40])
def test_combine_rows_sharing_warps(ek, B, n_items):
    """Up to 8 rows, 8 / 4 / 2 warps take turns at the items of a pair of rows (4 items a turn, the
    statistics of 32 in registers); from 9 rows on each pair has one warp.  One long sequence among
    short ones, and an empty one."""
    w = gen.shrink(gen.LLAMA7B_75, B=B, ctx=128 * n_items)
    st = H.setup(w, lens=([128 * n_items] + [65, 0, 300, 1, 128, 129, 77, 64])[:B], decode_kernel=2)
    H.check_parity(st, H.run_decode(st), H.sample_units(st, 24, seed=n_items))


# ------------------------------------------------------------------ work plans
@pytest.mark.parametrize("B,n_workers", [(255, 148), (256, 1), (256, 3840), (256, 3841), (257, 148)])
def test_plans_on_both_sides_of_a_sequence_per_thread(ek, B, n_workers):
    """Up to 256 sequences (and 4096 items) the plan has a thread per sequence, then a thread per item;
    beyond that a sequence's items are written one after the other.  Both against the rules the
    plans promise, with empty sequences at both ends of a thread's neighbours."""
    from . import test_gpu_parity as T
    lens = [0 if b % 5 in (0, 4) else 1 + (7919 * b) % 9000 for b in range(B)]
    T.test_worker_plan_structure(ek, lens, 64, n_workers, 2)
    T.test_plan_partitions_every_sequence(ek, lens, B + 300)


@pytest.mark.parametrize("B", [1, 32, 33, 257])
def test_cluster_kernel_behind_every_form_of_the_plan(ek, B):
    """The cluster kernel starts from the plan's record of each worker's first item, which a plan of a lane per
    sequence (up to 32), of a thread per sequence (256) and of a loop writes in its own way; empty
    sequences at the front, and workers without items."""
    w = gen.shrink(gen.LLAMA7B_75, B=B, ctx=300)
    st = H.setup(w, lens=[300] if B == 1 else [0 if b % 7 == 0 else 1 + (37 * b) % 150 for b in range(B)])
    assert ek.elitekv_decode_plan_info(st.layer, st.cache, B)[0] == 4
    H.check_parity(st, H.run_decode(st), H.sample_units(st, 24, seed=B))


@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("B", [1, 2, 31, 32, 33, 224, 225, 256, 257])
@pytest.mark.parametrize("kernel", [1, 2, 4])
def test_plan_that_a_call_makes(ek, kernel, B, ragged):
    """The exported plans take lengths of any size, in 64 bits; a decode call's own plan is another form of the code: 32-bit
    sums, a lane per sequence (balanced plans, up to 32), a thread per sequence (224 beside the warp that makes the dry
    trip, 256 without it), a loop beyond.  Read from the call's workspace (items and first items at its start, first items and
    records of the workers at its end): the same plan, and each worker's record is its first item."""
    w = gen.shrink(gen.LLAMA7B_75, B=B, ctx=200) if kernel > 1 else replace(gen.TINY, B=B, ctx=200)
    lens = [0 if b % 5 in (0, 4) else 1 + (7919 * b) % 199 for b in range(B)] if ragged else [200] * B
    st = H.setup(w, lens=[max(n, 1) for n in lens], fill=False, decode_kernel=kernel)
    dev = torch.tensor(lens, dtype=torch.int32, device="cuda")
    size = ek.elitekv_decode_workspace_size(st.layer, B)
    ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
    q_rope = torch.zeros((B, w.n_h, 2 * w.r), dtype=torch.bfloat16, device="cuda")
    q_abs = torch.zeros((B, w.n_h, st.layer.kw), dtype=torch.bfloat16, device="cuda")
    ek.elitekv_decode(st.layer, st.cache, q_rope, q_abs, dev, ws)
    got_kernel, tile, n_workers, max_items, overhead = ek.elitekv_decode_plan_info(st.layer, st.cache, B)
    assert got_kernel == kernel and ek.elitekv_check_status(st.layer) == 0
    up = lambda n: (n + 255) // 256 * 256
    words = lambda at, n: ws[at:at + 4 * n].view(torch.int32).cpu()
    if n_workers == 0:
        items, first = ek.elitekv_plan(dev, tile, max_items)
    else:
        items, first, wfirst = ek.elitekv_plan_workers(dev, tile, n_workers, max_items, overhead)
    assert torch.equal(words(0, 4 * max_items).view(-1, 4), items.cpu())
    assert torch.equal(words(up(16 * max_items), B + 1), first.cpu())
    if n_workers == 0:
        return
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    at_rec = size - up(32 * sms)
    at_first = at_rec - up(4 * (sms + 2))
    assert torch.equal(words(at_first, n_workers + 1), wfirst.cpu())
    if kernel == 4:
        rec, items, wfirst = words(at_rec, 8 * n_workers).view(-1, 8), items.cpu(), wfirst.tolist()
        for i in range(n_workers):
            lo, hi = wfirst[i], wfirst[i + 1]
            assert rec[i, :2].tolist() == [lo, hi]
            if lo < hi:
                assert rec[i, 2:5].tolist() == items[lo, :3].tolist()


MOST = 2 ** 31 - 1


@pytest.mark.parametrize("lens,tile", [([MOST] * 3, 1), ([MOST - 5, 0, 7, MOST], 1), ([MOST] * 256, 1), ([MOST] * 257, 3),
                                       ([MOST, 5] * 150, 1), ([MOST] * 3, 64), ([MOST], 2)])
def test_plans_of_more_tiles_than_31_bits_hold(ek, lens, tile):
    """The lengths' tiles sum to more than 2^31 on both sides of the sequence-per-thread line; items
    of both plans against the plans' rules in 64 bits (lengths alone: there is no cache)."""
    B, n_workers, overhead = len(lens), 148, 2
    t = torch.tensor(lens, dtype=torch.int32, device="cuda")
    lens = np.array(lens, dtype=np.int64)
    tiles = -(-lens // tile)
    for balanced in (False, True):
        n_max = B + (n_workers if balanced else 300)
        if balanced:
            items, first, wfirst = ek.elitekv_plan_workers(t, tile, n_workers, n_max, overhead)
        else:
            items, first = ek.elitekv_plan(t, tile, n_max)
        items, first = items.cpu().numpy().astype(np.int64), first.cpu().numpy()
        assert first[0] == 0 and np.all(np.diff(first) >= (lens > 0)) and first[B] <= n_max
        assert np.all(items[first[B]:, 0] == -1)
        for b in range(B):
            rows = items[first[b]:first[b + 1]]
            assert np.all(rows[:, 0] == b) and np.all(rows[:, 2] > 0) and np.all(rows[:, 1] % tile == 0)
            assert np.array_equal(np.cumsum(rows[:, 2]), np.append(rows[1:, 1], lens[b])[:len(rows)])
        its = items[:first[B]]
        if balanced:
            slots = np.where(tiles > 0, tiles + overhead, 0)
            g0, total = np.concatenate([[0], np.cumsum(slots)]), int(slots.sum())
            bound = np.array([w * total // n_workers for w in range(n_workers + 1)])
            ga = g0[its[:, 0]] + overhead + its[:, 1] // tile
            assert np.all(bound[its[:, 3]] <= ga) and np.all(ga - its[:, 1] // tile + -(-(its[:, 1] + its[:, 2]) // tile) <= bound[its[:, 3] + 1])
            assert np.array_equal(wfirst.cpu().numpy(), np.searchsorted(its[:, 3], np.arange(n_workers + 1)))
        else:
            target = -(-int(tiles.sum()) // (n_max - B))
            assert np.all(its[:, 2] <= target * tile)


@pytest.mark.parametrize("d", [64, 128, 320, 4096])
@pytest.mark.parametrize("T", [1, 127, 129, 257, 700])
def test_project_append_depth_shares(ek, T, d):
    """7B shape, 16 column tiles: 1, 2, 3 and 6 token tiles run with 4, 4, 2 and 1 blocks per tile where the
    depth has a step for each; rows a block finishes (32, 64, 128) end inside and at its range."""
    from .test_gpu_parity import _projection_case
    w = gen.shrink(gen.LLAMA7B_75, B=1, ctx=T)
    _projection_case(ek, w, d, [T], False, T + d)


# ------------------------------------------------------------------ append, staged form
@pytest.mark.parametrize("T", [2047, 2048, 2049, 4 * 148 * 4 * 2 + 3])
@pytest.mark.parametrize("shape", [dict(), dict(n_h=4, r=2, d_c=64), dict(r=48, d_c=3072)])
def test_append_staged_groups(ek, shape, T):
    """The staged form starts at 2048 tokens; groups of 4 tokens (7B rows), of 16 (the most) and of one
    (12 KB rows); a ragged last group, and more groups than one round of the grid.  Latent rows are
    copied bit for bit; the rotation is the register form's, bit for bit."""
    w = gen.shrink(replace(gen.LLAMA7B_75, **shape), B=1, ctx=T)
    st = H.setup(w, lens=[T], fill=False)
    perm = torch.randperm(T, generator=torch.Generator().manual_seed(T)).cuda()
    args = [x[perm].contiguous() for x in (st.k_e, st.c, st.seq_id, st.pos)]
    ek.elitekv_append(st.layer, st.cache, *args)
    rope, latent = st.rope_plane.clone(), st.latent_plane.clone()
    st.rope_plane.zero_()
    for a in range(0, T, 1000):
        ek.elitekv_append(st.layer, st.cache, *[x[a:a + 1000].contiguous() for x in args])
    assert ek.elitekv_check_status(st.layer) == 0
    assert torch.equal(rope, st.rope_plane)
    assert torch.equal(latent[st.pos.long()].view(torch.int16), st.c.view(torch.int16).view(T, -1))


@pytest.mark.parametrize("T", [1153, 1500, 2305, 4096])
def test_project_append_paired_forms_with_late_epilogue_warps(ek, T):
    """40 of 41 tokens have a position outside the cache: every thread that meets one records it with
    atomics on one word, so the epilogue warps of the paired forms come to their shared-memory units long
    after the ring has gone round.  The faults are reported as such (no wait runs out), the other tokens'
    rows are written and no other row is touched."""
    d, w = 4096, gen.LLAMA7B_75
    g = torch.Generator().manual_seed(T)
    rope_w = w.n_h * 2 * w.r
    W_ke, W_down = ((torch.randn(d, n, generator=g) / 64).to(torch.bfloat16).cuda() for n in (rope_w, w.d_c))
    idx = gen.elite_index_sets(w)
    layer = ek.Layer(w.n_h, w.d_h, w.r, w.d_c, idx, *gen.up_projections(w, "cuda"), T, W_ke=W_ke, W_down=W_down)
    rope, latent = (torch.zeros((T, n), dtype=torch.bfloat16, device="cuda") for n in (rope_w, w.d_c))
    cache = ek.make_cache(rope, latent, n_seqs=1, max_ctx=T)
    x = torch.randn(T, d, generator=g).to(torch.bfloat16).cuda()
    seq, pos = torch.zeros(T, dtype=torch.int32), torch.arange(T, dtype=torch.int32)
    good = pos % 41 == 7
    pos[~good] += T
    ek.elitekv_project_append(layer, cache, x, seq.cuda(), pos.cuda())
    assert ek.elitekv_check_status(layer) == ek.ERR_BAD_POSITION
    assert ek.elitekv_check_status(layer) == 0
    assert not rope[~good.cuda()].any() and not latent[~good.cuda()].any()
    zeros = [np.zeros((T, n), dtype=np.uint16) for n in (rope_w, w.d_c)]
    _, _, rows64, c64 = O.project_append_expected(*zeros, H.f64(x[good.cuda()]), H.f64(W_ke), H.f64(W_down), seq[good].numpy(),
                                                  pos[good].numpy(), idx.numpy(), w.d_h, base=w.rope_base, max_ctx=T,
                                                  page_table=None, page_size=w.page_size)
    for got, want in ((rope, rows64), (latent, c64)):
        # as for the other projections: one bf16 rounding plus fp32 accumulation over d terms
        assert np.all(np.abs(H.f64(got[good.cuda()]) - want) <= np.abs(want) * 2.0 ** -8 + 2e-5 * d ** 0.5)


@pytest.mark.parametrize("T", [100, 1153, 4096])
def test_project_append_table_on_any_8_bytes(ek, T):
    """A caller's (cos, sin) table that starts 8 bytes past a 16-byte boundary gives the bits of the same
    table on one, in the split-depth form and in both paired forms."""
    d, w = 1024, replace(gen.LLAMA7B_75, seed=T)
    g = torch.Generator().manual_seed(T)
    rope_w = w.n_h * 2 * w.r
    W_ke, W_down = ((torch.randn(d, n, generator=g) / 32).to(torch.bfloat16).cuda() for n in (rope_w, w.d_c))
    x = torch.randn(T, d, generator=g).to(torch.bfloat16).cuda()
    tab = torch.from_numpy(O.rope_table_f32(T, w.d_h, w.rope_base)).cuda()
    room = torch.zeros(tab.numel() + 2, device="cuda")
    shifted = room[2:].view(tab.shape).copy_(tab)
    assert shifted.data_ptr() % 16 == 8 and tab.data_ptr() % 16 == 0
    seq, pos = torch.zeros(T, dtype=torch.int32, device="cuda"), torch.arange(T, dtype=torch.int32, device="cuda")
    rows = []
    for cs in (tab, shifted):
        layer = ek.Layer(w.n_h, w.d_h, w.r, w.d_c, gen.elite_index_sets(w), *gen.up_projections(w, "cuda"), T, cos_sin=cs,
                         W_ke=W_ke, W_down=W_down)
        rope, latent = (torch.zeros((T, n), dtype=torch.bfloat16, device="cuda") for n in (rope_w, w.d_c))
        ek.elitekv_project_append(layer, ek.make_cache(rope, latent, n_seqs=1, max_ctx=T), x, seq, pos)
        assert ek.elitekv_check_status(layer) == 0
        rows.append((rope, latent))
    assert all(torch.equal(a, b) for a, b in zip(*rows))


def test_more_rows_than_a_grid_dimension(ek):
    """Blocks of 16 rows (combine) and of 64 (query preparation) past the 65535 that a grid's third dimension
    holds: sequences of one token, whose output is the up-projected latent, and absorbed queries whose
    last rows are those of a small call."""
    B = 16 * 65535 + 17
    w = replace(gen.LLAMA7B_75, n_h=1, r=2, d_c=128, B=B, ctx=1)
    layer = ek.Layer(1, w.d_h, w.r, w.d_c, gen.elite_index_sets(w), *(W := gen.up_projections(w, "cuda")), 2)
    g = torch.Generator(device="cuda").manual_seed(5)
    latent = torch.randn((B, w.d_c), generator=g, device="cuda").to(torch.bfloat16)
    rope = torch.zeros((B, 2 * w.r), dtype=torch.bfloat16, device="cuda")
    q_rope, q_abs = torch.zeros((B, 1, 2 * w.r), dtype=torch.bfloat16, device="cuda"), torch.zeros((B, 1, w.d_c), dtype=torch.bfloat16, device="cuda")
    lens = torch.ones(B, dtype=torch.int32, device="cuda")
    ws = torch.empty(ek.elitekv_decode_workspace_size(layer, B), dtype=torch.uint8, device="cuda")
    out = ek.elitekv_decode(layer, ek.make_cache(rope, latent, n_seqs=B, max_ctx=1), q_rope, q_abs, lens, ws)
    assert ek.elitekv_check_status(layer) == 0
    for at in (slice(0, 40), slice(B - 60, B)):
        want = H.f64(latent[at]) @ H.f64(W[1])
        assert np.linalg.norm(H.f64(out[at, 0]) - want) <= H.REL_L2_TOL * np.linalg.norm(want)
    del latent, rope, q_rope, q_abs, ws, out
    B = 64 * 65535 + 70
    w = replace(w, d_h=16, d_c=8, B=B)
    layer = ek.Layer(1, w.d_h, w.r, w.d_c, gen.elite_index_sets(w), *gen.up_projections(w, "cuda"), 2)
    q = torch.randn((B, 1, w.d_h), generator=g, device="cuda").to(torch.bfloat16)
    got = ek.elitekv_absorb_query(layer, q, lens.new_zeros(B))
    assert ek.elitekv_check_status(layer) == 0
    for at in (slice(0, 100), slice(B - 200, B)):
        want = ek.elitekv_absorb_query(layer, q[at].contiguous(), lens.new_zeros(q[at].shape[0]))
        assert all(torch.equal(a[at], b) for a, b in zip(got, want))


def test_project_append_more_tokens_than_a_grid_dimension(ek):
    """More 128-token tiles than the 65535 of a grid's second dimension, at a depth that the paired forms
    leave to them: the rows around the end are those of small calls."""
    d, T, ctx = 64, 65535 * 128 + 200, 1000
    w = replace(gen.LLAMA7B_75, n_h=16, r=4, d_c=128)
    B, rope_w = -(-T // ctx), 128
    g = torch.Generator(device="cuda").manual_seed(9)
    W_ke, W_down = ((torch.randn((d, 128), generator=g, device="cuda") / 8).to(torch.bfloat16) for _ in range(2))
    layer = ek.Layer(w.n_h, w.d_h, w.r, w.d_c, gen.elite_index_sets(w), *gen.up_projections(w, "cuda"), ctx, W_ke=W_ke, W_down=W_down)
    x = torch.empty((T, d), dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    t = torch.arange(T, device="cuda")
    seq, pos = (t // ctx).to(torch.int32), (t % ctx).to(torch.int32)
    planes = [torch.zeros((B * ctx, n), dtype=torch.bfloat16, device="cuda") for n in (rope_w, w.d_c)]
    cache = ek.make_cache(*planes, n_seqs=B, max_ctx=ctx)
    ek.elitekv_project_append(layer, cache, x, seq, pos)
    assert ek.elitekv_check_status(layer) == 0
    for at in (slice(0, 300), slice(T - 400, T - 200), slice(T - 200, T)):
        want = [p[at].clone() for p in planes]
        assert all(p[at].any(dim=1).all() for p in planes)
        for p in planes:
            p[at] = 0
        ek.elitekv_project_append(layer, cache, x[at].contiguous(), seq[at].contiguous(), pos[at].contiguous())
        # the same fp32 sums in another order may round to the next bf16: one unit of 2^-7 at most
        assert all(torch.allclose(p[at].float(), y.float(), rtol=2.0 ** -7, atol=1e-5) for p, y in zip(planes, want))


def test_layers_of_several_shapes_step_in_several_threads(ek):
    """Threads that step layers whose kernels are the same and want more or less shared memory each: no
    launch is refused, and the outputs are those of a thread alone."""
    import functools
    import threading
    shapes = [gen.LLAMA7B_75, gen.SWEEP_75_SLRD, replace(gen.LLAMA7B_75, d_c=1024), gen.SWEEP_75_SLRD]
    steps = []
    for w in shapes:
        st = H.setup(gen.shrink(w, B=2, ctx=100), lens=[100, 70])
        last = torch.from_numpy(st.starts[1:] - 1).cuda()
        k_e, c, seq, pos = (x[last].contiguous() for x in (st.k_e, st.c, st.seq_id, st.pos))
        q_rope, q_abs, out = (torch.empty((2, w.n_h, n), dtype=torch.bfloat16, device="cuda") for n in (2 * w.r, st.layer.kw, w.d_h))
        steps.append((st, functools.partial(ek.elitekv_decode_step, st.layer, st.cache, k_e, c, seq, pos, st.q, st.lens_dev,
                                            q_rope, q_abs, st.workspace, out)))
    alone = []
    for st, step in steps:
        alone.append(step().clone())
    torch.cuda.synchronize()
    failed = []

    def loop(step):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(2000):
                    step()
                torch.cuda.current_stream().synchronize()
        except Exception as e:
            failed.append(e)

    threads = [threading.Thread(target=loop, args=(step,)) for _, step in steps]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[:2]
    for (st, step), want in zip(steps, alone):
        assert ek.elitekv_check_status(st.layer) == 0
        assert torch.equal(step(), want)


def test_step_of_a_cache_that_declares_more_tiles_than_31_bits_hold(ek):
    """A page table of 2048 entries for pages of 2^20 tokens: the plan's sums are 64 bits wide and the step's
    front end is the separate launches, with the same bits as the three calls."""
    w = replace(gen.TINY, B=2)
    layer = ek.Layer(w.n_h, w.d_h, w.r, w.d_c, gen.elite_index_sets(w), *gen.up_projections(w, "cuda"), 300)
    table = torch.full((2, 2048), -1, dtype=torch.int32, device="cuda")
    table[:, 0] = torch.tensor([1, 0], dtype=torch.int32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda *shape: torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    lens = torch.tensor([270, 31], dtype=torch.int32, device="cuda")
    seq, pos = torch.arange(2, dtype=torch.int32, device="cuda"), lens - 1
    k_e, c, q = rand(2, w.n_h, w.r, 2), rand(2, w.d_c), rand(2, w.n_h, w.d_h)
    rope, latent = rand(2 << 20, w.n_h * 2 * w.r), rand(2 << 20, w.d_c)
    cache = ek.make_cache(rope, latent, n_seqs=2, page_table=table, page_size=1 << 20)
    ws = torch.empty(ek.elitekv_decode_workspace_size(layer, 2), dtype=torch.uint8, device="cuda")
    q_rope, q_abs, out = (torch.empty((2, w.n_h, n), dtype=torch.bfloat16, device="cuda") for n in (2 * w.r, layer.kw, w.d_h))
    ek.elitekv_decode_step(layer, cache, k_e, c, seq, pos, q, lens, q_rope, q_abs, ws, out)
    assert ek.elitekv_check_status(layer) == 0
    assert torch.equal(latent[(table[:, 0].long() << 20) + pos.long()], c)
    want = ek.elitekv_decode(layer, cache, *ek.elitekv_absorb_query(layer, q, pos), lens, ws)
    assert torch.isfinite(out).all() and out.any() and torch.equal(out, want)
