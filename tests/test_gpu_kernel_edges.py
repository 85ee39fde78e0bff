"""GPU parity at the sizes where a kernel or a rule of its dispatch changes: edges of tiles, remainders, the smallest
and the largest of a range, against the float64 oracle."""
import pytest
import torch

from oracle import ficoco_oracle as fo, gaps
from paper_2411_17686_b200 import binding, synth
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    c = binding.Context(max_tokens=36000, max_dim=4096, max_batch=180, max_text=64, device=0)
    yield c
    c.close()


def run_v(ctx, seed, batch, gh, gw, dim, keep, dtype="bf16", cls=True, p=fo.Params()):
    b = synth.make_v_batch(seed, batch, gh, gw, dim, 2, keep, dtype, cls, 1.0)
    gaps.repair_v(b, p)
    parity.run_and_compare_v(ctx, b, p, DEV, what=f"{batch} x {gh} x {gw} x {dim} {dtype} keep {keep}")


@pytest.mark.parametrize("batch,gh,gw,dim,keep,dtype", [
    (1, 9, 9, 64, 1, "bf16"),          # one row with every source
    (1, 33, 34, 64, 1, "bf16"),        # more sources than a CTA files: the in-order rescan
    (2, 8, 8, 4096, 9, "fp32"),        # rows of 16 KB: few rows per CTA
    (1, 6, 7, 72, 41, "bf16"),         # one source; rows that are no multiple of 32 vectors
    (24, 20, 20, 64, 300, "bf16"),     # many rows per CTA, dealt out with a stride
    (1, 1, 73, 72, 1, "bf16"),         # 72 sources: the longest list that is not split over groups of lanes
    (1, 2, 37, 72, 1, "bf16"),         # 73: the shortest that is, in a row that ends inside its second part
    (1, 7, 14, 1280, 1, "fp32"),       # 97: the groups' lists differ in length by a batch
], ids=["hub", "rescan", "wide-rows", "one-source", "many-rows", "72", "73", "97"])
def test_merge_rows(ctx, batch, gh, gw, dim, keep, dtype):
    run_v(ctx, 91, batch, gh, gw, dim, keep, dtype)


@pytest.mark.parametrize("kind,batch,dim,dtype", [("l", 16, 4096, "bf16"), ("v", 40, 1664, "fp32"), ("v", 24, 4096, "fp32")])
def test_most_rows_kept_of_wide_rows(kind, batch, dim, dtype):
    """Many output rows of which a merge CTA's shared memory takes few: the work table has to hold them all."""
    n, keep, heads, text = 576, 560, 2, 64
    rows = n + (text if kind == "l" else 0)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((batch * rows, dim), generator=g, device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    c = binding.Context(max_tokens=batch * rows, max_dim=dim, max_batch=batch, max_text=text, device=0)
    try:
        if kind == "l":
            attn = torch.softmax(torch.randn((batch, heads, text, n), generator=g, device="cuda"), dim=3)
            r = c.ficoco_l_reduce(x, attn, keep, n, text, heads, params=binding.make_params(max_targets=0))
            kept = keep + text
        else:
            attn = torch.softmax(torch.randn((batch, heads, n), generator=g, device="cuda"), dim=2)
            r = c.ficoco_v_reduce(x, attn, keep, 24, 24, heads, n_tokens=n,
                                  params=binding.make_params(has_cls=False, max_targets=0))
            kept = keep
        first = torch.arange(batch, device="cuda").repeat_interleave(kept) * rows
        assert torch.equal(r.out_tokens, x[first + r.kept_idx])          # pruning: rows pass through
        assert c.ficoco_status() == 0
    finally:
        c.close()


@pytest.mark.parametrize("gh,gw,dim,keep,fused", [
    (31, 33, 64, 900, True), (32, 32, 64, 1, True),       # 1023 and 1024 tokens: two per thread in registers
    (25, 41, 64, 1024, True), (25, 41, 64, 4, True),      # 1025, the fewest of the histogram: 1 and 1021 discarded
    (48, 45, 64, 40, True),
    (64, 64, 64, 2000, False), (17, 241, 64, 4096, False),     # the fused filter's ring is too small to work in
    (64, 64, 256, 2000, True), (17, 241, 256, 4096, True),     # the same by slices, each on the CTA that scored it
])
def test_selection_sizes(ctx, gh, gw, dim, keep, fused):
    """With the local penalty.  Up to 1024 tokens in registers, more by a histogram over the value range."""
    run_v(ctx, 92, 1, gh, gw, dim, keep, cls=False, p=fo.Params(max_targets=0) if gh * gw > 4000 else fo.Params())
    assert (ctx.ficoco_last_launch_count() < 6) == fused       # filter in one kernel or in four


@pytest.mark.parametrize("fused", [True, False], ids=["fused", "unfused"])
@pytest.mark.parametrize("n,keep,levels", [(1100, 500, 1), (2000, 1300, 2), (1100, 1099, 2000), (3000, 40, 4), (4100, 2000, 40)])
def test_selection_of_equal_scores(n, keep, levels, fused):
    """Scores that take few values (lambda = 0: the attention alone): ties at the threshold go to the lower index whether
    they fit the list of the part it lies in or not."""
    dim = 256 if fused else 4096
    g = torch.Generator(device="cuda").manual_seed(n)
    a = torch.randint(0, levels, (1, 1, n), generator=g, device="cuda").float() / 4096
    x = torch.randn((n, dim), generator=g, device="cuda").to(torch.bfloat16)
    c = binding.Context(max_tokens=n, max_dim=dim, max_batch=1, device=0)
    try:
        r = c.ficoco_v_reduce(x, a, keep, n // 50, 50, 1, n_tokens=n,
                              params=binding.make_params(lam=0.0, has_cls=False, local_penalty=False, max_targets=0))
        gone = (-a[0, 0]).argsort(descending=True, stable=True)[:n - keep]
        left = torch.ones(n, dtype=torch.bool, device="cuda")
        left[gone] = False
        assert torch.equal(r.kept_idx.long(), left.nonzero()[:, 0])
    finally:
        c.close()


@pytest.mark.parametrize("dim,n_src,n_tgt", [
    (64, 1, 16), (64, 128, 17), (128, 129, 256), (192, 127, 257), (320, 8, 255), (448, 40, 300)])
def test_correlate_tiles(ctx, dim, n_src, n_tgt):
    """Odd and even numbers of 64-element blocks (one and two per ring stage), tiles and splits around their edges."""
    n = n_src + n_tgt
    gw = next(g for g in (16, 11, 9, 7, 5, 4, 3, 2, 1) if n % g == 0)
    run_v(ctx, 93, 2, n // gw, gw, dim, n_tgt)


@pytest.mark.parametrize("n_vision,n_text,dim,keep,p", [
    (65, 1, 64, 1, fo.Params()),                        # one k-block, one text token, one column
    (130, 3, 1088, 17, fo.Params()),                    # 17 k-blocks: the last stage of four holds one
    (300, 100, 512, 30, fo.Params(eps=0.5)),            # top lists of 16 entries merged over lanes and splits
    (272, 100, 64, 271, fo.Params()),                   # one source, two splits, much text
    (140, 101, 128, 60, fo.Params()),                   # the most text that tiles are planned for
    (140, 102, 128, 60, fo.Params()),                   # one more: the SIMT kernel
], ids=["one", "last-stage", "long-lists", "one-source", "most-text", "simt"])
def test_correlate_text_weights(n_vision, n_text, dim, keep, p):
    """FiCoCo-L tiles: odd numbers of blocks, little and much text."""
    c = binding.Context(max_tokens=2 * (n_vision + n_text), max_dim=dim, max_batch=2, max_text=n_text, device=0)
    try:
        b = synth.make_l_batch(96, 2, n_vision, n_text, dim, 3, keep)
        gaps.repair_l(b, p)
        parity.run_and_compare_l(c, b, p, DEV, what=f"L {n_vision} + {n_text}, {dim}, keep {keep}")
    finally:
        c.close()


@pytest.mark.parametrize("batch,n_vision,n_text,dim,keep,eps", [
    (20, 800, 101, 64, 200, 0.998),                     # 120 x 112 tokens per tile, one k-block, two splits
    (10, 1500, 101, 320, 300, 0.998),                   # 120 x 80, four splits, five k-blocks in two stages
    (20, 800, 80, 64, 200, 0.986),                      # lists of four
    (80, 400, 85, 64, 133, 0.9),                        # lists of 15, 96 x 144, not split
], ids=["two-splits", "five-blocks", "lists-of-4", "lists-of-15"])
def test_correlate_text_weights_in_the_ring(batch, n_vision, n_text, dim, keep, eps):
    """Grids of more than one CTA per SM with much text: the weights take the place of the operand ring."""
    p = fo.Params(eps=eps)
    c = binding.Context(max_tokens=batch * (n_vision + n_text), max_dim=dim, max_batch=batch, max_text=n_text, device=0)
    try:
        b = synth.make_l_batch(101, batch, n_vision, n_text, dim, 2, keep)
        gaps.repair_l(b, p)
        parity.run_and_compare_l(c, b, p, DEV, what=f"L {batch} x {n_vision} + {n_text}, {dim}, keep {keep}")
    finally:
        c.close()


@pytest.mark.parametrize("n_vision,n_text,dim,heads,dtype", [
    (37, 3, 2112, 17, "bf16"),         # 111 attention values, no multiple of four; one head more than are in flight
    (130, 8, 2112, 3, "bf16"),         # 1040: a second part of 16 values
    (64, 16, 4096, 16, "fp32"),        # 1024: one full part; rows of 16 KB
    (205, 5, 1032, 2, "fp32"),         # 1025: parts of 256 and one value; rows just past the narrower kernels
    (64, 8, 64, 9, "bf16"),            # a kernel of its own: 512 values, one full part; one head more than are in flight
    (130, 4, 64, 3, "bf16"),           # 520: a second part of 8 values
    (129, 1, 64, 17, "bf16"),          # 129: a part of 128 single values and one of one
], ids=["scalar", "two-parts", "full-part", "one-value", "own-full-part", "own-two-parts", "own-one-value"])
def test_head_mean(n_vision, n_text, dim, heads, dtype):
    """In the grid of the column sums where rows are wide, else in a grid of its own."""
    c = binding.Context(max_tokens=3 * (n_vision + n_text), max_dim=dim, max_batch=3, max_text=n_text, device=0)
    try:
        b = synth.make_l_batch(100, 3, n_vision, n_text, dim, heads, n_vision // 2, dtype)
        gaps.repair_l(b, fo.Params())
        parity.run_and_compare_l(c, b, fo.Params(), DEV, what=f"L {n_vision} + {n_text}, {dim}, {heads} heads")
    finally:
        c.close()


@pytest.mark.parametrize("eps,keep", [(0.998, 96), (0.9, 96), (0.9, 150)], ids=["2", "11", "16"])
def test_lists_merged_over_splits(ctx, eps, keep):
    """One image, whose tiles are split over many CTAs: lists of 2 to 16 entries merged by groups of lanes."""
    run_v(ctx, 98, 1, 18, 40, 1024, keep, p=fo.Params(eps=eps))


@pytest.mark.parametrize("batch,n_src,n_tgt,dim", [
    (1, 1, 16, 64), (1, 33, 65, 192), (2, 95, 31, 576), (1, 64, 200, 1024), (3, 100, 300, 320), (8, 128, 257, 128)])
def test_correlate_fp32_tiles(ctx, batch, n_src, n_tgt, dim):
    """Tiles of 32 x 32 and 128 x 64 around their edges, fewer and more k-blocks than slots in flight."""
    n = n_src + n_tgt
    gw = next(g for g in (16, 11, 9, 7, 5, 4, 3, 2, 1) if n % g == 0)
    run_v(ctx, 99, batch, n // gw, gw, dim, n_tgt, dtype="fp32")


@pytest.mark.parametrize("batch,gh,gw,dim", [(149, 7, 7, 64), (170, 10, 10, 256), (3, 44, 44, 512), (1, 3, 11, 64), (2, 33, 3, 1280),
                                               (1, 5, 5, 2048), (2, 7, 9, 1408), (2, 7, 9, 1664)])
def test_pieces_dealt_to_filter_ctas(ctx, batch, gh, gw, dim):
    """More images than SMs, images of several pieces, and warps without a row."""
    run_v(ctx, 94, batch, gh, gw, dim, gh * gw // 2)


@pytest.mark.parametrize("wait_ns", [20_000, 200_000, 2_000_000])
def test_barrier_wait_ends_soon_after_its_limit(ctx, wait_ns):
    """The limit counts cycles of a 2 GHz clock; a failed try suspends the thread for about 8000 cycles, and the one
    before the clock is first read and the one that outlasts the limit come on top."""
    ctx.ficoco_debug_waits(wait_ns, 0)
    try:
        cycles = ctx.ficoco_debug_barrier_wait()
    finally:
        ctx.ficoco_debug_waits(0, 0)
    assert 2 * wait_ns < cycles < 2 * wait_ns + 3 * 8000


@pytest.mark.parametrize("batch,gh,gw,dim", [(1, 61, 67, 64), (170, 10, 10, 2048)], ids=["large-image", "large-batch"])
def test_unfused_filter(batch, gh, gw, dim):
    """The three plain kernels: a selection whose work area outgrows the fused kernel's ring, and more images than
    SMs with more than 64 MB of tokens."""
    c = binding.Context(max_tokens=batch * (gh * gw + 1), max_dim=dim, max_batch=batch, max_text=0, device=0)
    try:
        c.ficoco_profile(True)
        run_v(c, 95, batch, gh, gw, dim, gh * gw // 2)
        assert "score" in [name for name, _, _ in c.ficoco_profile_read()]
    finally:
        c.close()


@pytest.mark.parametrize("fused", [True, False], ids=["fused", "unfused"])
@pytest.mark.parametrize("n,gh,gw,same", [(600, 20, 40, False), (1000, 32, 32, True), (1100, 30, 40, False), (2000, 40, 50, True)])
def test_positions_that_occur_twice(n, gh, gw, same, fused):
    """The best token of a window gets the penalty wherever several tokens share a cell, in every repetition: positions
    drawn with replacement, and half of the tokens in one cell."""
    dim = 64 if fused else 4096
    b = synth.make_v_batch(97, 2, n // 50, 50, dim, 2, n // 2, "bf16", False, 1.0)
    for i in range(2):
        r = synth.rng_for(97, i, 8)
        b.pos[i] = r.integers(0, gh * gw, n).astype("int32")
        if same:
            b.pos[i][r.permutation(n)[:n // 2]] = 7
        b.grid[i] = (gh, gw)
    prune = fo.Params(max_targets=0)
    gaps.repair_v(b, prune)
    c = binding.Context(max_tokens=2 * n, max_dim=dim, max_batch=2, device=0)
    try:
        for _ in range(3):
            parity.run_and_compare_v(c, b, prune, DEV, what=f"{n} tokens, repeated positions")
    finally:
        c.close()
