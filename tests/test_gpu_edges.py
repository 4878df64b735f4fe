"""GPU parity at the sizes where a kernel's split or a dispatch changes: edges of tiles, strips,
runs and clusters, the smallest and largest of each range, against the fp64 oracle."""
import math

import numpy as np
import pytest
import torch

from oracle import pace_oracle as O
from paper_2608_27206_gb300 import synth
from tests.helpers import assert_scores_close, bf16_tensor, f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pace():
    from paper_2608_27206_gb300 import build
    build.build()
    from paper_2608_27206_gb300 import pace as P
    P.pace_init(0)
    P.pace_device_status(clear=True)
    yield P
    assert P.pace_device_status(clear=True)[0] == 0


# The distance of two unit vectors is off by no more than the vectors are.  Their norms come from fp32 sums of at most 50
# additions per lane and five over the lanes, which the square root halves; means, quotients and the distance itself
# add a few roundings.  (The largest seen is 4 units of 2^-24.)
TIGHT = 32 * 2.0 ** -24


def assert_tight(got, ref):
    np.testing.assert_allclose(got, ref, rtol=0, atol=TIGHT)


def _cu(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)


# last query tile of 128 rows or fewer (half a tile) and above, alone (rows past the image are the
# tensor's zero fill) and followed by another image (rows overwritten), one tile and several
@pytest.mark.parametrize("lens", [(4,), (128,), (132,), (256,), (384,), (388, 4), (260, 128), (516, 1284, 1028)])
def test_vit_last_tile(pace, lens):
    cu = _cu(lens)
    q, k = (synth.random_small_qk(s + len(lens), int(cu[-1]), 3, 80) for s in (1, 2))
    got = pace.pace_vit_attn_importance(bf16_tensor(q), bf16_tensor(k), cu, merge=4).cpu().numpy()
    assert_scores_close(got, O.vit_attn_importance(f64(q), f64(k), cu, 80 ** -0.5, 4))


# a merge of 0 is refused by the library, whatever the caller brings
@pytest.mark.parametrize("given", [False, True])
def test_vit_merge_of_zero(pace, given):
    q = bf16_tensor(synth.random_small_qk(1, 8, 3, 80))
    out = torch.empty(8, device="cuda") if given else None
    ev = torch.cuda.Event()
    ev.record()
    for call in (lambda: pace.pace_vit_attn_importance(q, q, [0, 8], merge=0, out=out),
                 lambda: pace.pace_vit_attn_importance_chunked(q, q, [0, 8], [8], [ev], merge=0, out=out)):
        with pytest.raises(pace.PaceError) as e:
            call()
        assert e.value.status == pace.PACE_ERR_INVALID_ARG


# few keys and several heads per KV head: pass 2 splits a group's heads over CTAs (7 heads; 1 and 2
# query tiles), down to one stream item per CTA
@pytest.mark.parametrize("tq,nv", [((1,), (1,)), ((128,), (300,)), ((129,), (128,)), ((257, 5), (40, 513))])
def test_llm_stream_splits(pace, tq, nv):
    cq, cv = _cu(tq), _cu(nv)
    q, k = synth.random_small_qk(3, int(cq[-1]), 14, 128), synth.random_small_qk(4, int(cv[-1]), 2, 128)
    got = pace.pace_llm_text_visual_importance(bf16_tensor(q), bf16_tensor(k), cq, cv).cpu().numpy()
    assert_scores_close(got, O.llm_text_visual_importance(f64(q), f64(k), cq, cv, 128 ** -0.5))


# causal streams whose lengths differ from CTA to CTA, split or not, in a batch
@pytest.mark.parametrize("before,nv,after", [((0,), (1,), (0,)), ((7,), (600,), (130,)), ((3, 20), (129, 700), (1, 300))])
@pytest.mark.parametrize("query_set", ["vision_text", "text", "last"])
def test_sequence_stream_splits(pace, before, nv, after, query_set):
    cu = _cu([a + b + c for a, b, c in zip(before, nv, after)])
    q, k = synth.random_small_qk(5, int(cu[-1]), 14, 128), synth.random_small_qk(6, int(cu[-1]), 2, 128)
    got = pace.pace_llm_sequence_importance(bf16_tensor(q), bf16_tensor(k), cu, before, nv, query_set).cpu().numpy()
    assert_scores_close(got, O.llm_sequence_importance(f64(q), f64(k), cu, before, nv, 128 ** -0.5, query_set))


# element widths 16, 4 and 1, blocks of 1024 elements with remainders, several tensors and slabs,
# rows out of range
@pytest.mark.parametrize("n_idx", [1, 63, 64, 65, 341, 8193])
def test_gather_multi_blocks(pace, n_idx):
    rng = np.random.default_rng(n_idx)
    idx = rng.integers(0, 50, n_idx).astype(np.int32)
    shapes = [((50, 8, 16), 0), ((3, 50), 1), ((2, 3, 50, 64), 2), ((50, 5), 0), ((2, 50, 3), 1)]
    src = [torch.from_numpy(rng.integers(0, 255, s, dtype=np.uint8)).cuda() for s, _ in shapes]
    src[1] = src[1].to(torch.int32)
    dst = [torch.zeros(s[:d] + (n_idx,) + s[d + 1:], dtype=t.dtype, device="cuda") for t, (s, d) in zip(src, shapes)]
    specs = [pace.gather_spec(a, b, d) for a, b, (_, d) in zip(src, dst, shapes)]
    pace.pace_gather_multi(specs, torch.from_numpy(idx).cuda())
    for a, b, (_, d) in zip(src, dst, shapes):
        assert torch.equal(b, a.index_select(d, torch.from_numpy(idx).cuda().long()))
    idx[0] = 50
    pace.pace_gather_multi(specs, torch.from_numpy(idx).cuda())
    assert pace.pace_device_status(clear=True) == (pace.PACE_ERR_INVALID_ARG, 13)
    for b, (_, d) in zip(dst, shapes):
        assert not b.select(d, 0).any()


# rows of 1- and 4-byte elements: a warp per row (64 elements and more, 4 and more where the rows are few, more than 256
# where they are many) and by elements, several steps of a warp with remainders, slabs, rows out of range
@pytest.mark.parametrize("n_idx,slabs", [(7, 1), (191, 2), (192, 2), (1024, 2), (1025, 2)])
@pytest.mark.parametrize("nbytes,strided", [(3, False), (4, False), (63, False), (64, False), (65, True), (127, False), (129, True),
                                            (255, False), (257, False), (252, True), (1024, False), (1028, True), (1022, False)])
def test_gather_multi_narrow_rows(pace, n_idx, slabs, nbytes, strided):
    rng = np.random.default_rng(nbytes + n_idx)
    idx = torch.from_numpy(rng.integers(0, 30, n_idx).astype(np.int32)).cuda()
    wide = torch.from_numpy(rng.integers(0, 255, (slabs, 30, nbytes + (4 if strided else 0)), dtype=np.uint8)).cuda()
    src, dst = wide[:, :, :nbytes], torch.full((slabs, n_idx, nbytes), 7, dtype=torch.uint8, device="cuda")
    g = pace.GatherTensor(src.data_ptr(), dst.data_ptr(), nbytes, src.stride(1), nbytes, slabs, src.stride(0), dst.stride(0), 30)
    pace.pace_gather_multi([g], idx)
    assert torch.equal(dst, src.index_select(1, idx.long()))
    idx[n_idx - 1] = -1
    pace.pace_gather_multi([g], idx)
    assert pace.pace_device_status(clear=True) == (pace.PACE_ERR_INVALID_ARG, 13)
    assert not dst[:, n_idx - 1].any() and torch.equal(dst[:, :n_idx - 1], src.index_select(1, idx[:-1].long()))


# strips of 8, 16 and 32 patches, full and partial, single last patches (odd widths: image rows on
# 2-byte boundaries), the last image row's odd end, several images per CTA
@pytest.mark.parametrize("shapes", [[(14, 14)], [(28, 42)], [(14, 14 * 33)], [(14 * 3, 14 * 31), (14, 14 * 8), (28, 14 * 9)],
                                    [(14 * 20, 14 * 17)], [(14 * 60, 14 * 35)], [(14 * 100, 14 * 97), (14, 28)]])
def test_density_strips(pace, shapes):
    rng = np.random.default_rng(len(shapes) + shapes[0][1])
    imgs = [synth.make_image(rng, h, w, max(1, w // 90), max(1, h // 90), 0.4) for h, w in shapes]
    imgs[0][-1, -1] = 255   # the image's very last bytes count
    buf, off = synth.pack_images(imgs)
    d, st = pace.pace_apc_density(torch.from_numpy(buf).cuda(), off, [s[0] for s in shapes], [s[1] for s in shapes])
    d, p0 = d.cpu().numpy(), 0
    for im, s in zip(imgs, pace.stats_dict(st)):
        ref = O.apc_density(im)
        assert_tight(d[p0:p0 + ref["N"]], ref["d"])
        assert abs(s["phi"] - ref["phi"]) <= TIGHT and abs(s["d_top"] - ref["d_top"]) <= TIGHT
        p0 += ref["N"]


# the black patch's weight is exactly 2^31, the white one's the smallest; identical patches have d = 0
# up to the rounding of 1/|t| (2^-24 of a unit vector, twice)
@pytest.mark.parametrize("value", [0, 255])
def test_density_extreme_values(pace, value):
    img = np.full((14 * 6, 14 * 40, 3), value, np.uint8)
    d, st = pace.pace_apc_density(torch.from_numpy(img.reshape(-1)).cuda(), [0], [84], [560])
    assert d.abs().max().item() <= 4 * 2.0 ** -24 and abs(pace.stats_dict(st)[0]["phi"] - 1) <= 1e-6
    img[:14, :14] = 255 - value
    d, _ = pace.pace_apc_density(torch.from_numpy(img.reshape(-1)).cuda(), [0], [84], [560])
    assert_tight(d.cpu().numpy(), O.apc_density(img)["d"])


# column sums whose high word passes 2^24 (from about 186000 patches on) are rounded once, as smaller ones: four times the same patches have exactly four times the sums, so the same means, bit for bit
@pytest.mark.parametrize("rows,cols,first,value", [(700, 520, 1, 241), (700, 520, 1, 201), (700, 520, 3, 201), (748, 498, 6, 201)])
def test_density_large_sums(pace, rows, cols, first, value):
    got = []
    for r, c in ((rows, cols), (rows // 2, cols // 2)):
        img = torch.zeros((r, 14, c, 14 * 3), dtype=torch.uint8, device="cuda")
        img[:, 0, :, :first] = value   # the first bytes of every patch
        d, st = pace.pace_apc_density(img.view(-1), [0], [14 * r], [14 * c])
        assert bool((d == d[0]).all())
        got.append((st[0, :2].tolist(), d[0].item()))
    assert got[0] == got[1]


# pictures so narrow that a group of threads meets more strips than its 32-bit sums are trusted with (2048, of one or
# two patches): four times the same four patches give the same means and distances, bit for bit
@pytest.mark.parametrize("cols", [1, 2])
def test_density_many_strips(pace, cols):
    pattern = torch.randint(0, 256, (4, 14, cols, 42), dtype=torch.uint8, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    got = []
    for rows in (1 << 20, 1 << 18):
        img = pattern.repeat(rows // 4, 1, 1, 1)
        d, st = pace.pace_apc_density(img.view(-1), [0], [14 * rows], [14 * cols])
        d = d.view(rows // 4, -1)
        assert bool((d == d[0]).all())
        got.append((st[0, :2].tolist(), d[0].tolist()))
    assert got[0] == got[1]
    ref = O.apc_density(pattern.reshape(56, cols * 14, 3).cpu().numpy())
    assert_tight(got[0][1], ref["d"])


# the tail over a cluster (more than 8192 distances): a bucket of equal distances too many for the
# list, a list ranked in rounds (quantised values: many equal, several different), a direct ranking
@pytest.mark.parametrize("kind", ["equal", "steps", "natural"])
def test_density_tail_cluster(pace, kind):
    rng = np.random.default_rng(9)
    side = 14 * 104
    img = synth.make_image(rng, side, side, 9, 9, 0.3) if kind == "natural" else np.full((side, side, 3), 120, np.uint8)
    n = 104 * 104
    for q in (rng.choice(n, size=n // 2 if kind == "steps" else n // 20, replace=False) if kind != "natural" else ()):
        y, x = divmod(int(q), 104)
        p = img[14 * y:14 * y + 14, 14 * x:14 * x + 14]
        if kind == "equal":
            p[:] = rng.integers(0, 256, p.shape, dtype=np.uint8)
        else:
            p[:7] = 120 + (q % 5)   # a few nearby values: thousands of distances in one bucket, five of them different
    d, st = pace.pace_apc_density(torch.from_numpy(img.reshape(-1)).cuda(), [0], [side], [side])
    ref = O.apc_density(img)
    assert_tight(d.cpu().numpy(), ref["d"])
    # the tail of the GPU's own distances, exactly up to fp32 rounding of the mean
    k = pace.stats_dict(st)[0]["k_tail"]
    top = np.sort(d.cpu().numpy().astype(np.float64))[::-1][:k].mean()
    assert abs(pace.stats_dict(st)[0]["d_top"] - top) <= 4e-7 * top + 1e-9


# the tail's bucket: ranked directly (up to 128 members), by rounds over the list (up to 4096), over the
# whole array, in one CTA (up to 8192 distances) and a cluster; in the first bucket and in another, a few
# and many different distances
@pytest.mark.parametrize("n", [128, 129, 256, 257, 600, 4096, 4300, 9000, 70000])
@pytest.mark.parametrize("offset,values", [(0.0, 3), (0.0, 128), (0.5, 2), (0.5, 128)])
def test_tail_members(pace, n, offset, values):
    rng = np.random.default_rng(n)
    # unit-ish tokens (1, +-offset, y): y moves the distance to the mean by less than a bucket (2^-11)
    T = np.zeros((n, 8))
    T[:, 0], T[:, 1] = 1.0, offset * np.where(np.arange(n) % 2, 1, -1)
    T[:, 2] = rng.integers(0, values, n) * ((2.0 ** -12 if offset == 0.0 else 2.0 ** -6) / values)
    bits = synth.f32_to_bf16_bits(T.astype(np.float32))
    d, st = pace.pace_apc_density_tokens(bf16_tensor(bits), [0, n], [252], [252])
    d, s = d.cpu().numpy(), pace.stats_dict(st)[0]
    assert_tight(d, O.apc_density_preview(f64(bits), 252, 252)["d"])
    top = np.sort(d.astype(np.float64))[::-1][:s["k_tail"]].mean()
    # fixed point of 2^-32 per distance, fp32 rounding of the mean
    assert abs(s["d_top"] - top) <= 4e-7 * top + 2.0 ** -32


# distances counted per warp (pictures: the first and the last live lane's bucket at once, the rest one
# by one) and per run of equal buckets (tokens): all equal, two values in turn, background with few or
# many others among it, partial warps
@pytest.mark.parametrize("kind", ["all", "two", "few", "half", "most", "none"])
@pytest.mark.parametrize("rows,cols", [(1, 3), (3, 33), (40, 60)])
def test_tail_counts_of_backgrounds(pace, kind, rows, cols):
    rng = np.random.default_rng(rows * cols)
    n, h, w = rows * cols, rows * 14, cols * 14
    share = {"all": 0.0, "two": 0.0, "few": 0.1, "half": 0.5, "most": 0.9, "none": 1.0}[kind]
    noise = rng.uniform(size=n) < share
    img = np.full((h, w, 3), 40, np.uint8)
    for q in range(n):
        y, x = divmod(q, cols)
        p = img[14 * y:14 * y + 14, 14 * x:14 * x + 14]
        if noise[q]:
            p[:] = rng.integers(0, 256, p.shape, dtype=np.uint8)
        elif kind == "two" and q % 2:
            p[:, :7] = 200

    def check(d, st):
        d = d.cpu().numpy().astype(np.float64)
        s = pace.stats_dict(st)[0]
        top = np.sort(d)[::-1][:s["k_tail"]].mean()
        assert abs(s["d_top"] - top) <= 4e-7 * top + 1e-9   # fp32 rounding of the mean
        return d

    src = torch.from_numpy(img.reshape(-1)).cuda()
    assert_tight(check(*pace.pace_apc_density(src, [0], [h], [w])), O.apc_density(img)["d"])
    check(*pace.pace_apc_density_pixel(src, [0], [h], [w], "rgb_stats"))
    T = np.where(noise[:, None], rng.normal(size=(n, 64)), 1.0 + (kind == "two") * (np.arange(n)[:, None] % 2) * np.arange(64))
    bits = synth.f32_to_bf16_bits(T.astype(np.float32))
    d = check(*pace.pace_apc_density_tokens(bf16_tensor(bits), [0, n], [h], [w]))
    assert_tight(d, O.apc_density_preview(f64(bits), w, h)["d"])


# more images than one table holds: the second table's feature kernel follows the first one's tail
def test_pixel_density_two_tables(pace):
    rng = np.random.default_rng(7)
    shapes = [(14 * int(a), 14 * int(b)) for a, b in rng.integers(1, 9, (70, 2))]
    buf, off = synth.pack_images([rng.integers(0, 256, (*s, 3), dtype=np.uint8) for s in shapes])
    H, W, src = [s[0] for s in shapes], [s[1] for s in shapes], torch.from_numpy(buf).cuda()
    n = [h * w // 196 for h, w in shapes]
    for f in ("rgb_stats", "color_entropy", "edge_density", "laplacian"):
        d, st = pace.pace_apc_density_pixel(src, off, H, W, f)
        for b in (0, 1, 62, 63, 64, 65, 69):   # each alone gives the same
            one, s = pace.pace_apc_density_pixel(src, [int(off[b])], [H[b]], [W[b]], f)
            assert torch.equal(one, d[sum(n[:b]):sum(n[:b + 1])]) and torch.equal(s[0], st[b])


# register kernels (whole 16-byte vectors, up to 1536) and the staged ones (other widths), runs of 8
# tokens with remainders, several images per CTA
@pytest.mark.parametrize("D", [8, 248, 256, 264, 1152, 1536, 1544, 1284, 6])
@pytest.mark.parametrize("lens", [(1,), (7, 8, 9), (300, 1, 2500)])
def test_token_widths(pace, D, lens):
    rng = np.random.default_rng(D)
    cu = _cu(lens)
    T = rng.normal(size=D)[None] * rng.uniform(0.5, 2, (int(cu[-1]), 1)) + rng.normal(size=(int(cu[-1]), D))
    T[0] = 0
    bits = synth.f32_to_bf16_bits(T.astype(np.float32))
    sides = [28 * 9] * len(lens)
    d, st = pace.pace_apc_density_tokens(bf16_tensor(bits), cu, sides, sides)
    d = d.cpu().numpy()
    for b, s in enumerate(pace.stats_dict(st)):
        ref = O.apc_density_preview(f64(bits)[cu[b]:cu[b + 1]], 252, 252)
        assert_tight(d[cu[b]:cu[b + 1]], ref["d"])
        assert abs(s["phi"] - ref["phi"]) <= TIGHT and abs(s["d_top"] - ref["d_top"]) <= TIGHT
    # the same bits in any batch
    one, _ = pace.pace_apc_density_tokens(bf16_tensor(bits[cu[-2]:cu[-1]]), [0, lens[-1]], [252], [252])
    np.testing.assert_array_equal(one.cpu().numpy(), d[cu[-2]:cu[-1]])


# tokens that start on a 4-byte, not a 16-byte boundary take the staged kernels: the same statistics
def test_tokens_unaligned_start(pace):
    rng = np.random.default_rng(8)
    bits = synth.f32_to_bf16_bits(rng.normal(0.4, 1.0, size=(700, 256)).astype(np.float32))
    flat = torch.empty(bits.size + 2, dtype=torch.bfloat16, device="cuda")
    flat[2:].copy_(bf16_tensor(bits).reshape(-1))
    shifted = flat[2:].view(700, 256)
    assert shifted.data_ptr() % 16 == 4
    ref = O.apc_density_preview(f64(bits), 252, 252)
    for T in (shifted, bf16_tensor(bits)):
        d, st = pace.pace_apc_density_tokens(T, [0, 700], [252], [252])
        s = pace.stats_dict(st)[0]
        assert_tight(d.cpu().numpy(), ref["d"])
        assert abs(s["phi"] - ref["phi"]) <= TIGHT and abs(s["d_top"] - ref["d_top"]) <= TIGHT


def test_tokens_with_non_finite_rows(pace):
    """A NaN or infinite token spoils its own distance and leaves the others finite."""
    rng = np.random.default_rng(2)
    T = rng.normal(size=(64, 256)).astype(np.float32)
    bits = synth.f32_to_bf16_bits(T)
    bits[20, 3], bits[41, 7] = 0x7FC0, 0x7F80
    d, _ = pace.pace_apc_density_tokens(bf16_tensor(bits), [0, 64], [252], [252])
    bad = ~np.isfinite(d.cpu().numpy())
    assert bad[20] and bad.sum() <= 2 and not bad[:20].any()


# |T|^2 of 1.125 and 1.477 units of the smallest subnormal is rounded to one: normalised, such tokens are a little
# longer than 1, by either kind of kernel, and must not count as nothing
@pytest.mark.parametrize("D", [256, 250])
@pytest.mark.parametrize("mantissa", [1.5, 1.71875])
def test_tokens_with_subnormal_squares(pace, D, mantissa):
    T = np.zeros((40, D), np.float32)
    T[:, 5] = mantissa * 2.0 ** -75
    d, st = pace.pace_apc_density_tokens(bf16_tensor(synth.f32_to_bf16_bits(T)), [0, 40], [252], [252])
    s, sq = pace.stats_dict(st)[0], mantissa * mantissa / 2   # |T|^2 over its rounded value
    assert abs(s["phi"] - sq) <= 1e-6 and bool((d <= 1e-6 + sq ** 0.5 - 1).all())


# scales 1 to 8 per side (filtered vertically first) and just above (generic), widths on 2-byte
# boundaries, one and several column strips, heights below a group of four rows, odd sizes
@pytest.mark.parametrize("shape,size", [((14, 14), (14, 14)), ((14, 14), (1, 1)), ((28, 14), (3, 2)), ((98, 42), (97, 41)),
                                        ((70, 1302), (35, 1301)), ((42, 2030), (30, 600)), ((560, 70), (70, 9)),
                                        ((560, 70), (69, 9)), ((126, 1036), (125, 130)), ((126, 1036), (45, 129)),
                                        ((700, 700), (501, 88))])
def test_resample_scales(pace, shape, size):
    rng = np.random.default_rng(shape[0] + size[1])
    img = synth.make_image(rng, *shape, 3, 3, 0.5)
    dst = torch.zeros(shape[0] * shape[1] * 3, dtype=torch.uint8, device="cuda")
    pace.pace_apc_resample_to(torch.from_numpy(img.reshape(-1)).cuda(), [0], [shape[0]], [shape[1]], [size[0]], [size[1]], dst, [0])
    n = size[0] * size[1] * 3
    out, ref = dst.cpu().numpy()[:n].reshape(*size, 3), O.apc_resample(img, *size)
    assert np.abs(out.astype(int) - ref.astype(int)).max() <= 1
    # bytes off by one are those whose exact value is within rounding of a half
    x = O.resample_float(img, *size)
    assert np.all(np.abs(x - np.floor(x) - 0.5)[out != ref] <= 2e-4)
    assert not dst[n:].any()


# an image alone (tiles of at most a column per thread) and the same one in a batch (wide tiles, other
# heights): the same bytes, whatever the tiles; aligned rows and rows on 2-byte boundaries
@pytest.mark.parametrize("shape,size", [((448, 448), (190, 190)), ((448, 448), (448, 401)), ((434, 462), (300, 257)),
                                        ((336, 322), (41, 129))])
def test_resample_tile_widths(pace, shape, size):
    rng = np.random.default_rng(size[1])
    img = synth.make_image(rng, *shape, 3, 3, 0.5)
    ref = O.apc_resample(img, *size).astype(int)
    n, pad = size[0] * size[1] * 3, (img.size + 255) // 256 * 256
    outs = []
    for B in (1, 24):
        src = torch.zeros(B, pad, dtype=torch.uint8, device="cuda")
        src[:, :img.size] = torch.from_numpy(img.reshape(-1)).cuda()
        dst, off = torch.zeros_like(src), [pad * b for b in range(B)]
        pace.pace_apc_resample_to(src.view(-1), off, [shape[0]] * B, [shape[1]] * B, [size[0]] * B, [size[1]] * B, dst.view(-1), off)
        outs.append(dst[:, :n])
        assert not dst[:, n:].any()
    assert np.abs(outs[0][0].cpu().numpy().reshape(*size, 3).astype(int) - ref).max() <= 1
    assert (outs[1] == outs[0]).all()


# small outputs (8 x 32 tiles) and the same image beside a large one (wide tiles): the same bytes; 2.75 per side and
# just above, tiles with remainders and below one tile, the image's last bytes, rows on 2-byte boundaries
@pytest.mark.parametrize("shape,size", [((14, 14), (14, 14)), ((14, 14), (6, 6)), ((28, 14), (11, 6)), ((308, 308), (112, 112)),
                                        ((308, 434), (112, 158)), ((308, 308), (111, 112)), ((42, 2030), (33, 740)),
                                        ((700, 28), (257, 27)), ((434, 462), (300, 257)), ((98, 896), (65, 544))])
def test_resample_small_tiles(pace, shape, size):
    rng = np.random.default_rng(shape[1] + size[1])
    img = rng.integers(0, 256, (*shape, 3), dtype=np.uint8)
    img[-1, -1] = 255
    n, big = size[0] * size[1] * 3, (1344, 1344)
    pad = (img.size + 255) // 256 * 256
    src = torch.zeros(pad + big[0] * big[1] * 3, dtype=torch.uint8, device="cuda")
    src[:img.size] = torch.from_numpy(img.reshape(-1)).cuda()
    one, two = torch.full_like(src, 7), torch.full_like(src, 7)
    pace.pace_apc_resample_to(src, [0], shape[:1], shape[1:], size[:1], size[1:], one, [0])
    pace.pace_apc_resample_to(src, [0, pad], [shape[0], big[0]], [shape[1], big[1]], [size[0], big[0]], [size[1], big[1]], two, [0, pad])
    assert torch.equal(one[:n], two[:n]) and bool((one[n:] == 7).all()) and bool((two[n:pad] == 7).all())
    assert np.abs(one[:n].cpu().numpy().reshape(*size, 3).astype(int) - O.apc_resample(img, *size).astype(int)).max() <= 1


# a batch in small tiles, more images than a warp has lanes, among them one with nothing to write
def test_resample_small_batch(pace):
    rng = np.random.default_rng(5)
    shapes = [(14 * int(a), 14 * int(b)) for a, b in rng.integers(1, 5, (40, 2))]
    sizes = [tuple(int(rng.integers(-(-4 * x // 11), x + 1)) for x in s) for s in shapes]
    off = np.concatenate([[0], np.cumsum([(h * w * 3 + 255) // 256 * 256 for h, w in shapes])])
    src = torch.from_numpy(rng.integers(0, 256, int(off[-1]), dtype=np.uint8)).cuda()
    # sizes read on the device; image 33's is out of range
    stats = torch.zeros((40, 10), dtype=torch.int32, device="cuda")
    stats[:, 8:10] = torch.tensor(sizes, dtype=torch.int32)
    stats[33, 8] = 0
    got = torch.full_like(src, 7)
    pace.pace_apc_resample(src, off[:-1].tolist(), [s[0] for s in shapes], [s[1] for s in shapes], stats, got, off[:-1].tolist())
    want = torch.full_like(src, 7)
    for b in range(40):
        if b != 33:
            pace.pace_apc_resample_to(src, [int(off[b])], shapes[b][:1], shapes[b][1:], sizes[b][:1], sizes[b][1:], want, [int(off[b])])
    assert torch.equal(got, want)


# steep downscales: tiles of eight rows where a call has many, else of four, remainders of both: the same bytes
@pytest.mark.parametrize("size", [(124, 124), (121, 97)])
def test_resample_generic_heights(pace, size):
    rng = np.random.default_rng(size[0])
    H = W = 1036
    img = synth.make_image(rng, H, W, 9, 9, 0.5)
    n, outs = size[0] * size[1] * 3, []
    pad = (img.size + 255) // 256 * 256
    for B in (1, 8):
        src = torch.zeros(B, pad, dtype=torch.uint8, device="cuda")
        src[:, :img.size] = torch.from_numpy(img.reshape(-1)).cuda()
        dst, off = torch.zeros_like(src), [pad * b for b in range(B)]
        pace.pace_apc_resample_to(src.view(-1), off, [H] * B, [W] * B, [size[0]] * B, [size[1]] * B, dst.view(-1), off)
        outs.append(dst)
    assert (outs[1][:, :n] == outs[0][0, :n]).all() and not outs[1][:, n:].any()
    assert np.abs(outs[0][0, :n].cpu().numpy().reshape(*size, 3).astype(int) - O.apc_resample(img, *size).astype(int)).max() <= 1


# every call's first kernel may be launched while the stream's previous work runs: inputs written right
# before a call, scratch and outputs used again right after one, in a stream and in a captured graph
@pytest.mark.parametrize("captured", [False, True])
def test_calls_back_to_back(pace, captured):
    from paper_2608_27206_gb300.hotpath import HotPath
    hp = HotPath(synth.make_workload("img448", seed=3), "cuda")
    names = ("stats", "dist", "resized", "s_vis", "s_llm", "s_final", "weights", "kept", "rows")
    inputs = {k: v.clone() for k, v in hp.d.items()}
    other = {k: (255 - v if k == "img" else -v.flip(0)) for k, v in inputs.items()}

    def run(src, sync):
        for _, call in hp.parts:
            for k, v in src.items():   # written just before each call
                hp.d[k].copy_(v)
            call()
            if sync:
                torch.cuda.synchronize()
        return {k: getattr(hp, k).clone() for k in names}

    want = [run(s, True) for s in (inputs, other)]
    torch.cuda.synchronize()
    stream, rounds = torch.cuda.Stream(), 5
    with torch.cuda.stream(stream):
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                out = [run(s, False) for s in (inputs, other)]
            got = []
            for _ in range(rounds):
                g.replay()
                got += [{k: v.clone() for k, v in o.items()} for o in out]
        else:
            got = [run(s, False) for _ in range(rounds) for s in (inputs, other)]
    torch.cuda.synchronize()
    for i, o in enumerate(got):
        for k in names:
            assert torch.equal(o[k].view(torch.uint8), want[i % 2][k].view(torch.uint8)), (i, k)


# the calls that the path above leaves out, each twice on one scratch with other inputs and never synchronised:
# their first kernels write scratch before they wait for earlier work, and the next call's may start early
@pytest.mark.parametrize("captured", [False, True])
def test_other_calls_back_to_back(pace, captured):
    rng = np.random.default_rng(4)
    H, W = [448, 224, 154], [448, 308, 14 * 40]
    n = sum(h * w for h, w in zip(H, W)) // 196
    buf, off = synth.pack_images([rng.integers(0, 256, (h, w, 3), dtype=np.uint8) for h, w in zip(H, W)])
    cu = _cu([h * w // 196 for h, w in zip(H, W)])
    seq, vis, nv, hq, hk = [0, 300, 700], [10, 0], [200, 333], 14, 2
    img, kept = torch.from_numpy(buf).cuda(), torch.arange(0, 533, 5, dtype=torch.int32, device="cuda")
    keep = _cu([40, 67])
    T = {D: bf16_tensor(synth.f32_to_bf16_bits(rng.normal(size=(n, D)).astype(np.float32))) for D in (256, 250)}
    q, k = (bf16_tensor(synth.random_small_qk(i, 700, h, 128)) for i, h in ((1, hq), (2, hk)))
    hid = torch.from_numpy(rng.integers(0, 255, (700, 1024), dtype=np.uint8)).cuda()
    pos = torch.arange(3 * 700, dtype=torch.int32, device="cuda").view(3, 700)
    inputs = [img, *T.values(), q, k, hid, pos]
    first = [x.clone() for x in inputs]
    other = [x.flip(0).contiguous() if i else 255 - x for i, x in enumerate(first)]
    d, st = torch.empty(n, device="cuda"), torch.zeros((3, 10), dtype=torch.int32, device="cuda")
    ws = torch.empty(max(pace.pace_apc_density_workspace_size(H, W), pace.pace_apc_density_pixel_workspace_size(H, W),
                         *(pace.pace_apc_density_tokens_workspace_size(cu, D) for D in T),
                         pace.pace_llm_sequence_importance_workspace_size(seq, vis, nv, hq, hk)), dtype=torch.uint8, device="cuda")
    tok, s_llm = torch.empty((n, 8), device="cuda"), torch.empty(533, device="cuda")
    idx = torch.empty(700 - 533 + 107, dtype=torch.int32, device="cuda")
    dst = torch.empty((idx.numel(), 1024), dtype=torch.uint8, device="cuda")
    dpos, small = torch.empty((3, idx.numel()), dtype=torch.int32, device="cuda"), torch.zeros_like(img)

    def gather():
        pace.pace_prune_index(seq, vis, [0, 200, 533], keep, kept, out=idx)
        pace.pace_gather_multi([pace.gather_spec(hid, dst, 0), pace.gather_spec(pos, dpos, 1)], idx)

    def chain():   # a resized image is the next call's picture, a gathered row list the next gather's
        pace.pace_apc_resample_to(img, off, H, W, [h // 2 // 14 * 14 for h in H], [w // 2 // 14 * 14 for w in W], small, off)
        pace.pace_apc_density(small, off, [h // 2 // 14 * 14 for h in H], [w // 2 // 14 * 14 for w in W], d_out=d, stats=st, ws=ws)

    calls = [(lambda D=D: pace.pace_apc_density_tokens(T[D], cu, H, W, d_out=d, stats=st, ws=ws), (d, st)) for D in T]
    calls += [(lambda f=f: pace.pace_apc_density_pixel(img, off, H, W, f, d_out=d, stats=st, ws=ws), (d, st))
              for f in ("edge_density", "rgb_stats")]
    calls += [(lambda: pace.pace_apc_pixel_features(img, off, H, W, "laplacian", out=tok), (tok,)),
              (lambda: pace.pace_apc_density_static(img, off, H, W, d_out=d, stats=st), (d, st)),
              (lambda: pace.pace_llm_sequence_importance(q, k, seq, vis, nv, out=s_llm, ws=ws), (s_llm,)),
              (gather, (idx, dst, dpos)), (chain, (small, d, st))]

    def run(sync):
        out = []
        for call, results in calls:
            for src in (first, other):
                for x, y in zip(inputs, src):
                    x.copy_(y)
                call()
                call()
                out += [r.clone() for r in results]
                if sync:
                    torch.cuda.synchronize()
        return out

    pace.pace_apc_density_static(img, off, H, W, d_out=d, stats=st)   # (its first call looks its scratch up)
    want = run(True)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                out = run(False)
            g.replay()
            g.replay()
        else:
            run(False)
            out = run(False)
    torch.cuda.synchronize()
    for i, (a, b) in enumerate(zip(out, want)):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), i


# scores held in registers for 4, 8 and 12 per thread of a block of 1024, and read again per pass above
@pytest.mark.parametrize("n", [4096, 4097, 8192, 8193, 12288, 12289, 16384, 20481])
def test_select_registers(pace, n):
    rng = np.random.default_rng(n)
    # one map for both: S_final is the map itself when it spans [0, 1] and the weights are 1/2
    x = (rng.permutation(n).astype(np.float32) / np.float32(1 << (14 if n <= 16384 else 15))).astype(np.float32)
    x[rng.integers(1, n - 1)] = 1.0
    x[0] = 0.0
    K = O.budget(n, 0.1)
    s = torch.from_numpy(x).cuda()
    s_final, w, kept = pace.pace_ddae_select(s, s, [0, n], [0, K])
    np.testing.assert_array_equal(s_final.cpu().numpy(), x)
    assert w.cpu().numpy().tolist() == [[0.5, 0.5]]
    np.testing.assert_array_equal(kept.cpu().numpy(), O.top_k_ascending(x.astype(np.float64), K))
