"""GPU parity of MLA causal chunk attention (pre-fill) over the latent cache,
bf16 and quantised, through the C ABI: every query row of the chunk attends
to its own causal prefix with the absorbed query (the decode path per row),
against the oracle's unabsorbed chunk attention on the dequantised cache.
Ragged lengths, one sequence shorter than the chunk, an inheriting layer;
bf16 chunks of an even number of rows decode two rows per CTA at d >= 256
(a pair may hold an empty row beside a one-position row), odd ones one."""
import ctypes
import math

import numpy as np
import pytest
import torch

from _parity import assert_close, f32
from oracle import attention as oatt
from oracle import cache as ocache

pytestmark = pytest.mark.gpu

H = 16


def _setup(width, fmt, lens, T, seed, H=H):
    from paper_2609_37988_gb300.cache import Cache, Layer
    B = len(lens)
    layer = dict(bits=16, width=width) if fmt is None else dict(bits=fmt[1], scheme=fmt[0], width=width)
    c = Cache(kind="mla", n_layers=2, n_q_heads=H, head_dim=128, latent_dim=512, rope_dim=64,
              max_batch=B, max_ctx=T, layers=[Layer(**layer), Layer(inherit=True)], max_splits=16)
    g = torch.Generator().manual_seed(seed)
    decay = torch.arange(512).add(1.0).rsqrt()
    n = max(lens)
    cl = (torch.randn((B, n, 512), generator=g) * decay).to(torch.bfloat16)
    kr = torch.randn((B, n, 64), generator=g).to(torch.bfloat16)
    c.append(0, cl.cuda(), kr.cuda(), n_per_seq=torch.tensor(lens, dtype=torch.int32, device="cuda"))
    wk = (torch.randn((H, 128, 512), generator=g) / math.sqrt(512)).to(torch.bfloat16)
    wv = (torch.randn((H, 128, 512), generator=g) / math.sqrt(512)).to(torch.bfloat16)
    if fmt is None:
        c_hat, kr_hat = f32(cl), f32(kr)
    else:
        st = ocache.mla_anchor_state(f32(cl), f32(kr), lens, width, fmt[1], fmt[0])
        c_hat, kr_hat = st["c_hat"], st["kr_hat"]
    return c, wk, wv, c_hat, kr_hat


@pytest.mark.parametrize("width,fmt", [(512, None), (64, None), (256, ("grouped", 8)),
                                       (128, ("symmetric", 4)), (512, ("symmetric", 2))],
                         ids=["bf16-d512", "bf16-d64", "g8-d256", "sym4-d128", "sym2-d512"])
def test_mla_prefill_parity(width, fmt):
    lens, n_q = [300, 129, 20], 40
    c, wk, wv, c_hat, kr_hat = _setup(width, fmt, lens, 320, seed=width + (fmt[1] if fmt else 16))
    g = torch.Generator().manual_seed(5)
    qn = torch.randn((len(lens), n_q, H, 128), generator=g).to(torch.bfloat16)
    qp = torch.randn((len(lens), n_q, H, 64), generator=g).to(torch.bfloat16)
    sigma = 1.0 / math.sqrt(192)
    out = c.prefill_mla(0, qn.cuda(), qp.cuda(), wk.cuda(), wv.cuda(), sigma)
    ref = oatt.mla_prefill_unabsorbed(f32(qn), f32(qp), c_hat, kr_hat, f32(wk), f32(wv), width, lens, sigma)
    assert_close(f32(out), ref, what=f"mla prefill d={width} {fmt}")
    # queries before position 0 give zeros; the inheritor reads the anchor
    assert (f32(out[2, : n_q - lens[2]]) == 0).all()
    again = c.prefill_mla(1, qn.cuda(), qp.cuda(), wk.cuda(), wv.cuda(), sigma)
    assert torch.equal(out, again)
    # the last query of each sequence is one decode step
    dec = c.decode_mla(0, qn[:, -1].contiguous().cuda(), qp[:, -1].contiguous().cuda(), wk.cuda(),
                       wv.cuda(), sigma)
    assert_close(f32(out[:, -1]), f32(dec), max_abs=2e-4, rel_l2=1e-4, what="last query = decode")
    assert c.device_error() == 0


def test_mla_prefill_rejections():
    from paper_2609_37988_gb300._lib import KVKError
    c, wk, wv, _, _ = _setup(64, None, [10, 10], 64, seed=1)
    qn = torch.zeros((2, 4, H, 128), dtype=torch.bfloat16, device="cuda")
    qp = torch.zeros((2, 4, H, 64), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(KVKError):
        c.prefill_mla(0, qn, qp, wk.cuda(), wv.cuda(), 0.0)  # scale
    with pytest.raises(KVKError):
        c.prefill_mla(0, torch.zeros((2, 65, H, 128), dtype=torch.bfloat16, device="cuda"),
                      torch.zeros((2, 65, H, 64), dtype=torch.bfloat16, device="cuda"), wk.cuda(),
                      wv.cuda(), 0.1)  # n_q > max_ctx


@pytest.mark.parametrize("width,n_q,heads", [(512, 40, 10), (512, 39, 16), (256, 40, 5), (256, 2, 16),
                                              (128, 40, 16)],
                         ids=["d512-pairs-h10", "d512-odd-rows", "d256-pairs-h5", "d256-one-pair", "d128-rows"])
def test_mla_prefill_row_pairs(width, n_q, heads):
    """Two rows per CTA: each row masks its own causal end inside the shared
    tiles; fewer than 16 heads; an odd row count keeps one row per CTA."""
    lens = [301, 130, 21]
    c, wk, wv, c_hat, kr_hat = _setup(width, None, lens, 320, seed=width + n_q, H=heads)
    g = torch.Generator().manual_seed(6)
    qn = torch.randn((len(lens), n_q, heads, 128), generator=g).to(torch.bfloat16)
    qp = torch.randn((len(lens), n_q, heads, 64), generator=g).to(torch.bfloat16)
    sigma = 1.0 / math.sqrt(192)
    out = c.prefill_mla(0, qn.cuda(), qp.cuda(), wk.cuda(), wv.cuda(), sigma)
    ref = oatt.mla_prefill_unabsorbed(f32(qn), f32(qp), c_hat, kr_hat, f32(wk), f32(wv), width, lens, sigma)
    assert_close(f32(out), ref, what=f"mla prefill pairs d={width} n_q={n_q} H={heads}")
    empty = max(0, n_q - lens[2])
    assert (f32(out[2, :empty]) == 0).all()
    if empty < n_q:
        assert (np.abs(f32(out[2, empty])) > 0).any()  # the one-position row
    assert c.device_error() == 0


def _scratch(c, n_q):
    out = ctypes.c_size_t()
    assert c.lib.kvk_prefill_scratch_size(c.handle, 0, n_q, ctypes.byref(out)) == 0
    return out.value


@pytest.mark.parametrize("width,fmt", [(512, None), (256, None), (128, None), (64, None), (512, ("grouped", 8)),
                                       (256, ("grouped", 4)), (128, ("symmetric", 8)), (64, ("symmetric", 4)),
                                       (512, ("symmetric", 2))],
                         ids=lambda x: str(x) if isinstance(x, int) else "bf16" if x is None else f"{x[0][:3]}{x[1]}")
@pytest.mark.parametrize("n_q,heads", [(256, 16), (387, 5)], ids=["nq256", "nq387-h5"])
def test_mla_prefill_formed(width, fmt, n_q, heads):
    """Chunks long enough to attend over keys and values formed per head: two
    whole row blocks and a remainder, lengths at, one past and one short of
    the 64- and 128-position blocks, sequences shorter than the chunk and an
    empty one."""
    lens = [385, 256, 191, 20, 0, 129]
    c, wk, wv, c_hat, kr_hat = _setup(width, fmt, lens, 400, seed=width + n_q, H=heads)
    g = torch.Generator().manual_seed(7)
    qn = torch.randn((len(lens), n_q, heads, 128), generator=g).to(torch.bfloat16)
    qp = torch.randn((len(lens), n_q, heads, 64), generator=g).to(torch.bfloat16)
    sigma = 1.0 / math.sqrt(192)
    assert _scratch(c, n_q) == _scratch(c, 400)  # the formed tiles' size, which no chunk changes
    out = c.prefill_mla(0, qn.cuda(), qp.cuda(), wk.cuda(), wv.cuda(), sigma)
    ref = oatt.mla_prefill_unabsorbed(f32(qn), f32(qp), c_hat, kr_hat, f32(wk), f32(wv), width, lens, sigma)
    assert_close(f32(out), ref, what=f"formed d={width} {fmt} n_q={n_q} H={heads}")
    assert (f32(out[3, : n_q - 20]) == 0).all() and (f32(out[4]) == 0).all()
    assert c.device_error() == 0


@pytest.mark.parametrize("cap", [262144, 65536], ids=["head-groups", "sequence-groups"])
def test_mla_prefill_formed_groups(cap):
    """Contexts whose formed tiles pass 2 GiB: the heads (262144 positions: 8
    heads at a time) or the sequences (65536: 2 of 3 at a time) go in groups
    through the same scratch.  The same call over a small cache is equal."""
    lens, n_q = [333, 70, 200], 300
    outs = []
    for T in (cap, 400):
        n = lens if T != 262144 and cap != 262144 else lens[:1]
        c, wk, wv, _, _ = _setup(512, None, n, T, seed=3)
        g = torch.Generator().manual_seed(8)
        qn = torch.randn((len(n), n_q, H, 128), generator=g).to(torch.bfloat16)
        qp = torch.randn((len(n), n_q, H, 64), generator=g).to(torch.bfloat16)
        outs.append(f32(c.prefill_mla(0, qn.cuda(), qp.cuda(), wk.cuda(), wv.cuda(), 0.07)))
        assert c.device_error() == 0
    assert np.array_equal(outs[0], outs[1])


def test_mla_prefill_scratch_limits():
    """The scratch size never shrinks with the chunk; a buffer that holds the
    absorbed path's rows but not the formed tiles still serves the call."""
    c, wk, wv, _, _ = _setup(512, None, [300, 80], 8192, seed=9)
    sizes = [_scratch(c, n) for n in list(range(1, 321)) + [1000, 8192]]
    assert sizes == sorted(sizes)
    n_q = 200
    g = torch.Generator().manual_seed(4)
    qn = torch.randn((2, n_q, H, 128), generator=g).to(torch.bfloat16).cuda()
    qp = torch.randn((2, n_q, H, 64), generator=g).to(torch.bfloat16).cuda()
    wk, wv = wk.cuda(), wv.cuda()
    full = c.prefill_mla(0, qn, qp, wk, wv, 0.07)
    rows = 2 * n_q * H
    small = rows * (2 * 512 + 64) * 2 + 256 + rows * 514 * 4  # absorbed queries and latent partials
    assert 1024 < small < _scratch(c, n_q) == sizes[-1]
    out = torch.empty_like(full)
    buf = torch.empty(small, dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    args = (c.handle, 0, p(qn), p(qp), p(wk), p(wv), n_q, 0.07, p(out), p(buf))
    assert c.lib.kvk_prefill_attention_mla(*args, small, ctypes.c_void_p(st)) == 0
    assert_close(f32(out), f32(full), max_abs=2e-4, rel_l2=1e-4, what="absorbed = formed")
    assert c.lib.kvk_prefill_attention_mla(*args, 1024, ctypes.c_void_p(st)) != 0
    assert c.device_error() == 0


@pytest.mark.parametrize("width,fmt", [(512, None), (64, None), (128, ("symmetric", 8))],
                         ids=["bf16-d512", "bf16-d64", "sym8-d128"])
def test_mla_prefill_non_finite_latents_stay_with_their_readers(width, fmt):
    """A latent with an infinite coordinate spoils the rows that see its
    position and no others, formed keys and values or not."""
    from paper_2609_37988_gb300.cache import Cache, Layer
    T, n_q, at = 700, 600, 555
    layer = dict(bits=16, width=width) if fmt is None else dict(bits=fmt[1], scheme=fmt[0], width=width)
    g = torch.Generator().manual_seed(9)
    cl = torch.randn((2, T, 512), generator=g).to(torch.bfloat16)
    kr = torch.randn((2, T, 64), generator=g).to(torch.bfloat16)
    wk, wv = ((torch.randn((H, 128, 512), generator=g) / math.sqrt(512)).to(torch.bfloat16).cuda() for _ in range(2))
    qn = torch.randn((2, n_q, H, 128), generator=g).to(torch.bfloat16).cuda()
    qp = torch.randn((2, n_q, H, 64), generator=g).to(torch.bfloat16).cuda()
    dirty = cl.clone()
    dirty[1, at, 7] = math.inf
    outs = []
    for x in (cl, dirty):
        c = Cache(kind="mla", n_layers=1, n_q_heads=H, head_dim=128, latent_dim=512, rope_dim=64, max_batch=2,
                  max_ctx=T, layers=[Layer(**layer)])
        c.append(0, x.cuda(), kr.cuda())
        outs.append(f32(c.prefill_mla(0, qn, qp, wk, wv, 0.07)).copy())
        assert c.device_error() == 0
    clean, out = outs
    first = at - (T - n_q)
    assert np.array_equal(out[0], clean[0])
    assert np.array_equal(out[1, :first], clean[1, :first])
    assert np.isnan(out[1, first:]).all()


@pytest.mark.parametrize("fmt", [None, ("symmetric", 4)], ids=["bf16", "sym4"])
@pytest.mark.parametrize("steep", [0.02, 1.0], ids=["flat", "steep"])
def test_mla_prefill_formed_scales_and_flushes(fmt, steep):
    """Formed values stored relative to a power of two per 32 positions
    (zero, tiny and large latents side by side, the first ones zero) and
    partial results that leave the accumulator every 16 (4-bit) or 32 tiles:
    8450 positions, four flushes and more or two, a whole last round.  An
    output that starts on 16 bytes but not on 32.  Bound: the accumulator
    drops up to 2^-24 of itself per 16 positions of a round, 32 x 8 x 2^-24 =
    1.5e-5 at most, 2e-5 with the other roundings (2^-20)."""
    T, n_q, heads = 8450, 200, 4
    from paper_2609_37988_gb300.cache import Cache, Layer
    layer = dict(bits=16, width=512) if fmt is None else dict(bits=fmt[1], scheme=fmt[0], width=512)
    g = torch.Generator().manual_seed(21)
    e = torch.randint(-20, 3, (T // 32 + 1,), generator=g)
    e[:3] = -200  # zeros
    e[70:73] = -200
    scale = torch.exp2(e.double()).float().repeat_interleave(32)[:T]
    cl = (torch.randn((1, T, 512), generator=g) * torch.arange(512).add(1.0).rsqrt() * scale[None, :, None])
    cl = cl.to(torch.bfloat16)
    kr = torch.randn((1, T, 64), generator=g).to(torch.bfloat16)
    wk = (torch.randn((heads, 128, 512), generator=g) / math.sqrt(512)).mul(steep).to(torch.bfloat16)
    wv = (torch.randn((heads, 128, 512), generator=g) / math.sqrt(512)).to(torch.bfloat16)
    qn = torch.randn((1, n_q, heads, 128), generator=g).to(torch.bfloat16)
    qp = torch.randn((1, n_q, heads, 64), generator=g).to(torch.bfloat16)
    c = Cache(kind="mla", n_layers=1, n_q_heads=heads, head_dim=128, latent_dim=512, rope_dim=64, max_batch=1,
              max_ctx=T, layers=[Layer(**layer)])
    c.append(0, cl.cuda(), kr.cuda())
    sigma = 1.0 / math.sqrt(192)
    args = (qn.cuda(), qp.cuda(), wk.cuda(), wv.cuda(), sigma)
    rows = n_q * heads * (2 * 512 + 64) * 2 + n_q * heads * 514 * 4
    assert _scratch(c, n_q) > 4 * rows  # over formed keys and values
    out = c.prefill_mla(0, *args)
    if fmt is None:
        c_hat, kr_hat = f32(cl), f32(kr)
    else:
        st = ocache.mla_anchor_state(f32(cl), f32(kr), [T], 512, fmt[1], fmt[0])
        c_hat, kr_hat = st["c_hat"], st["kr_hat"]
    ref = oatt.mla_prefill_unabsorbed(f32(qn), f32(qp), c_hat, kr_hat, f32(wk), f32(wv), 512, [T], sigma)
    err = np.linalg.norm(f32(out).astype(np.float64) - ref) / np.linalg.norm(ref)
    assert err < 2e-5, err
    buf = torch.empty(out.numel() + 8, device="cuda")
    for off in (0, 4):
        view = buf[off:off + out.numel()].view(out.shape)
        assert view.data_ptr() % 32 == 4 * off
        assert torch.equal(c.prefill_mla(0, *args, out=view), out)
    assert c.device_error() == 0


@pytest.mark.parametrize("fmt", [None, ("grouped", 4), ("symmetric", 4)], ids=["bf16", "int4", "sym4"])
def test_mla_prefill_formed_is_no_less_exact(fmt):
    """The same chunk over formed keys and values and (in a buffer too small
    for them) by absorbed rows, against 64 bits."""
    n_q, T = 512, 700
    c, wk, wv, c_hat, kr_hat = _setup(128, fmt, [T, T], T, seed=17)
    g = torch.Generator().manual_seed(6)
    qn = torch.randn((2, n_q, H, 128), generator=g).to(torch.bfloat16)
    qp = torch.randn((2, n_q, H, 64), generator=g).to(torch.bfloat16)
    sigma = 1.0 / math.sqrt(192)
    dev = [t.cuda() for t in (qn, qp, wk, wv)]
    ref = oatt.mla_prefill_unabsorbed(f32(qn), f32(qp), c_hat, kr_hat, f32(wk), f32(wv), 128, [T, T], sigma)
    small = 2 * n_q * H * ((2 * 128 + 64) * 2 + 130 * 4)
    assert small < _scratch(c, n_q)
    rows = torch.empty((2, n_q, H, 128), device="cuda")
    buf = torch.empty(small, dtype=torch.uint8, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert c.lib.kvk_prefill_attention_mla(c.handle, 0, *map(p, dev), n_q, sigma, p(rows), p(buf), small,
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    formed = c.prefill_mla(0, *dev, sigma)
    assert not torch.equal(formed, rows)
    err = [np.linalg.norm(f32(x).astype(np.float64) - ref) / np.linalg.norm(ref) for x in (formed, rows)]
    assert err[0] <= err[1], err
    assert c.device_error() == 0


def _rows_bytes(B, n_q, width, H=H):
    return -(-B * n_q * H * (2 * width + 64) * 2 // 256) * 256 + B * n_q * H * (width + 2) * 4


@pytest.mark.parametrize("width,fmt", [(512, ("grouped", 8)), (128, ("symmetric", 4)), (512, None)],
                         ids=["g8-d512", "sym4-d128", "bf16-d512"])
def test_mla_prefill_chooses_by_the_lengths(width, fmt):
    """A short context in a large cache goes by rows, in the rows' memory, and
    no buffer is kept; the same cache grown takes the formed path where it is
    faster.  Every buffer that the size call named at one length serves at
    the others."""
    from paper_2609_37988_gb300.cache import Cache, Layer
    layer = dict(bits=16, width=width) if fmt is None else dict(bits=fmt[1], scheme=fmt[0], width=width)
    cap, n_q, first, grown = 32768, 64, 128, 8192
    c = Cache(kind="mla", n_layers=1, n_q_heads=H, head_dim=128, latent_dim=512, rope_dim=64, max_batch=1,
              max_ctx=cap, layers=[Layer(**layer)])
    g = torch.Generator().manual_seed(2)
    wk, wv = ((torch.randn((H, 128, 512), generator=g) / math.sqrt(512)).to(torch.bfloat16).cuda() for _ in range(2))
    qn = torch.randn((1, 512, H, 128), generator=g).to(torch.bfloat16).cuda()
    qp = torch.randn((1, 512, H, 64), generator=g).to(torch.bfloat16).cuda()
    c.append(0, torch.randn((1, first, 512), generator=g).to(torch.bfloat16).cuda(),
             torch.randn((1, first, 64), generator=g).to(torch.bfloat16).cuda())
    least = ctypes.c_size_t()
    assert c.lib.kvk_prefill_scratch_least(c.handle, 0, n_q, ctypes.byref(least)) == 0
    assert least.value == _rows_bytes(1, n_q, width) == _scratch(c, n_q)
    sizes = {_scratch(c, n) for n in (n_q, 512)}
    short = c.prefill_mla(0, qn[:, :n_q].contiguous(), qp[:, :n_q].contiguous(), wk, wv, 0.07)
    assert c._prefill_scratch is None
    c.append(0, torch.randn((1, grown - first, 512), generator=g).to(torch.bfloat16).cuda(),
             torch.randn((1, grown - first, 64), generator=g).to(torch.bfloat16).cuda())
    sizes |= {_scratch(c, n) for n in (n_q, 512)}
    assert max(sizes) >= 256 << 20
    ref = c.prefill_mla(0, qn, qp, wk, wv, 0.07)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    for nbytes in sizes:
        buf = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        out = torch.full_like(ref, math.nan)
        st = c.lib.kvk_prefill_attention_mla(c.handle, 0, p(qn), p(qp), p(wk), p(wv), 512, 0.07, p(out), p(buf),
                                             nbytes, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == (0 if nbytes >= min(_rows_bytes(1, 512, width), _scratch(c, 512)) else 1)
        if st == 0:
            assert_close(f32(out), f32(ref), max_abs=2e-4, rel_l2=1e-4, what=f"{nbytes} bytes")
    c.rewind(grown - first)
    again = c.prefill_mla(0, qn[:, :n_q].contiguous(), qp[:, :n_q].contiguous(), wk, wv, 0.07)
    assert torch.equal(again, short)
    assert c.device_error() == 0


def test_mla_prefill_falls_back_to_the_rows_memory(monkeypatch):
    """Where the device has no room for the formed tiles, the call runs by
    rows in the memory that they take."""
    c, wk, wv, _, _ = _setup(512, None, [900, 800], 8192, seed=9)
    n_q = 256
    g = torch.Generator().manual_seed(4)
    qn = torch.randn((2, n_q, H, 128), generator=g).to(torch.bfloat16).cuda()
    qp = torch.randn((2, n_q, H, 64), generator=g).to(torch.bfloat16).cuda()
    wk, wv = wk.cuda(), wv.cuda()
    formed = c.prefill_mla(0, qn, qp, wk, wv, 0.07)
    room, empty, asked = _rows_bytes(2, n_q, 512), torch.empty, []

    def scarce(*size, **kw):
        if kw.get("dtype") is torch.uint8:
            asked.append(size[0])
            if size[0] > room:
                raise torch.cuda.OutOfMemoryError("no room")
        return empty(*size, **kw)

    monkeypatch.setattr(torch, "empty", scarce)
    rows = c.prefill_mla(0, qn, qp, wk, wv, 0.07)
    monkeypatch.undo()
    assert asked == [_scratch(c, n_q), room]
    assert not torch.equal(rows, formed)
    assert_close(f32(rows), f32(formed), max_abs=2e-4, rel_l2=1e-4, what="rows = formed")
    assert c.device_error() == 0
