"""The outer round on host-resident state (aloco_sync_host): theta, v and the
replicas in page-locked host memory, streamed through the GPU in chunks.
Per-element results must equal the device round's bit for bit.  The
statistics agree within the statistics tolerance: chunking changes which
elements share a thread's fp32 partial sum before it is added in fp64."""
import pytest
import torch

import oracle as O
from paper_2609_36662_gb300 import aloco as A
from paper_2609_36662_gb300 import workloads as W
from _parity import RTOL_STAT, assert_field, gpu_inputs, schedule_pair

pytestmark = pytest.mark.gpu


def _pinned(t):
    return t.detach().cpu().pin_memory()


def _bits(t):
    return t.view(torch.int16) if t.dtype == torch.bfloat16 else t.view(torch.int32)


def _rounds(w, chunk, stream=None):
    g, v, xs = gpu_inputs(w)
    v.normal_(0, 1e-3, generator=torch.Generator("cuda").manual_seed(w.M))
    gh, vh, xh = _pinned(g), _pinned(v), [_pinned(x) for x in xs]
    x_before = [x.clone() for x in xh]
    sa, _ = schedule_pair(w.schedule)
    kw = dict(H_sel=w.H_sel[0], H_base=w.H_base, step=w.start_step, schedule=sa,
              outer_lr=w.outer_lr, outer_beta=w.outer_beta)
    st_d = A.sync(g, v, xs, **kw)
    st_h = A.sync_host(gh, vh, xh, chunk_elems=chunk, stream=stream, **kw)
    return g, v, xs, gh, vh, xh, x_before, st_d, st_h


@pytest.mark.parametrize("dt,M,N,chunk", [
    ("f32", 1, 1000, 0),                 # one chunk shorter than a pack row
    ("f32", 3, 1_000_003, 65_536),       # many chunks, ragged tail
    ("bf16", 8, 1_000_003, 100_000),
    ("bf16", 5, 300_001, 8),             # the smallest chunk: 37,501 chunks
    ("f32", 8, 4_194_309, 0),            # default chunk, one chunk
    ("bf16", 16, 2_000_000, 1 << 20),
    ("f32", 32, 50_000, 4096),
    ("f32", 4, 40_000_001, 0),           # default chunk, three chunks
])
def test_host_round_equals_device_round(dt, M, N, chunk):
    w = W.small(N, M, dt, seed=60 + M)
    g, v, xs, gh, vh, xh, x_before, st_d, st_h = _rounds(w, chunk)
    assert st_h["status"] == A.OK
    assert torch.equal(_bits(gh), _bits(g.cpu()))
    assert torch.equal(_bits(vh), _bits(v.cpu()))
    for a, b in zip(xh, x_before):          # host replicas are inputs only
        assert torch.equal(_bits(a), _bits(b))
    for key in ("D", "C", "mean_sq_norm"):
        assert st_h[key] == pytest.approx(st_d[key], rel=RTOL_STAT), key
    for a, b in zip(st_h["drift"][:M], st_d["drift"][:M]):
        assert a == pytest.approx(b, rel=RTOL_STAT)
    assert st_h["nonfinite"] == st_d["nonfinite"] == 0
    assert st_h["corr"] == st_d["corr"]


def test_host_round_matches_the_oracle():
    w = W.small(777_777, 4, "f32", seed=3)
    g, v, xs = gpu_inputs(w)
    gh, vh, xh = _pinned(g), _pinned(v), [_pinned(x) for x in xs]
    sa, so = schedule_pair(w.schedule)
    orc = O.sync_round(gh.numpy(), vh.numpy(), [x.numpy() for x in xh], O.F32,
                       so, w.start_step, w.H_sel[0], w.H_base,
                       w.outer_lr, w.outer_beta)
    st = A.sync_host(gh, vh, xh, H_sel=w.H_sel[0], H_base=w.H_base,
                     step=w.start_step, schedule=sa, outer_lr=w.outer_lr,
                     outer_beta=w.outer_beta, chunk_elems=100_000)
    assert_field(gh.numpy(), orc["g"], "theta'")
    assert_field(vh.numpy(), orc["v"], "v'")
    for key in ("D", "C"):
        assert st[key] == pytest.approx(orc[key], rel=RTOL_STAT)


def test_side_stream_and_nonfinite_counts():
    w = W.small(500_000, 3, "bf16", seed=8)
    g, v, xs = gpu_inputs(w)
    xs[1][12345] = float("nan")
    xs[2][499_999] = float("inf")
    gh, vh, xh = _pinned(g), _pinned(v), [_pinned(x) for x in xs]
    sa, _ = schedule_pair(w.schedule)
    kw = dict(H_sel=w.H_sel[0], H_base=w.H_base, step=w.start_step, schedule=sa,
              outer_lr=w.outer_lr, outer_beta=w.outer_beta)
    st_d = A.sync(g, v, xs, **kw)
    s = torch.cuda.Stream()
    st_h = A.sync_host(gh, vh, xh, chunk_elems=65_536, stream=s,
                       opts=A.default_opts(time_kernel=1), **kw)
    assert st_d["status"] == st_h["status"] == A.ERR_NONFINITE
    assert st_h["nonfinite"] == st_d["nonfinite"] == 2
    assert st_h["kernel_ms"] > 0
    assert torch.equal(_bits(gh), _bits(g.cpu()))


def test_pageable_memory_and_bulk_copy_are_rejected():
    w = W.small(10_000, 2, "f32", seed=1)
    g, v, xs = gpu_inputs(w)
    sa, _ = schedule_pair(w.schedule)
    kw = dict(H_sel=w.H_sel[0], H_base=w.H_base, step=w.start_step, schedule=sa,
              outer_lr=w.outer_lr, outer_beta=w.outer_beta)
    pageable = g.cpu()
    with pytest.raises(A.AlocoError) as ei:
        A.sync_host(pageable, _pinned(v), [_pinned(x) for x in xs], **kw)
    assert ei.value.status == A.ERR_ARG and "page-locked" in str(ei.value)
    with pytest.raises(A.AlocoError) as ei:                  # device memory
        A.sync_host(g, v, xs, **kw)
    assert ei.value.status == A.ERR_ARG
    with pytest.raises(A.AlocoError) as ei:
        A.sync_host(_pinned(g), _pinned(v), [_pinned(x) for x in xs],
                    opts=A.default_opts(pass_=A.PASS_BULK_COPY), **kw)
    assert ei.value.status == A.ERR_ARG


@pytest.mark.parametrize("chunk", [0, 4096])
@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("off,off_v", [(0, 0), (3, 3), (5, 5), (3, 2)])
def test_host_round_on_views(off, off_v, dt, chunk):
    """Views of page-locked vectors: cut at one element (read and written in
    place, behind a head of elements) or at two (staged), the round equals the
    device round bit for bit and touches nothing outside the views."""
    N, M = 70_003, 3
    w = W.small(N, M, dt, seed=9)
    g, v, xs = gpu_inputs(w)
    v.normal_(0, 1e-3, generator=torch.Generator("cuda").manual_seed(2))

    def view(t, k):
        whole = torch.full((N + 16,), 3.5, dtype=t.dtype).pin_memory()
        whole[k:k + N] = t.cpu()
        return whole, whole[k:k + N]
    pairs = [view(g, off), view(v, off_v)] + [view(x, off) for x in xs]
    x_before = [p[0].clone() for p in pairs[2:]]
    sa, _ = schedule_pair(w.schedule)
    kw = dict(H_sel=w.H_sel[0], H_base=w.H_base, step=w.start_step, schedule=sa,
              outer_lr=w.outer_lr, outer_beta=w.outer_beta)
    st_d = A.sync(g, v, xs, **kw)
    st_h = A.sync_host(pairs[0][1], pairs[1][1], [p[1] for p in pairs[2:]],
                       chunk_elems=chunk, **kw)
    assert st_d["status"] == st_h["status"] == A.OK
    for (whole, part), want, k in zip(pairs[:2], (g, v), (off, off_v)):
        assert torch.equal(_bits(part), _bits(want.cpu()))
        assert bool((whole[:k] == 3.5).all()) and bool((whole[k + N:] == 3.5).all())
    for (whole, _), before in zip(pairs[2:], x_before):
        assert torch.equal(_bits(whole), _bits(before))
    assert st_h["D"] == pytest.approx(st_d["D"], rel=RTOL_STAT)
    assert st_h["C"] == pytest.approx(st_d["C"], rel=RTOL_STAT)


def _on_pages(t, pages):
    """A copy of the CPU vector t that starts on a 64 KB page of ordinary
    memory, `pages` of them, and the address of the first."""
    whole = torch.full(((pages + 1) * 65536 // t.element_size(),), 3.5, dtype=t.dtype)
    skip = (-whole.data_ptr() % 65536) // t.element_size()
    part = whole[skip:skip + t.numel()]
    part.copy_(t)
    return whole, part


@pytest.mark.parametrize("chunk", [0, 4096])
@pytest.mark.parametrize("short", [0, 1, 3])
def test_memory_locked_in_part_is_rejected(short, chunk):
    """A buffer (theta, v, a replica) whose page-locked range ends before the
    vector does is refused before anything is launched or written."""
    w = W.small(40_000, 3, "f32", seed=2)   # 160,000 bytes: 2.4 pages of 64 KB
    g, v, xs = gpu_inputs(w)
    bufs = [_pinned(t) for t in (g, v, *xs)]
    whole, part = _on_pages(bufs[short], 3)
    cudart = torch.cuda.cudart()
    assert int(cudart.cudaHostRegister(part.data_ptr(), 65536, 0)) == 0
    try:
        bufs[short] = part
        before = [b.clone() for b in bufs]
        sa, _ = schedule_pair(w.schedule)
        with pytest.raises(A.AlocoError) as ei:
            A.sync_host(bufs[0], bufs[1], bufs[2:], H_sel=w.H_sel[0], H_base=w.H_base,
                        step=w.start_step, schedule=sa, outer_lr=w.outer_lr,
                        outer_beta=w.outer_beta, chunk_elems=chunk)
        assert ei.value.status == A.ERR_ARG and "page-locked" in str(ei.value)
        assert all(torch.equal(b, c) for b, c in zip(bufs, before))
    finally:
        assert int(cudart.cudaHostUnregister(part.data_ptr())) == 0


def test_memory_locked_in_pieces_is_staged():
    """Buffers page-locked in pieces, with chunks that end where the pieces do:
    copied piece by piece."""
    N = 3 * 16384
    w = W.small(N, 2, "f32", seed=2)
    g, v, xs = gpu_inputs(w)
    v.normal_(0, 1e-3, generator=torch.Generator("cuda").manual_seed(2))
    pages = [_on_pages(t.cpu(), 3) for t in (g, v, *xs)]
    cudart = torch.cuda.cudart()
    pieces = [part.data_ptr() + 65536 * k for _, part in pages for k in range(3)]
    locked = []
    try:
        for p in pieces:
            assert int(cudart.cudaHostRegister(p, 65536, 0)) == 0
            locked.append(p)
        sa, _ = schedule_pair(w.schedule)
        kw = dict(H_sel=w.H_sel[0], H_base=w.H_base, step=w.start_step, schedule=sa,
                  outer_lr=w.outer_lr, outer_beta=w.outer_beta)
        A.sync(g, v, xs, **kw)
        st = A.sync_host(pages[0][1], pages[1][1], [p for _, p in pages[2:]],
                         chunk_elems=16384, **kw)
        assert st["status"] == A.OK and st["grid"] == 3   # chunks
        assert torch.equal(_bits(pages[0][1]), _bits(g.cpu()))
        assert torch.equal(_bits(pages[1][1]), _bits(v.cpu()))
    finally:
        for p in locked:
            assert int(cudart.cudaHostUnregister(p)) == 0


@pytest.mark.parametrize("dt,M", [("f32", 1), ("f32", 8), ("bf16", 1), ("bf16", 32)])
def test_host_round_leaves_most_sms_to_other_streams(dt, M):
    """The round without staging runs on less than half of the SMs unless the
    caller asks for blocks on every one; the results do not depend on it."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = W.small(1_000_003, M, dt, seed=12)
    g, v, xs = gpu_inputs(w)
    sa, _ = schedule_pair(w.schedule)
    kw = dict(H_sel=w.H_sel[0], H_base=w.H_base, step=w.start_step, schedule=sa,
              outer_lr=w.outer_lr, outer_beta=w.outer_beta)
    outs = []
    for opts in (A.default_opts(), A.default_opts(blocks_per_sm=1)):
        gh, vh, xh = _pinned(g), _pinned(v), [_pinned(x) for x in xs]
        outs.append((A.sync_host(gh, vh, xh, opts=opts, **kw), gh, vh))
    (a, ga, va), (b, gb, vb) = outs
    assert a["grid"] < sms / 2 and b["grid"] == sms
    assert torch.equal(ga, gb) and torch.equal(va, vb)
    assert a["D"] == pytest.approx(b["D"], rel=RTOL_STAT)
