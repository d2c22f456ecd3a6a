"""The tile transform's plan, walked on the host with the kernel's own integer arithmetic: the reciprocal divisions are
exact for every unit, every input and output index lies in its job's range, and both ranges lie in their buffers for every
16-byte phase.  And what a failed index check is reported as."""
import ctypes
import random

import numpy as np
import pytest

from paper_2306_14320_b200 import binding as b
from paper_2306_14320_b200 import build
from paper_2306_14320_b200 import workloads as wl


@pytest.fixture(scope="module", autouse=True)
def _test_library():
    build.build_library()
    b.use_test_library(True)
    yield
    b.use_test_library(False)


def _shapes():
    rng = random.Random(11)
    shapes = [(2, 32, 21, 25, 3, 2), (3, 5, 9, 9, 3, 1), (1, 2, 7, 1, 7, 1), (2, 3, 227, 227, 11, 4), (130, 40, 5, 3, 3, 1),
              (1, 3, 225, 225, 7, 2), (2, 3, 61, 301, 11, 3), (1, 2, 60, 1001, 3, 1), (1, 1, 11, 11, 11, 1)]
    shapes += [d[:4] + (d[5], d[7]) for d in (layer.dims() for layer in wl.CONFIGS.values())]
    for _ in range(1500):
        fh = rng.choice((1, 2, 3, 3, 4, 5, 5, 7, 7, 11))
        w = rng.choice((rng.randint(1, 40), rng.randint(1, 300), 2 * rng.randint(1, 600) + 1))
        shapes.append((rng.randint(1, 200), rng.randint(1, 300), rng.randint(fh, fh + rng.choice((3, 30, 250))), w, fh, rng.randint(1, 5)))
    return shapes


def _walk(shape, out16):
    n, c, h, w, fh, s = shape
    v = (ctypes.c_int64 * 11)()
    rc = b.lib().im2win_debug_tile_plan(ctypes.byref(b.Shape(n, c, h, w, 1, fh, 1, s)), out16, v)
    if rc != b.OK:
        assert rc == b.EUNSUPPORTED
        return None
    mb_max, nblk, pb, qw, cols, magic_qw, magic_mq, off_out, off_bar, smem, ctas = v
    ho, row_out = (h - fh) // s + 1, w * fh
    whole, planes, es, opc = nblk == 1, n * c, (2 if out16 else 4), (8 if out16 else 4)
    assert cols == 0 or (fh % 2 and fh > 1 and w % 2)
    assert qw == (w if cols else (w + 3) // 4)
    assert off_out % 128 == 0 and off_bar % 16 == 0 and smem >= off_bar + 8 and smem <= 227 * 1024
    assert ctas == (-(-planes // pb) if whole else planes * nblk)
    if whole:
        assert mb_max == ho
        jobs = {(min(pb, planes), ho), ((planes - 1) % pb + 1, ho)}
    else:
        assert pb == 1 and (nblk - 1) * mb_max < ho <= nblk * mb_max
        jobs = {(1, mb_max), (1, ho - (nblk - 1) * mb_max)}
    for npl, mb in jobs:
        rows_in = h if whole else (mb - 1) * s + fh
        assert whole or rows_in <= h
        n_in, n_out = npl * rows_in * w, npl * mb * row_out
        units_plane = mb * qw
        q = np.arange(npl * units_plane, dtype=np.uint64)
        pl = (q * np.uint64(magic_mq)) >> np.uint64(32) if npl > 1 else np.zeros_like(q)
        rem = q - pl * np.uint64(units_plane)
        mm = (rem * np.uint64(magic_qw)) >> np.uint64(32)
        k = rem - mm * np.uint64(qw)
        assert npl == 1 or int(q[-1]) * magic_mq < 2 ** 64
        assert np.array_equal(pl, q // np.uint64(units_plane)) and np.array_equal(mm, rem // np.uint64(qw))
        assert int(mm.max()) < mb and int(k.max()) < qw and int(pl.max()) < npl
        cols0 = k.astype(np.int64) * (1 if cols else 4)
        last = np.minimum(cols0 + (0 if cols else 3), w - 1)  # (the last quad of a row stops at the row's end)
        src = pl.astype(np.int64) * rows_in * w + mm.astype(np.int64) * s * w
        dst = pl.astype(np.int64) * mb * row_out + mm.astype(np.int64) * row_out
        assert int((src + cols0).min()) >= 0 and int((src + (fh - 1) * w + last).max()) < n_in
        assert int((dst + cols0 * fh).min()) >= 0 and int((dst + last * fh + fh - 1).max()) == n_out - 1
        for skew in range(4):
            assert ((skew + n_in + 3) & ~3) * 4 <= off_out
        assert off_out + (opc - 1 + n_out) * es <= off_bar
    return bool(cols)


@pytest.mark.parametrize("out16", [0, 1], ids=["fp32", "bf16"])
def test_every_index_of_the_tile_transform_stays_in_its_range(out16):
    forms = [_walk(shape, out16) for shape in _shapes()]
    assert forms.count(True) > 200 and forms.count(False) > 200


def _far_strides():
    """Strides far above the filter: one block per plane stages many rows that it does not read."""
    rng = random.Random(5)
    shapes = [(1, 2, 102, 1000, 3, 100), (1, 2, 34, 1900, 3, 32), (2, 3, 60, 700, 5, 90), (1, 1, 300, 300, 7, 299), (3, 4, 41, 90, 11, 30)]
    for _ in range(600):
        fh, s = rng.choice((1, 2, 3, 4, 5, 7, 11)), rng.randint(6, 300)
        shapes.append((rng.randint(1, 9), rng.randint(1, 30), fh + rng.randint(0, 2 * s), rng.choice((rng.randint(1, 60), rng.randint(1, 2500))), fh, s))
    return shapes


def _walk_pairs(shape):
    """The pairs kernel's plan; whether it takes the shape."""
    n, c, h, w, fh, s = shape
    v = (ctypes.c_int64 * 11)()
    rc = b.lib().im2win_debug_tile_plan(ctypes.byref(b.Shape(n, c, h, w, 1, fh, 1, s)), 2, v)
    if rc != b.OK:
        assert rc == b.EUNSUPPORTED
        return False
    mb_max, nblk, pb, qw, _, magic_qw, magic_mq, off_out, off_bar, smem, ctas = v
    ho, row_out = (h - fh) // s + 1, w * fh
    whole, planes = nblk == 1, n * c
    assert fh in (3, 5, 7, 11) and qw == w // 2 + 1
    assert off_out % 128 == 0 and off_bar % 16 == 0 and smem >= off_bar + 8 and smem <= 227 * 1024
    assert ctas == (-(-planes // pb) if whole else planes * nblk)
    if whole:
        assert mb_max == ho
        jobs = {(min(pb, planes), ho), ((planes - 1) % pb + 1, ho)}
    else:
        assert pb == 1 and (nblk - 1) * mb_max < ho <= nblk * mb_max
        jobs = {(1, mb_max), (1, ho - (nblk - 1) * mb_max)}
    for npl, mb in jobs:
        rows_in = h if whole else (mb - 1) * s + fh
        n_in, n_out = npl * rows_in * w, npl * mb * row_out
        units_plane = mb * qw
        q = np.arange(npl * units_plane, dtype=np.uint64)
        pl = (q * np.uint64(magic_mq)) >> np.uint64(32) if npl > 1 else np.zeros_like(q)
        rem = q - pl * np.uint64(units_plane)
        mm = (rem * np.uint64(magic_qw)) >> np.uint64(32)
        assert npl == 1 or int(q[-1]) * magic_mq < 2 ** 64
        assert np.array_equal(pl, q // np.uint64(units_plane)) and np.array_equal(mm, rem // np.uint64(qw))
        pl, mm, k = (a.astype(np.int64) for a in (pl, mm, rem - mm * np.uint64(qw)))
        for phase in (0, 1):  # of the job's output range; the strips' phases follow
            row = phase + pl * mb * row_out + mm * row_out
            first = 2 * k - (row & 1)
            lo, hi = np.maximum(first, 0), np.minimum(first + 1, w - 1)  # the columns it takes, none where hi < lo
            took = hi >= lo
            columns = (pl * mb + mm)[took] * w
            seen = np.concatenate([columns + lo[took], (columns + hi[took])[hi[took] > lo[took]]])
            assert np.array_equal(np.sort(seen), np.arange(npl * mb * w))  # every column of every strip once
            src = (pl * rows_in * w + mm * s * w)[took]
            assert int((src + lo[took]).min()) >= 0 and int((src + (fh - 1) * w + hi[took]).max()) < n_in
            pair = hi > lo
            assert not ((row + first * fh)[pair & took] & 1).any()  # 32-bit stores
        for skew in range(4):
            assert ((skew + n_in + 3) & ~3) * 4 <= off_out
        assert off_out + (7 + n_out) * 2 <= off_bar
    return True


def test_every_index_of_the_pairs_transform_stays_in_its_range():
    assert sum(_walk_pairs(shape) for shape in _shapes() if shape[4] in (3, 5, 7, 11)) > 500


def test_what_the_pairs_transform_declines():
    """The column form of tall filters, or the other transforms: no bf16 tile kernel but that is built for these heights."""
    columns = 0
    for shape in _shapes() + _far_strides() + [(1, 2, h, w, fh, s) for h in (30, 90, 230) for w in (130, 227, 500, 901) for fh in (5, 7, 11) for s in (1, 2)]:
        if shape[4] in (3, 5, 7, 11) and not _walk_pairs(shape):
            form = _walk(shape, 1)
            assert form is None or (form and shape[4] >= 7)
            columns += form is not None
    assert columns > 10


def test_strides_far_above_the_filter():
    """What a plan accepts fits shared memory; what it declines is another kernel's."""
    for shape in _far_strides():
        for out16 in (0, 1):
            _walk(shape, out16)
        if shape[4] in (3, 5, 7, 11):
            _walk_pairs(shape)


def test_a_failed_index_check_is_an_error():
    of = b.lib().im2win_debug_status_of_word
    assert of(0) == b.OK
    assert all(of(code) == b.ETIMEOUT for code in range(101, 110))
    assert of(201) == b.ERANGE
    assert "index check" in b.strerror(b.ERANGE)
