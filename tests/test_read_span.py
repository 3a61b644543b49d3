"""Memory safety of the bulk-copy kernels' reads, checked on the host.

The kernels fetch 16-byte-aligned ranges although rows may start at any element; the library's
read-span hooks replay the kernels' own address arithmetic (one header shared by both) for a
matrix at any address.  For every shape and misalignment below: no tile / row part breaks a rule
(faults == 0) and the union of all reads is exactly the matrix's own extent -- nothing before its
first logit, nothing past its last one, nothing left out at the ends."""
import itertools

import pytest

from paper_2603_11243_b200 import binding as ssd

BASE = 0x7F0000000000          # any 16-byte-aligned address; nothing is dereferenced


def _extent(rows, ld, V, es):
    return ((rows - 1) * ld + V) * es


VS = (1, 2, 3, 5, 7, 8, 9, 15, 16, 17, 31, 33, 129, 348, 1025, 4097)
NS = tuple(range(1, 41)) + (63, 64, 65, 100, 1000, 4095, 4096, 4097, 4099, 8191, 8192, 8193,
                            12289, 14674)


@pytest.mark.parametrize("dtype,es", [(ssd.F32, 4), (ssd.BF16, 2)])
def test_ctc_reads_stay_inside_the_matrix(dtype, es):
    checked_bulk = 0
    for V in VS:
        for pad in (0, 1, 3, 8):
            ld = V + pad
            for N in NS:
                for mis in range(0, 16, es) if N < 50 else (0, es, 16 - es):
                    base = BASE + mis
                    r = ssd.ssd_ctc_draft_read_span(base, dtype, V, ld, N)
                    assert r.faults == 0, (V, ld, N, mis)
                    assert r.lo == base and r.hi == base + _extent(N, ld, V, es), (V, ld, N, mis)
                    checked_bulk += r.kernel == 2
    assert checked_bulk > 1000          # the sweep really exercised the bulk-copy kernel


def test_ctc_reads_with_forced_shapes():
    # small stages, many warps, the shapes the launch options can force
    for V, N in itertools.product((1, 3, 129, 1025), (1, 5, 33, 1000, 4097)):
        for stage_bytes, stages, warps in ((1, 1, 1), (1, 8, 24), (64, 2, 3), (100000, 1, 24)):
            o = ssd.LaunchOpts()
            o.stage_bytes, o.stages, o.warps = stage_bytes, stages, warps
            for mis in (0, 2, 6, 14):
                try:
                    r = ssd.ssd_ctc_draft_read_span(BASE + mis, ssd.BF16, V, V + 1, N, o)
                except ssd.SsdError:
                    continue                       # a shape the library refuses
                assert r.faults == 0 and r.lo == BASE + mis
                assert r.hi == BASE + mis + _extent(N, V + 1, V, 2)


def test_ctc_reads_of_the_kernel_that_runs():
    """Tiles, which short rows only take where they are asked for, rows read into registers, and rows that
    are longer than either takes: 2 GB and more for a row's own bytes."""
    tiles = ssd.LaunchOpts()
    tiles.kernel = 2
    reached = {0: 0, 1: 0}
    for V, pad, N in itertools.product(VS, (0, 1, 3, 8), (1, 2, 33, 1000, 4097)):
        for dtype, es in ((ssd.F32, 4), (ssd.BF16, 2)):
            for mis, o in itertools.product((0, es, 16 - es), (None, tiles)):
                r = ssd.ssd_ctc_draft_read_span(BASE + mis, dtype, V, V + pad, N, o)
                assert r.faults == 0 and r.kernel == 2 and not (o and r.direct), (V, pad, N, mis)
                assert r.lo == BASE + mis and r.hi == BASE + mis + _extent(N, V + pad, V, es), (V, pad, N, mis)
                reached[r.direct] += 1
    assert min(reached.values()) > 1000
    # a matrix so much wider than its rows that no tile would hold them: still registers
    r = ssd.ssd_ctc_draft_read_span(BASE + 2, ssd.BF16, 348, 2000, 500)
    assert (r.faults, r.kernel, r.direct, r.hi) == (0, 2, 1, BASE + 2 + _extent(500, 2000, 348, 2))
    for V in ((1 << 29) - 1, 1 << 29, (1 << 29) + 5, (1 << 31) - 1):
        r = ssd.ssd_ctc_draft_read_span(BASE + 4, ssd.F32, V, V, 3)
        assert (r.faults, r.kernel, r.direct) == (0, 1, 0), V
        assert r.lo == BASE + 4 and r.hi == BASE + 4 + _extent(3, V, V, 4), V


@pytest.mark.parametrize("dtype,es", [(ssd.F32, 4), (ssd.BF16, 2)])
def test_verify_reads_stay_inside_each_row(dtype, es):
    checked_bulk = 0
    for V in (1, 2, 7, 8, 9, 33, 1000, 4097, 32000, 49152, 49153, 100352, 152064, 152065):
        for pad in (0, 1, 5):
            ld = V + pad
            for M in (1, 2, 3, 17, 148, 149, 1200):
                if V > 50000 and M > 149:
                    continue
                for mis in range(0, 16, es) if M < 20 else (0, es):
                    base = BASE + mis
                    r = ssd.ssd_verify_read_span(base, dtype, V, ld, M, B=3)
                    assert r.faults == 0, (V, ld, M, mis)
                    assert r.lo == base and r.hi == base + _extent(M, ld, V, es), (V, ld, M, mis)
                    checked_bulk += r.kernel == 2
    assert checked_bulk > 300


@pytest.mark.parametrize("dtype,es", [(ssd.F32, 4), (ssd.BF16, 2)])
def test_verify_reads_of_the_kernel_by_choice_and_of_the_ring(dtype, es):
    """The same shapes as the library's own choice and with the ring forced, which the early-exit kernel
    shares its arithmetic with: most bf16 shapes go to direct loads by themselves."""
    ring = ssd.LaunchOpts()
    ring.kernel = 2
    reached = {"ring": 0, "direct": 0}
    for V in (1, 2, 7, 8, 9, 33, 1000, 4097, 32000, 49152, 49153, 100352, 152065):
        for pad, M in itertools.product((0, 1, 5), (1, 3, 149, 1200)):
            if V > 50000 and M > 149:
                continue
            for mis in range(0, 16, es) if M < 20 else (0, es):
                for o in (None, ring):
                    r = ssd.ssd_verify_read_span(BASE + mis, dtype, V, V + pad, M, B=3, opts=o)
                    assert r.faults == 0 and r.kernel == 2, (V, pad, M, mis)
                    assert r.lo == BASE + mis and r.hi == BASE + mis + _extent(M, V + pad, V, es), (V, pad, M, mis)
                    assert not (o and r.direct)
                    reached["direct" if r.direct else "ring"] += 1
    assert reached["ring"] > 400
    assert reached["direct"] > 400 if dtype == ssd.BF16 else reached["direct"] == 0


def test_verify_reads_with_forced_shapes():
    for V, M in itertools.product((7, 1025, 49153), (1, 5, 300)):
        for split, stage_bytes, warps in ((1, 1024, 4), (3, 4096, 16), (7, 1024, 8), (64, 2048, 12),
                                          (2, 65536, 16)):
            o = ssd.LaunchOpts()
            o.split, o.stage_bytes, o.warps = split, stage_bytes, warps
            for mis in (0, 2, 10):
                r = ssd.ssd_verify_read_span(BASE + mis, ssd.BF16, V, V + 3, M, 2, o)
                assert r.faults == 0 and r.lo == BASE + mis
                assert r.hi == BASE + mis + _extent(M, V + 3, V, 2)


def test_verify_reads_of_a_large_batch():
    """More rows than the direct-load kernel has warps: the finer cuts that it may take when some are
    skipped are replayed as well."""
    for V, pad, mis in itertools.product((1, 700, 4099, 8192), (0, 3), (0, 2, 18)):
        r = ssd.ssd_verify_read_span(BASE + mis, ssd.BF16, V, V + pad, 5000, B=40)
        assert r.faults == 0 and r.lo == BASE + mis, (V, pad, mis)
        assert r.hi == BASE + mis + _extent(5000, V + pad, V, 2), (V, pad, mis)


def test_read_span_argument_errors():
    with pytest.raises(ssd.SsdError):
        ssd.ssd_ctc_draft_read_span(BASE + 1, ssd.BF16, 8, 8, 4)        # off the element size
    with pytest.raises(ssd.SsdError):
        ssd.ssd_verify_read_span(BASE, ssd.F32, 8, 7, 4)                # ld < V
    with pytest.raises(ssd.SsdError):
        ssd.ssd_ctc_draft_read_span(BASE, 7, 8, 8, 4)                   # bad dtype
    r = ssd.ssd_ctc_draft_read_span(BASE, ssd.F32, 8, 8, 0)             # nothing to read
    assert r.faults == 0 and r.lo == r.hi == BASE
