"""The GEMM tile queue (Section 4: tile queues in chunk-pipeline DAG order), decoded on the host by
the routine the device runs.  The in-order schedulers cannot deadlock only if every gemm0 tile
that a gemm1 tile waits for comes earlier in the queue; every tile must appear exactly once."""
import numpy as np
import pytest

import paper_2609_21483_b200 as pk


def replay(rows, nt0, nt1):
    rows = np.atleast_2d(np.asarray(rows, dtype=np.int32))
    q = pk.gemm_queue(rows, nt0, nt1)
    mbs = (rows + 127) // 128
    nmb = int(mbs.sum())
    assert len(q) == int(((mbs + 1) // 2).sum()) * (nt0 + nt1)
    done0 = np.zeros(nmb, np.int64)
    seen = set()
    chunk_of_mb = np.repeat(np.arange(rows.shape[0]), mbs.sum(axis=1))
    last_chunk = 0
    for ty, mb, pmb, n, chunk, nrows in q.tolist():
        gemm = ty % 3 if ty < 3 else ty - 3
        swapped = ty >= 3
        assert gemm in (0, 1) and 0 <= n < (nt0 if gemm == 0 else nt1)
        assert chunk >= last_chunk                                # chunk by chunk
        last_chunk = chunk
        blocks = [mb] if swapped else [mb, pmb]
        assert 0 < nrows <= 128
        for m in blocks:
            assert 0 <= m < nmb and chunk_of_mb[m] == chunk
            assert (gemm, m, n) not in seen
            seen.add((gemm, m, n))
            if gemm == 0:
                done0[m] += 1
            else:
                assert done0[m] == nt0, f"gemm1 tile of m-block {m} queued before its gemm0 tiles"
    # every (m-block, n-tile) of both GEMMs exactly once: a regular pair tile may cover a missing
    # second half only when the segment's m-block count is even, so the sets match exactly
    assert len(seen) == nmb * (nt0 + nt1)
    return q


SHAPES = {
    "tiny experts": lambda r, E: r.integers(0, 129, E),
    "mixed": lambda r, E: r.integers(0, 5000, E),
    "heavy tail": lambda r, E: (r.pareto(1.0, E) * 200).astype(np.int64),
    "edges": lambda r, E: r.choice([0, 1, 127, 128, 129, 255, 256, 257, 384, 2061], E),
    "mostly tiny, few huge": lambda r, E: np.where(r.random(E) < 0.9, r.integers(0, 129, E), r.integers(1000, 9000, E)),
}


@pytest.mark.parametrize("kind", list(SHAPES))
def test_dependencies_precede_and_every_tile_once(kind):
    rng = np.random.default_rng(abs(hash(kind)) % (1 << 31))
    for trial in range(40):
        E = int(rng.integers(1, 70))
        K = int(rng.choice([1, 1, 2, 4, 8]))
        rows = np.stack([SHAPES[kind](rng, E) for _ in range(K)])
        replay(rows, int(rng.integers(1, 12)), int(rng.integers(1, 9)))


def test_empty_layer_and_single_block():
    assert len(pk.gemm_queue(np.zeros((1, 5), np.int32), 3, 2)) == 0
    q = replay([[0, 7, 0]], 3, 2)
    assert (q[:, 0] >= 3).all() and len(q) == 5                   # one swapped unit: 3 gemm0 then 2 gemm1 tiles


def test_an_unpaired_block_reads_each_weight_panel_beside_its_expert():
    """One expert with five m-blocks: its last, unpaired m-block is a member of the group, so the tile
    of n-tile j comes right after the two regular pair tiles of n-tile j (same weight panel)."""
    q = replay([[128 * 5]], 3, 2)
    g0 = q[:9]
    assert list(g0[:, 0]) == [0, 0, 3] * 3 and list(g0[:, 3]) == [0, 0, 0, 1, 1, 1, 2, 2, 2]
    assert list(g0[:, 1]) == [0, 2, 4] * 3


def test_bad_arguments():
    with pytest.raises(pk.WeaveError):
        pk.gemm_queue(np.ones((3, 4), np.int32), 2, 2)            # 3 chunks
    with pytest.raises(pk.WeaveError):
        pk.gemm_queue(np.ones((8, 200), np.int32), 2, 2)          # more than 1024 segments


def check_tiles(rows, nt0, nt1, split=None):
    """The tiles themselves: each segment's rows exactly once per GEMM and n-tile, cut in units of 16 rows into as few
    tiles of at most 256 as that allows, of almost equal size; regular where they fill the 256-row MMA (more than 240),
    swapped otherwise; the ready counter that the dispatch counts a row in on is its tile's; gemm1 tiles behind
    the gemm0 tiles of their rows, in their own list."""
    rows = np.atleast_2d(np.asarray(rows, dtype=np.int32))
    EE = rows.shape[1]
    q = pk.gemm_tiles(rows, nt0, nt1, split)
    n_rt = (rows + 255) // 256
    assert len(q) == int(n_rt.sum()) * (nt0 + nt1)
    assert (np.diff(q[:, 1]) >= 0).all()                                # the first list, then the second
    seg_row0 = np.concatenate([[0], np.cumsum(rows.ravel())])
    seg_rt0 = np.concatenate([[0], np.cumsum(n_rt.ravel())])
    spans, done0, seen = {}, {}, set()
    for ty, lst, chunk, e, n, rt, row0, nr, peer, mapped in q.tolist():
        gemm, seg = ty % 3, chunk * EE + e
        assert ty in (0, 1, 3, 4) and 0 <= n < (nt0 if gemm == 0 else nt1)
        assert lst == (1 if split is not None and e >= split else 0)
        assert (ty < 3) == (nr > 240) and 0 < nr <= 256 and mapped == nr
        assert peer == (row0 + 128 if ty < 3 else row0)
        assert seg_rt0[seg] <= rt < seg_rt0[seg + 1] and (gemm, rt, n) not in seen
        seen.add((gemm, rt, n))
        assert spans.setdefault(rt, (seg, row0, nr)) == (seg, row0, nr)
        if gemm == 0:
            done0[rt] = done0.get(rt, 0) + 1
        else:
            assert done0[rt] == nt0
    assert len(spans) == n_rt.sum() and len(seen) == len(q)
    for s in range(rows.size):
        mine = [spans[rt] for rt in range(seg_rt0[s], seg_rt0[s + 1])]
        at, units = seg_row0[s], []
        for seg, row0, nr in mine:
            assert seg == s and row0 == at and (row0 - seg_row0[s]) % 16 == 0
            at += nr
            units.append((nr + 15) // 16)
        assert at == seg_row0[s + 1] and (not units or max(units) - min(units) <= 1)
    return q


def test_row_tiles_of_one_expert_of_every_size():
    for r in range(0, 1300):
        check_tiles([r], 1, 1)
    assert [t[0] for t in check_tiles([640], 1, 1)] == [3, 3, 3, 4, 4, 4]      # 224, 208, 208 rows
    assert [t[0] for t in check_tiles([497], 1, 1)] == [0, 0, 1, 1]            # 256, 241


@pytest.mark.parametrize("kind", list(SHAPES))
def test_row_tiles_of_one_list_and_of_two(kind):
    rng = np.random.default_rng(11 + list(SHAPES).index(kind))
    for trial in range(20):
        E = int(rng.integers(1, 40))
        K = int(rng.choice([1, 1, 1, 2, 4, 8]))
        rows = np.stack([SHAPES[kind](rng, E) for _ in range(K)])
        nt0, nt1 = int(rng.integers(1, 7)), int(rng.integers(1, 5))
        whole = check_tiles(rows, nt0, nt1)
        if K == 1:
            for split in {0, E, int(rng.integers(0, E + 1)), int(rng.integers(0, E + 1))}:
                two = check_tiles(rows, nt0, nt1, split)
                # the same tiles; each list in the order of the whole
                assert sorted(map(tuple, np.delete(two, 1, 1).tolist())) == sorted(map(tuple, np.delete(whole, 1, 1).tolist()))
                for lst, sel in ((0, whole[:, 3] < split), (1, whole[:, 3] >= split)):
                    np.testing.assert_array_equal(np.delete(two[two[:, 1] == lst], 1, 1), np.delete(whole[sel], 1, 1))


def test_bad_arguments_of_the_tile_list():
    for rows, split in [(np.ones((3, 4)), None), (np.ones((1, 4)), 5), (np.ones((1, 4)), -1), (np.ones((2, 4)), 2), (-np.ones((1, 4)), None)]:
        with pytest.raises(pk.WeaveError):
            pk.gemm_tiles(rows, 2, 2, split)
