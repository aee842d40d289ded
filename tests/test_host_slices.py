"""Host planning of the preconditioner's sparse slices (no GPU): read as the row
kernel reads them - a slice's rounds of 32 (or 256) consecutive entries, entry j
of a row on lane j mod lanes - they give back every entry of every row once, in
order, for empty matrices and rows, rows at the lane and CTA thresholds and each
of the three numbers of rounds."""
import numpy as np
import pytest

FULL = 152 * 2048   # threads resident on the GPU


def _read(plan, rows):
    """{row: [(column, value), ...]} from a plan."""
    n_cta, hdr, slot_row, idx, val = plan
    out, slots = {}, 0
    last = None
    for s, (first, rounds, lanes, slot) in enumerate(hdr.tolist()):
        wide = s < n_cta
        width = 256 if wide else 32
        assert (lanes == 256) == wide and slot == slots
        if not wide:
            assert lanes in (1, 2, 4, 8, 16, 32)
            key = (rounds, lanes)
            assert last is None or key <= last          # longest first
            last = key
        n_rows = width // lanes
        e = np.arange(32 * first, 32 * first + rounds * width).reshape(rounds, n_rows, lanes)
        for r in range(n_rows):
            row = int(slot_row[slot + r])
            at = e[:, r, :].ravel()
            if row < 0:
                assert (idx[at] == -1).all() and (val[at] == 0).all()
                continue
            assert row not in out
            used = idx[at] >= 0
            assert not used.any() or used[:used.sum()].all()   # entries first, padding after them
            out[row] = list(zip(idx[at][used].tolist(), val[at][used].tolist()))
        slots += n_rows
    assert slots == len(slot_row) and sorted(out) == list(range(rows))
    return out


def _check(B, lens):
    ptr = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    plan = B.plan_slices(ptr)
    got = _read(plan, len(lens))
    for i, n in enumerate(lens):
        want = [(j % 1000, float(j)) for j in range(ptr[i], ptr[i] + n)]
        assert got[i] == want, i
    return plan


def test_empty(built_lib):
    assert len(_check(built_lib, [])[1]) == 0
    n_cta, hdr, *_ = _check(built_lib, [0] * 40)
    assert n_cta == 0 and (hdr[:, 1] == 0).all()


@pytest.mark.parametrize("rounds", [4, 8, 16])
def test_rows_at_every_threshold(built_lib, rounds):
    """Rows around each width, and short ones enough for the matrix to take so
    many rounds: half the GPU's threads a lane at 16, at 8 but not 16, at
    neither.  Rows of more than 128 rounds' entries or 1024 take a CTA."""
    edge = [0, 1, 2, 3]
    for lanes in (1, 2, 4, 8, 16, 32):
        edge += [lanes * rounds - 1, lanes * rounds, lanes * rounds + 1]
    wide = min(1024, 128 * rounds)
    edge += [wide - 1, wide, wide + 1, wide + 256, 3000]
    rng = np.random.default_rng(rounds)
    more = {4: 0, 8: FULL // 4, 16: FULL // 2}[rounds]   # rows of 16: one lane, or two at 8 rounds
    lens = np.array(edge * 2 + [16] * more)
    rng.shuffle(lens)
    n_cta, hdr, slot_row, _, _ = _check(built_lib, lens.tolist())
    assert n_cta == int((lens > wide).sum())
    assert np.array_equal(lens[slot_row[:n_cta]], np.sort(lens[lens > wide])[::-1])
    narrow = hdr[n_cta:]
    # the widest row of one lane tells the rounds
    assert narrow[narrow[:, 2] == 1, 1].max() == rounds


def test_filled_on_several_threads(built_lib):
    """Large enough for the entries to be written in parts, long rows among them."""
    rng = np.random.default_rng(3)
    lens = np.concatenate([rng.integers(0, 60, 20000), rng.integers(1025, 9000, 12)])
    rng.shuffle(lens)
    plan = _check(built_lib, lens.tolist())
    assert len(plan[3]) >= 4 << 17


@pytest.mark.parametrize("seed", [0, 1])
def test_random_rows(built_lib, seed):
    rng = np.random.default_rng(seed)
    lens = np.concatenate([rng.integers(0, 12, 2000), rng.integers(0, 300, 200), rng.integers(900, 2500, 9)])
    rng.shuffle(lens)
    _check(built_lib, lens.tolist())
