"""The planner's forms at the row counts where they change, cascade subgroups
at the edges of an item's 16 query vectors, the launch order taken when a call
has as many tokens as rows, the merge at the part counts where it spreads a
row over more warps, windows at the size up to which rows are not split, and
append items that end on half a block of keys (GPU, against the oracle)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import workloads as W
from _gpu import Run, assert_parity, oracle_full

pytestmark = pytest.mark.gpu


def _check(batch, **kw):
    run = Run(batch)
    run.append()
    run.forward(**kw)
    assert run.status()[0] == 0
    ref_out, ref_lse, _ = oracle_full(batch)
    assert_parity(*run.out_host(), ref_out, ref_lse, batch.name)
    return run.header()


@pytest.mark.parametrize("B", [2, 7, 8, 9, 255, 256, 257, 512, 513, 1024, 1025])
def test_row_counts_where_the_planner_changes(B):
    # groups of 40 rows (across warps and, above 1024 rows, threads' row pairs)
    # sharing 5 or 6 pages, some rows empty or appending
    rng = np.random.default_rng(B)
    grp = np.arange(B) // 40
    prompt = rng.integers(80, 110, size=B)[grp]
    L = rng.choice([0, 1, 1, 1, 1, 1, 1, 9], size=B)
    S = prompt + rng.integers(0, 50, size=B) + L
    b = W.build_batch(f"rows{B}", B, S, L, 8, 1, shared_prefix_pages=prompt // 16, prompt_lens=prompt,
                      group_of_row=grp)
    hdr = _check(b)
    assert hdr["n_cascade"] >= B // 40 and hdr["n_append"] == int((L > 1).sum())


@pytest.mark.parametrize("size", [2, 3, 17])
@pytest.mark.parametrize("g", [1, 2, 4, 8])
def test_cascade_subgroups(g, size):
    rng = np.random.default_rng(10 * g + size)
    B = 2 * size
    grp = np.arange(B) // size
    prompt = np.array([70, 333])[grp]
    S = prompt + rng.integers(1, 60, size=B)
    b = W.build_batch(f"sub{g}_{size}", 10 * g + size, S, np.ones(B, np.int64), 2 * g, 2,
                      shared_prefix_pages=prompt // 16, prompt_lens=prompt, group_of_row=grp)
    assert _check(b)["n_cascade"] >= 2 * -(-size * g // 16)


@pytest.mark.parametrize("heads,size,prompt", [(64, 24, 4000), (64, 25, 4010), (64, 47, 2100), (32, 45, 4100),
                                               (16, 67, 5700), (8, 177, 4040)])
def test_wide_cascade_items(heads, size, prompt):
    # decode steps with enough shared pages take cascade items of 32 query vectors
    # (full and partial ones), the same with phase events or on one stream; a group
    # of two rows and a row of no group beside
    from paper_2608_22167_gb300 import mcpu

    rng = np.random.default_rng(size)
    g, grp = heads // 8, np.r_[np.zeros(size, int), np.ones(size, int), 2, 2, -1]
    pr = np.r_[np.full(size, prompt), np.full(size, prompt + 64), 100, 100, 0]
    S = pr + rng.integers(1, 60, size=2 * size + 3)
    b = W.build_batch(f"wide{heads}_{size}", size, S, np.ones(S.size, np.int64), heads, 8, shared_prefix_pages=pr // 16,
                      prompt_lens=pr, group_of_row=grp)
    run = Run(b)
    run.append()
    run.forward()
    assert run.status()[0] == 0
    assert int(run.ws[40:44].view(torch.int32)) == 1  # header: wide items
    C, subs = run.header()["split_pages"], -(-size // (32 // g))
    splits = [-(-(p // 16) // C) for p in (prompt, prompt + 64, 100)]
    assert run.header()["n_cascade"] == subs * (splits[0] + splits[1]) + splits[2]
    one = run.out_host()
    ref_out, ref_lse, _ = oracle_full(b)
    assert_parity(*one, ref_out, ref_lse, b.name)
    for kw in (dict(flags=mcpu.FLAG_SERIAL), "events"):
        run.out.fill_(float("nan"))
        if kw == "events":
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(mcpu.NUM_PHASE_EVENTS)]
            for e in ev:  # torch creates the CUDA event at its first record
                e.record()
            mcpu.mcpu_paged_attention_forward(run.q, run.kc, run.vc, run.bt, run.sl, run.qsl, 0, b.softmax_scale,
                                              run.out, run.lse, run.ws, phase_events=ev)
        else:
            run.forward(**kw)
        for x, y in zip(one, run.out_host()):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("extra", [-1, 0, 1])
@pytest.mark.parametrize("window", [0, 100])
@pytest.mark.parametrize("n_app", [0, 1, 5])
def test_as_many_tokens_as_rows_or_one_more_or_less(n_app, window, extra):
    # append rows beside empty ones: with as many tokens as rows the kernels go
    # in one chain, else in the fork; both equal the serial order
    from paper_2608_22167_gb300 import mcpu

    rng = np.random.default_rng(100 * n_app + window + extra + 1)
    B = 48
    L = np.ones(B, np.int64)
    L[2:2 + n_app] = 7
    L[-6 * n_app:] = 0 if n_app else 1
    L[1] += extra
    grp = np.where(np.arange(B) < 24, np.arange(B) // 8, -1)
    prompt = np.where(grp >= 0, 700, 0)
    S = prompt + rng.integers(8, 900, size=B)
    b = W.build_batch(f"chain{n_app}", 7, S, L, 16, 4, layer_windows=(window,), shared_prefix_pages=prompt // 16,
                      prompt_lens=prompt, group_of_row=grp)
    assert b.total_q == B + extra
    hdr = _check(b)
    assert hdr["n_append"] == int((L > 1).sum()) and (hdr["n_cascade"] > 0) == (window == 0)
    run = Run(b)
    run.append()
    run.forward()
    one = run.out_host()
    run.out.fill_(float("nan"))
    run.forward(flags=mcpu.FLAG_SERIAL)
    for x, y in zip(one, run.out_host()):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("B,heads", [(1, 8), (5, 32), (40, 64)])
@pytest.mark.parametrize("parts", [8, 9, 16, 17, 33, 70])
def test_merge_of_few_rows_with_many_parts(B, heads, parts):
    S = np.full(B, parts * 32) - np.arange(B) % 20
    b = W.build_batch(f"merge{B}_{parts}", parts, S, np.ones(B, np.int64), heads, heads // 4)
    assert _check(b, split_pages=2)["n_merge"] == B


@pytest.mark.parametrize("window", [1, 17, 127, 128, 129])
def test_windows_that_are_not_split(window):
    # every alignment of a window's first and last page, rows shorter than the
    # window, append rows beside them; a forced split still splits
    S = np.concatenate([np.arange(1, 20), np.arange(300, 333), [40, 500]])
    L = np.concatenate([np.ones(52, np.int64), [30, 200]])
    b = W.build_batch(f"win{window}", window, S, L, 16, 4, layer_windows=(window,))
    hdr = _check(b)
    assert hdr["n_merge"] == 0 if window <= 128 else hdr["n_merge"] > 0
    assert (_check(b, split_pages=1)["n_merge"] > 0) == (window > 1)


@pytest.mark.parametrize("g", [1, 8])
@pytest.mark.parametrize("window", [1, 33, 64, 65, 128, 1024, 1025])
def test_append_items_that_end_on_half_a_block(window, g):
    # items whose last block holds 1 .. 128 keys (steps of 21 with every page
    # remainder), for windows up to and beyond the short form's limit
    L = np.array([2, 5, 31, 32, 33, 64, 65, 200] * 8)
    S = np.maximum(L, 20 + 21 * np.arange(64)) + np.arange(64) % 16
    b = W.build_batch(f"half{window}_{g}", window, S, L, 2 * g, 2, layer_windows=(window,))
    assert _check(b)["n_append"] > 0
