"""GPU parity of batched layers (ara_run_layers: several layers in one pass
over the YET) against the FP64 oracle run layer by layer, and against the
single-layer path.  Same tolerances as the single-layer parity tests: each
year loss within 1e-5 of max(|Y|, gross loss) of its layer's oracle run.
"""

import numpy as np
import pytest

import oracle
from paper_1501_06326_gb300 import synth

pytestmark = pytest.mark.gpu

YLT_TOL = 1e-5


@pytest.fixture(scope="module")
def eng():
    import __graft_entry__

    __graft_entry__.build()
    from paper_1501_06326_gb300 import ara

    e = ara.Ara(0)
    yield e
    e.close()


def check_ylt(ylt, ref, tol=YLT_TOL):
    scale = np.maximum(np.abs(ref["ylt"]), ref["gross"])
    err = np.abs(ylt - ref["ylt"])
    bad = err > tol * scale
    worst = float(np.max(err / np.where(scale > 0, scale, 1.0))) if err.size else 0.0
    assert not bad.any(), f"{bad.sum()} trials out of tolerance, worst {worst:.3e}"
    return worst


def _batch_case(n_trials, catalogue, mean_events, n_elts, entries, n_layers, max_elts, seed, recipe="plain"):
    yet = synth.make_yet(n_trials, mean_events, catalogue, seed)
    pool = synth.make_elt_pool(n_elts, entries, catalogue, seed + 1, recipe=recipe)
    layer_ids = synth.draw_layers(n_layers, pool.elt_ids, max_elts, seed + 2)
    layers = []
    for ids in layer_ids:
        sub = pool.subset([int(np.flatnonzero(pool.elt_ids == i)[0]) for i in ids])
        layers.append((ids, oracle.calibrate_layer_terms(yet, sub), sub))
    return yet, pool, layers


def _run_batch(eng, yet, pool, layers, seed, t0=0, t1=None, index=False, **kw):
    t1 = yet.n_trials if t1 is None else t1
    eng.load_yet(yet.offsets, yet.event_ids, yet.catalogue_size)
    if index:
        eng.build_yet_index()
    eng.load_pool(pool)
    out = np.zeros((len(layers), t1 - t0))
    eng.run_layers([(ids, terms) for ids, terms, _ in layers], seed, t0, t1, out, **kw)
    return out


@pytest.fixture(scope="module")
def small_batch():
    # 1,000 trials x Poisson(100) over a catalogue of 10,000; a pool of 12 ELTs x 1,000
    # records; 6 layers of 1..8 ELTs (overlapping), terms per layer
    return _batch_case(1000, 10_000, 100.0, 12, 1000, 6, 8, 4242)


def test_batch_matches_oracle_layer_by_layer(eng, small_batch):
    yet, pool, layers = small_batch
    for seed in (0, 77):
        out = _run_batch(eng, yet, pool, layers, seed)
        for l, (ids, terms, sub) in enumerate(layers):
            ref = oracle.run_layer(yet, sub, terms, seed=seed)
            check_ylt(out[l], ref)


def test_batch_matches_the_single_layer_path(eng, small_batch):
    # the two paths differ only in the FP32 rounding of multi-ELT event sums and in
    # how a trial's sum is carried, so they agree well inside the oracle tolerance
    # (scaled, as there, by the trial's gross loss: terms are 1-Lipschitz)
    yet, pool, layers = small_batch
    out = _run_batch(eng, yet, pool, layers, 5)
    for l, (ids, terms, sub) in enumerate(layers):
        single = np.zeros(yet.n_trials)
        eng.run_layer(ids, terms, 5, 0, yet.n_trials, single)
        gross = oracle.run_layer(yet, sub, terms, seed=5)["gross"]
        scale = np.maximum(np.abs(single), gross)
        assert np.all(np.abs(out[l] - single) <= 1e-6 * scale + 1e-300)


def test_batch_is_deterministic_and_order_free(eng, small_batch):
    yet, pool, layers = small_batch
    a = _run_batch(eng, yet, pool, layers, 3)
    b = _run_batch(eng, yet, pool, layers, 3)
    assert np.array_equal(a, b)
    # listing the layers in another order permutes the outputs exactly
    perm = [3, 0, 5, 1, 4, 2]
    c = _run_batch(eng, yet, pool, [layers[i] for i in perm], 3)
    assert np.array_equal(c, a[perm])


def test_batch_subrange_primary_only_and_halley(eng, small_batch):
    yet, pool, layers = small_batch
    t0, t1 = 137, 911
    out = _run_batch(eng, yet, pool, layers, 9, t0, t1, primary_only=True)
    for l, (ids, terms, sub) in enumerate(layers):
        ref = oracle.run_layer(yet, sub, terms, seed=9, primary_only=True, trials=np.arange(t0, t1))
        check_ylt(out[l], ref)
    out = _run_batch(eng, yet, pool, layers, 9, 0, 300, newton_only=True)
    for l, (ids, terms, sub) in enumerate(layers):
        ref = oracle.run_layer(yet, sub, terms, seed=9, trials=np.arange(0, 300))
        check_ylt(out[l], ref)


def test_batch_of_one_layer_and_of_full_layers(eng):
    # one layer; then 32 layers, all 32 ELTs each (the batch limits), over a small YET
    yet, pool, layers = _batch_case(300, 5000, 60.0, 32, 400, 1, 32, 777)
    out = _run_batch(eng, yet, pool, layers, 1)
    check_ylt(out[0], oracle.run_layer(yet, layers[0][2], layers[0][1], seed=1))
    ids = pool.elt_ids
    terms = oracle.calibrate_layer_terms(yet, pool)
    full = [(ids, terms, pool)] * 32
    out = _run_batch(eng, yet, pool, full, 1)
    ref = oracle.run_layer(yet, pool, terms, seed=1)
    for l in range(32):
        check_ylt(out[l], ref)


def test_paper_shaped_batch_sampled(eng):
    # the paper-1m YET (first 2,000 trials), a pool of 64 ELTs x 10,000 records,
    # 16 layers of 1..32 ELTs: the shapes of the batched workload
    spec = synth.WORKLOADS["paper-1m"]
    yet = synth.make_yet(2000, spec["mean_events"], spec["catalogue"], spec["seed"])
    pool = synth.make_elt_pool(64, spec["entries"], spec["catalogue"], spec["seed"] + 7)
    layer_ids = synth.draw_layers(16, pool.elt_ids, 32, spec["seed"] + 8)
    layers = []
    for ids in layer_ids:
        sub = pool.subset([int(np.flatnonzero(pool.elt_ids == i)[0]) for i in ids])
        layers.append((ids, oracle.calibrate_layer_terms(yet, sub), sub))
    out = _run_batch(eng, yet, pool, layers, 0)
    for l, (ids, terms, sub) in enumerate(layers):
        check_ylt(out[l], oracle.run_layer(yet, sub, terms, seed=0))


def test_a_layer_alone_and_in_a_batch_agree(eng):
    # each layer of a 16-layer batch (about 320 hit records per trial) against the
    # layer alone (at most about 160): the same fixed-point sums, so each layer's
    # year losses are identical bit for bit
    spec = synth.WORKLOADS["paper-1m"]
    yet = synth.make_yet(1200, spec["mean_events"], spec["catalogue"], spec["seed"])
    pool = synth.make_elt_pool(64, spec["entries"], spec["catalogue"], spec["seed"] + 7)
    layer_ids = synth.draw_layers(16, pool.elt_ids, 32, spec["seed"] + 8)
    layers = [(ids, (50.0, 5e6, 1e4, 5e7), None) for ids in layer_ids]
    both = _run_batch(eng, yet, pool, layers, 5)
    for l, layer in enumerate(layers):
        alone = _run_batch(eng, yet, pool, [layer], 5)
        assert np.array_equal(alone[0], both[l])
    assert np.count_nonzero(both) > both.size // 2


def test_batch_errors(eng, small_batch):
    from paper_1501_06326_gb300 import ara

    yet, pool, layers = small_batch
    eng.load_yet(yet.offsets, yet.event_ids, yet.catalogue_size)
    eng.load_pool(pool)
    out = np.zeros((40, 10))
    spec = [(l[0], l[1]) for l in layers]
    with pytest.raises(ara.AraError) as e:  # too many layers
        eng.run_layers(spec * 7, 0, 0, 10, out)
    assert e.value.code == ara.ARA_EINVAL
    with pytest.raises(ara.AraError) as e:  # an ELT that is not loaded
        eng.run_layers(spec + [([999], spec[0][1])], 0, 0, 10, out)
    assert e.value.code == ara.ARA_ENOTLOADED
    with pytest.raises(ara.AraError) as e:  # bad range
        eng.run_layers(spec, 0, 5, 5, out)
    assert e.value.code == ara.ARA_EINVAL
    big = synth.make_elt_pool(70, 20, yet.catalogue_size, 5)
    big.elt_ids = big.elt_ids + 1000
    eng.load_pool(big)
    wide = [(big.elt_ids[:32], spec[0][1]), (big.elt_ids[32:64], spec[0][1]), (big.elt_ids[64:], spec[0][1])]
    with pytest.raises(ara.AraError) as e:  # union of 70 ELTs
        eng.run_layers(wide, 0, 0, 10, out)
    assert e.value.code == ara.ARA_EINVAL


def test_batch_with_empty_and_long_trials(eng):
    # empty trials (also at tile starts and ends), a trial longer than a gather step,
    # a partial last tile: the per-trial record ranges of each tile
    rng = np.random.default_rng(11)
    C = 2003
    lens = [0, 0, 3, 0, 4097, 0, 0, 0, 0, 1, 0, 250] + list(rng.integers(0, 40, 203)) + [0, 0]
    offsets = np.zeros(len(lens) + 1, np.int64)
    offsets[1:] = np.cumsum(lens)
    yet = synth.YET(offsets, rng.integers(0, C, offsets[-1]).astype(np.int32), C)
    pool = synth.make_elt_pool(6, 300, C, 31)
    layer_ids = [np.array([0, 1, 2], np.int32), np.array([2, 3, 4, 5], np.int32), np.array([5], np.int32)]
    layers = []
    for ids in layer_ids:
        sub = pool.subset([int(i) for i in ids])
        layers.append((ids, (100.0, 5e5, 1e3, 5e6), sub))
    out = _run_batch(eng, yet, pool, layers, 2)
    for l, (ids, terms, sub) in enumerate(layers):
        check_ylt(out[l], oracle.run_layer(yet, sub, terms, seed=2))
    out = _run_batch(eng, yet, pool, layers, 2, 3, 200)
    for l, (ids, terms, sub) in enumerate(layers):
        check_ylt(out[l], oracle.run_layer(yet, sub, terms, seed=2, trials=np.arange(3, 200)))


def test_autotuner_keeps_the_results_and_caches_its_choice(eng, small_batch):
    """ARA_AUTOTUNE measures the losses kernel's configurations on the first pass
    of a batch shape and keeps the fastest; every configuration gives the same
    bits, so the tuned pass equals the default one, and a later pass of the same
    shape (without the flag) reuses the choice."""
    yet, pool, layers = small_batch
    t1 = yet.n_trials - 3  # a shape of its own: nothing cached for it yet
    base = _run_batch(eng, yet, pool, layers, 5, t1=t1)
    assert eng.stats()["batch_tuned"] == 0
    tuned = _run_batch(eng, yet, pool, layers, 5, t1=t1, autotune=True)
    st = eng.stats()
    assert st["batch_tuned"] == 1 and st["batch_item"] in (0, 1, 2) and 2 <= st["batch_blocks_per_sm"] <= 16
    again = _run_batch(eng, yet, pool, layers, 5, t1=t1)
    st2 = eng.stats()
    assert st2["batch_tuned"] == 1
    assert (st2["batch_item"], st2["batch_blocks_per_sm"]) == (st["batch_item"], st["batch_blocks_per_sm"])
    assert np.array_equal(base, tuned) and np.array_equal(base, again)


def _run_items(eng, yet, pool, layers, seed, t0=0, t1=None, blocks=(0,), **kw):
    """The pass under each work item (and CTAs per SM) pinned by ara_set_batch_config;
    the indexed item after the YET's event-major index is built."""
    from paper_1501_06326_gb300 import ara

    outs = {}
    try:
        for item in (ara.ARA_BATCH_ITEM_TILE, ara.ARA_BATCH_ITEM_TRIAL, ara.ARA_BATCH_ITEM_DENSE,
                     ara.ARA_BATCH_ITEM_INDEXED):
            for b in blocks:
                eng.set_batch_config(item, b)
                outs[(item, b)] = _run_batch(eng, yet, pool, layers, seed, t0, t1,
                                             index=item == ara.ARA_BATCH_ITEM_INDEXED, **kw)
                st = eng.stats()
                assert st["batch_item"] == item and st["batch_tuned"] == 0
                assert b == 0 or st["batch_blocks_per_sm"] == b
    finally:
        eng.set_batch_config(ara.ARA_BATCH_AUTO)
    return outs


def _assert_same_bits(outs):
    ref = next(iter(outs.values()))
    for key, out in outs.items():
        assert np.array_equal(out, ref), f"work item / blocks {key} differs"
    return ref


def test_work_items_give_the_same_bits(eng):
    """The three losses kernels (a lane per record over a tile or over one trial,
    a lane per pair over a tile) add the same fixed-point numbers: identical
    bits on the paper-shaped 16-layer batch, at 2 CTAs per SM and at the most
    an SM holds; the dense kernel's result against the oracle."""
    spec = synth.WORKLOADS["paper-1m"]
    yet = synth.make_yet(600, spec["mean_events"], spec["catalogue"], spec["seed"] + 3)
    pool = synth.make_elt_pool(64, spec["entries"], spec["catalogue"], spec["seed"] + 7)
    layer_ids = synth.draw_layers(16, pool.elt_ids, 32, spec["seed"] + 8)
    layers = []
    for ids in layer_ids:
        sub = pool.subset([int(np.flatnonzero(pool.elt_ids == i)[0]) for i in ids])
        layers.append((ids, oracle.calibrate_layer_terms(yet, sub), sub))
    out = _assert_same_bits(_run_items(eng, yet, pool, layers, 4, blocks=(0, 2)))
    for l in (0, 7, 15):
        check_ylt(out[l], oracle.run_layer(yet, layers[l][2], layers[l][1], seed=4))
    # a subrange whose first tile is partial, and the Halley path for every pair
    _assert_same_bits(_run_items(eng, yet, pool, layers, 4, 13, 470))
    out = _assert_same_bits(_run_items(eng, yet, pool, layers[:4], 4, 0, 100, newton_only=True))
    for l in range(4):
        check_ylt(out[l], oracle.run_layer(yet, layers[l][2], layers[l][1], seed=4, trials=np.arange(100)))


def test_work_items_on_events_with_64_pairs(eng):
    """Every ELT of a 64-ELT pool holds every event of a 300-event catalogue, so
    each hit event has one pair per ELT (64, the most a record holds): long
    records cross the dense kernel's compute rounds and fill its pair ring; one
    trial has 4,097 such events.  32 layers of up to 32 ELTs; all work items
    agree, and match the oracle."""
    C = 300
    base = synth.make_yet(160, 40.0, C, 91)
    # and a 4,097-event trial (262,208 pairs in one tile) between empty ones
    rng = np.random.default_rng(94)
    lens = np.diff(base.offsets).tolist()
    lens[17:17] = [0, 4097, 0]
    offsets = np.zeros(len(lens) + 1, np.int64)
    offsets[1:] = np.cumsum(lens)
    ev = np.concatenate([base.event_ids[: base.offsets[17]], rng.integers(0, C, 4097).astype(np.int32),
                         base.event_ids[base.offsets[17]:]])
    yet = synth.YET(offsets, ev, C)
    pool = synth.make_elt_pool(64, C, C, 92)
    layer_ids = synth.draw_layers(32, pool.elt_ids, 32, 93)
    layers = []
    for ids in layer_ids:
        sub = pool.subset([int(np.flatnonzero(pool.elt_ids == i)[0]) for i in ids])
        layers.append((ids, oracle.calibrate_layer_terms(yet, sub), sub))
    out = _assert_same_bits(_run_items(eng, yet, pool, layers, 6))
    for l in (0, 13, 31):
        check_ylt(out[l], oracle.run_layer(yet, layers[l][2], layers[l][1], seed=6))


@pytest.mark.parametrize("n_elts,n_layers", [(31, 16), (32, 17), (33, 5), (40, 32)])
def test_work_items_around_a_window(eng, n_elts, n_layers):
    """Events whose pairs just fill the dense kernel's window of 32, or are one
    more (taken alone), among events of one pair, in trials of 0 to 70 events,
    and a subrange of them: all work items agree."""
    C = 500
    rng = np.random.default_rng(n_elts)
    base = synth.make_elt_pool(n_elts, 250, C, 55)
    wide = rng.choice(C, 150, replace=False)  # held by every ELT
    ids = np.concatenate([np.sort(np.concatenate([wide, rng.choice(np.setdiff1d(np.arange(C), wide), 100, replace=False)]))
                          for _ in range(n_elts)]).astype(np.int32)
    pool = synth.ELTPool(elt_ids=base.elt_ids, rec_offsets=base.rec_offsets, event_ids=ids, mean=base.mean,
                         sigma=base.sigma, exposure=base.exposure, terms=base.terms)
    offsets = np.zeros(302, np.int64)
    offsets[1:] = np.cumsum(rng.integers(0, 71, 301))
    yet = synth.YET(offsets, rng.integers(0, C, int(offsets[-1])).astype(np.int32), C)
    layers = [(np.sort(rng.choice(pool.elt_ids, rng.integers(1, min(n_elts, 32) + 1), replace=False)),
               (10.0 * l, 1e6, 1e2, 1e8), None) for l in range(n_layers - 1)] + [(pool.elt_ids[-32:], (0.0, 1e9, 0.0, 1e12), None)]
    layers[0] = (pool.elt_ids[:32], layers[0][1], None)
    _assert_same_bits(_run_items(eng, yet, pool, layers, 9))
    _assert_same_bits(_run_items(eng, yet, pool, layers, 9, 5, 290))


def test_work_items_on_empty_and_long_trials(eng):
    """Empty trials (at tile starts and ends), a 4,097-event trial, a partial last
    tile, and a subrange: all work items agree."""
    rng = np.random.default_rng(12)
    C = 2003
    lens = [0, 0, 3, 0, 4097, 0, 0, 0, 0, 1, 0, 250] + list(rng.integers(0, 40, 203)) + [0, 0]
    offsets = np.zeros(len(lens) + 1, np.int64)
    offsets[1:] = np.cumsum(lens)
    yet = synth.YET(offsets, rng.integers(0, C, offsets[-1]).astype(np.int32), C)
    pool = synth.make_elt_pool(6, 300, C, 32)
    layers = [(np.array(ids, np.int32), (100.0, 5e5, 1e3, 5e6), None)
              for ids in ([0, 1, 2], [2, 3, 4, 5], [5], [0, 5])]
    _assert_same_bits(_run_items(eng, yet, pool, layers, 2))
    _assert_same_bits(_run_items(eng, yet, pool, layers, 2, 3, 200))
    _assert_same_bits(_run_items(eng, yet, pool, layers, 2, 4, 5))


def test_indexed_pass_across_slices_and_grid_cells(eng):
    """A YET of 600,000 trials and 32 layers: the indexed pass runs in three
    slices of 262,144 trials, over three cells of the index's trial grid.
    Passes whose bounds are on the grid, inside a cell, inside one cell at both
    ends, and up to the YET's end; the indexed item gives the dense item's bits
    on each, and sampled trials match the oracle."""
    yet = synth.make_yet(600_000, 4.0, 3000, 61)
    pool = synth.make_elt_pool(8, 1000, 3000, 62)
    layer_ids = synth.draw_layers(32, pool.elt_ids, 4, 63)
    layers = [(ids, (10.0, 5e5, 1e2, 5e6), pool.subset([int(i) for i in ids])) for ids in layer_ids]
    for t0, t1 in ((0, 600_000), (262_144, 524_288), (70_001, 590_001), (262_145, 262_999),
                   (262_143, 600_000), (599_999, 600_000)):
        out = _assert_same_bits(_run_items(eng, yet, pool, layers, 8, t0, t1))
        assert np.count_nonzero(out) > 0
    # trials on both sides of a grid and slice bound, against the oracle
    t0, t1 = 262_000, 262_300
    out = _assert_same_bits(_run_items(eng, yet, pool, layers, 8, t0, t1))
    for l in (0, 11, 31):
        ids, terms, sub = layers[l]
        check_ylt(out[l], oracle.run_layer(yet, sub, terms, seed=8, trials=np.arange(t0, t1)))


@pytest.mark.parametrize("n_layers", [1, 2, 3, 4, 6, 32])
def test_indexed_layers_of_an_event(eng, n_layers):
    """The indexed item's adds by lanes of four, two and one: ELT i serves the
    first i + 1 layers, so events serve 1 to n_layers of them, events of one
    pair and of several, of every kind of record, with 0 to 70 occurrences
    (windows of 32 and what is left over); the dense item's bits."""
    rng = np.random.default_rng(n_layers)
    C = 1_500
    base = synth.make_elt_pool(n_layers, 220, C, 70, recipe="stress")
    sigma = np.where(rng.random(len(base.sigma)) < 0.1, 0.0, base.sigma).astype(base.sigma.dtype)
    mean = np.where(rng.random(len(base.mean)) < 0.1, 0.0, base.mean).astype(base.mean.dtype)
    pool = synth.ELTPool(elt_ids=base.elt_ids, rec_offsets=base.rec_offsets, event_ids=base.event_ids, mean=mean,
                         sigma=sigma, exposure=base.exposure, terms=base.terms)
    ev = np.repeat(np.arange(C), rng.integers(0, 71, C)).astype(np.int32)
    rng.shuffle(ev)
    n = 5_003
    offsets = np.zeros(n + 1, np.int64)
    offsets[1:] = np.sort(rng.integers(0, len(ev) + 1, n))
    offsets[-1] = len(ev)
    yet = synth.YET(offsets, ev, C)
    ids = pool.elt_ids
    layers = [(ids[l:], (50.0 * l, 4e5, 1e2, 5e7), None) for l in range(n_layers)]
    for kw in ({}, {"primary_only": True}):
        out = _assert_same_bits(_run_items(eng, yet, pool, layers, 3, **kw))
        assert np.count_nonzero(out[0]) > 0
    _assert_same_bits(_run_items(eng, yet, pool, layers, 3, 17, 4_001))


def test_yet_index_by_radix_sort_where_an_event_is_frequent(eng):
    """An event in every trial of a 3,000-trial YET (a bucket of 3,000
    occurrences, above the bucket build's 2,048) has the index built by the
    radix sort; the indexed passes give the dense item's bits there, and on
    the same YET without the frequent event, built by buckets."""
    pool = synth.make_elt_pool(6, 400, 1500, 72)
    e_hot = int(pool.event_ids[0])  # an event of ELT 0
    base = synth.make_yet(3000, 30.0, 1500, 71)
    lens = np.diff(base.offsets) + 1
    offsets = np.zeros(len(lens) + 1, np.int64)
    offsets[1:] = np.cumsum(lens)
    ev = np.empty(offsets[-1], np.int32)
    for t in range(base.n_trials):  # the frequent event first in every trial, then the trial's own events
        ev[offsets[t]] = e_hot
        ev[offsets[t] + 1: offsets[t + 1]] = base.event_ids[base.offsets[t]: base.offsets[t + 1]]
    hot = synth.YET(offsets, ev, 1500)
    layers = [(np.array(ids, np.int32), (10.0, 5e5, 1e2, 5e6), None) for ids in ([0, 1], [1, 2, 3], [0, 4, 5])]
    for yet, method in ((hot, "radix sort"), (base, "buckets")):
        for t0, t1 in ((0, yet.n_trials), (17, 2903)):
            _assert_same_bits(_run_items(eng, yet, pool, layers, 3, t0, t1))
            assert eng.yet_index_info()["method"] == method


def test_batch_config_errors(eng):
    from paper_1501_06326_gb300 import ara

    for item, blocks in ((4, 0), (-2, 0), (ara.ARA_BATCH_ITEM_DENSE, -1), (ara.ARA_BATCH_ITEM_TILE, 17)):
        with pytest.raises(ara.AraError) as e:
            eng.set_batch_config(item, blocks)
        assert e.value.code == ara.ARA_EINVAL
    eng.set_batch_config(ara.ARA_BATCH_AUTO)


def test_yet_index_default_and_errors(eng, small_batch):
    """Without an index the indexed item is refused; once built, batched passes
    default to it and give the same bits as the dense item; a new YET load drops
    the index; building needs a YET."""
    from paper_1501_06326_gb300 import ara

    yet, pool, layers = small_batch
    fresh = ara.Ara(0)
    with pytest.raises(ara.AraError) as e:
        fresh.build_yet_index()
    assert e.value.code == ara.ARA_ENOTLOADED
    fresh.close()
    dense = _run_batch(eng, yet, pool, layers, 8)
    assert eng.stats()["batch_item"] == ara.ARA_BATCH_ITEM_DENSE
    eng.set_batch_config(ara.ARA_BATCH_ITEM_INDEXED)
    try:
        with pytest.raises(ara.AraError) as e:
            _run_batch(eng, yet, pool, layers, 8)
        assert e.value.code == ara.ARA_EINVAL
    finally:
        eng.set_batch_config(ara.ARA_BATCH_AUTO)
    indexed = _run_batch(eng, yet, pool, layers, 8, index=True)
    assert eng.stats()["batch_item"] == ara.ARA_BATCH_ITEM_INDEXED
    info = eng.yet_index_info()
    assert info["built"] and info["bytes"] >= 8 * yet.n_events and info["method"] == "buckets"
    assert np.array_equal(dense, indexed)
    eng.load_yet(yet.offsets, yet.event_ids, yet.catalogue_size)
    assert not eng.yet_index_info()["built"] and eng.yet_index_info()["method"] is None


@pytest.mark.parametrize("shape", ["one-event", "tile", "tile-and-one", "short-trials", "long-trials", "two-digits",
                                   "wide-digits", "beyond-the-fields"])
def test_yet_index_partitions(eng, shape):
    """The partition build of the index at the edges of its tiles (16,384
    occurrences), of its digits (2,048 ids each) and of its trial lookup (many
    empty trials, trials longer than a tile): whole passes and passes whose
    bounds lie inside a grid cell (found by a search over the occurrences'
    trials) give the dense item's bits.  A catalogue beyond the partitions'
    fields (2^22 ids) takes the bucket build."""
    rng = np.random.default_rng(len(shape))
    lens, C = {
        "one-event": ([0, 1, 0], 300),
        "tile": ([16_384 // 64] * 64, 2_048),
        "tile-and-one": ([16_384 // 64] * 64 + [1], 2_049),
        "short-trials": (list(rng.integers(0, 3, 30_000)) + [0] * 5_000 + list(rng.integers(0, 2, 20_000)), 5_000),
        "long-trials": ([3, 40_000, 0, 17_000, 20_011], 70_001),
        "two-digits": (list(rng.integers(0, 90, 3_001)), 131_072),
        "wide-digits": (list(rng.integers(0, 400, 2_003)), 1 << 22),
        "beyond-the-fields": (list(rng.integers(0, 400, 503)), (1 << 22) + 1),
    }[shape]
    offsets = np.zeros(len(lens) + 1, np.int64)
    offsets[1:] = np.cumsum(lens)
    n = int(offsets[-1])
    pool = synth.make_elt_pool(5, min(C, 4_000), C, 33)
    ev = rng.integers(0, C, n).astype(np.int32)
    held = rng.random(n) < 0.5  # half the occurrences are of events that ELTs hold
    ev[held] = rng.choice(pool.event_ids, int(held.sum()))
    yet = synth.YET(offsets, ev, C)
    layers = [(np.array(ids, np.int32), (10.0, 5e5, 1e2, 5e7), None) for ids in ([0, 1, 2], [2, 3, 4], [4])]
    N = len(lens)
    for t0, t1 in {(0, N), (N // 3, N - N // 5), (N // 2, N // 2 + 1)}:
        _assert_same_bits(_run_items(eng, yet, pool, layers, 2, t0, t1))
    assert eng.yet_index_info()["method"] == "buckets"


def test_yet_index_at_its_event_limit(eng):
    """A YET of 2^32 - 2 events, the most an index takes: the last digit's
    bucket and the last events' occurrences end within a block and a window of
    2^32, where a 32-bit position would wrap.  The indexed passes over the
    first and last trials give the dense item's bits."""
    import torch

    from paper_1501_06326_gb300 import ara

    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 140 << 30:
        pytest.skip("needs 140 GB of device memory")
    C, N, n = 1 << 22, 2048, (1 << 32) - 2
    offsets = np.minimum(np.arange(N + 1, dtype=np.int64) << 21, n)
    # the last 2,048 ids have 500 occurrences, in the last two trials
    ids = torch.randint(0, C - 2048, (n,), dtype=torch.int32, device="cuda")
    late = torch.arange(C - 2048, C, dtype=torch.int32, device="cuda")[-50:].repeat(10)
    ids[n - (1 << 21):][torch.randperm(1 << 21, device="cuda")[:250]] = late[:250]
    ids[n - (1 << 22): n - (1 << 21)][:250] = late[250:]
    torch.cuda.synchronize()
    pool = synth.make_elt_pool(3, 2_000, C, 8)
    held = np.sort(np.random.default_rng(8).choice(C - 2048, 1_950, replace=False))
    pool.event_ids[:2_000] = np.concatenate([held, late[:50].cpu().numpy()])
    big = ara.Ara(0)
    try:
        big.load_yet(offsets, ids, C)
        del ids, late
        torch.cuda.empty_cache()
        big.load_pool(pool)
        big.build_yet_index()
        layers = [([0, 1], (10.0, 5e5, 1e2, 5e9)), ([0], (0.0, 1e9, 0.0, 1e12))]
        for t0, t1 in ((0, 2), (N - 3, N), (N - 1, N)):
            got = {}
            for item in (ara.ARA_BATCH_ITEM_DENSE, ara.ARA_BATCH_ITEM_INDEXED):
                big.set_batch_config(item)
                got[item] = np.zeros((2, t1 - t0))
                big.run_layers(layers, 5, t0, t1, got[item])
            assert np.array_equal(got[ara.ARA_BATCH_ITEM_DENSE], got[ara.ARA_BATCH_ITEM_INDEXED])
            assert np.all(got[ara.ARA_BATCH_ITEM_DENSE][1] > 0.0)
    finally:
        big.close()


def _on_two_threads(work, arguments):
    """work(engine, argument) on two host threads, each with its own context."""
    import threading

    from paper_1501_06326_gb300 import ara

    errors = []

    def go(argument):
        own = ara.Ara(0)
        try:
            work(own, argument)
        except Exception as e:  # noqa: BLE001
            errors.append(e)
        finally:
            own.close()

    threads = [threading.Thread(target=go, args=(a,)) for a in arguments]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_contexts_on_threads_with_unlike_catalogues(eng):
    """Two contexts on two threads whose gathers need 40 and 195 KB of shared
    memory: a call on one does not lower the other's limit."""

    def layers(own, catalogue):
        yet, pool = synth.make_yet(200, 20.0, catalogue, 3), synth.make_elt_pool(2, 300, catalogue, 4)
        own.load_yet(yet.offsets, yet.event_ids, catalogue)
        own.load_pool(pool)
        first, out = np.zeros(yet.n_trials), np.zeros(yet.n_trials)
        own.run_layer(pool.elt_ids, (10.0, 1e6, 1e2, 1e8), 1, 0, yet.n_trials, first)
        for _ in range(2_000):
            own.run_layer(pool.elt_ids, (10.0, 1e6, 1e2, 1e8), 1, 0, yet.n_trials, out)
            assert np.array_equal(out, first)

    _on_two_threads(layers, (1_000, 2_000_000))


def test_contexts_on_threads_index_unlike_yets(eng):
    """Two contexts on two threads that index YETs of one and of eight grid
    cells (8 and 64 KB of shared memory for the cells' counts)."""

    def build(own, shape):
        trials, per_trial = shape
        offsets = np.arange(trials + 1, dtype=np.int64) * per_trial
        ids = np.random.default_rng(1).integers(0, 1 << 22, int(offsets[-1])).astype(np.int32)
        for _ in range(60):
            own.load_yet(offsets, ids, 1 << 22)
            own.build_yet_index()
            assert own.yet_index_info()["method"] == "buckets"

    _on_two_threads(build, ((2_000, 1_050), (2_097_152, 1)))


def _even_yet(trials, per_trial, C, seed):
    offsets = np.arange(trials + 1, dtype=np.int64) * per_trial
    return synth.YET(offsets, np.random.default_rng(seed).integers(0, C, trials * per_trial).astype(np.int32), C)


@pytest.mark.parametrize("use", ["a pass", "a tail"])
def test_yet_index_holds_its_own_memory_only(use):
    """A build keeps the index's bytes and nothing else; after the next YET's
    load the first call other than the build gives them back to the device,
    and a build straight after the load takes them over."""
    import torch

    from paper_1501_06326_gb300 import ara

    yet, pool = _even_yet(8_000, 1_000, 1 << 20, 3), synth.make_elt_pool(2, 500, 1 << 20, 4)
    out = np.zeros(50)
    own = ara.Ara(0)

    def call():
        if use == "a pass":
            own.run_layer(pool.elt_ids, (10.0, 1e6, 1e2, 1e8), 1, 0, 50, out)
        else:
            own.pml_tvar(out, [2.0])

    try:
        own.load_pool(pool)
        free = []
        for step in ("load", "call", "build", "load", "call", "build", "load", "build", "call"):
            if step == "load":
                own.load_yet(yet.offsets, yet.event_ids, yet.catalogue_size)
            elif step == "build":
                own.build_yet_index()
            else:
                call()
            free.append(torch.cuda.mem_get_info()[0])
        slack = 12 << 20  # six buffers' rounding to 2 MB
        index = own.yet_index_info()["bytes"]
        assert index >= 8 * yet.n_events
        assert abs(free[1] - free[2] - index) <= slack
        assert abs(free[1] - free[4]) <= slack
        assert abs(free[1] - free[5] - index) <= slack and abs(free[1] - free[8] - index) <= slack
    finally:
        own.close()


def test_yet_index_leaves_captured_calls_their_buffers():
    """A layer call captured over a few trials replays with the same bits after
    an index build, whose scratch is larger than the call's event buffer."""
    import torch

    from paper_1501_06326_gb300 import ara

    yet, pool = _even_yet(8_000, 1_000, 20_000, 4), synth.make_elt_pool(3, 500, 20_000, 5)
    stream = torch.cuda.Stream()
    own = ara.Ara(0, 0, stream.cuda_stream)
    try:
        own.load_yet(yet.offsets, yet.event_ids, yet.catalogue_size)
        own.load_pool(pool)
        out = torch.zeros(50, dtype=torch.float64, device="cuda")
        run = lambda: own.run_layer(pool.elt_ids, (10.0, 1e6, 1e2, 1e8), 1, 0, 50, out)  # noqa: E731
        run()
        torch.cuda.synchronize()
        first = out.cpu().numpy()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            run()
        own.build_yet_index()
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), first) and np.count_nonzero(first) > 0
    finally:
        own.close()


@pytest.mark.parametrize("shape", ["short-trials", "dense", "dense-long-trials", "uneven"])
def test_yet_index_of_many_tiles(eng, shape):
    """YETs whose partitions take several tiles of 16,384 occurrences a CTA: in
    the first (above 608 tiles; trials from none to thousands of events, so that
    a tile ends in any of them) and in the second (a catalogue of 300 ids, whose
    events have far more occurrences than a thread would sort, and which the
    partitions still index).  A fifth of the events alike: one CTA's
    bucket, left to the radix sort.  The dense item's bits, over all trials and
    within a grid cell."""
    rng = np.random.default_rng(len(shape))
    lens, C, method = {
        "short-trials": (np.where(rng.random(400_000) < 0.9, rng.integers(0, 40, 400_000), 0), 1 << 21, "buckets"),
        "dense": (rng.integers(0, 60, 400_000), 300, "buckets"),
        "dense-long-trials": (np.concatenate([[0, 3_000_000, 0, 1], rng.integers(0, 20_000, 950)]), 4_000, "buckets"),
        "uneven": (rng.integers(0, 60, 100_000), 4_000, "radix sort"),
    }[shape]
    if shape == "short-trials":
        lens[::5_000] = 60_000
    offsets = np.zeros(len(lens) + 1, np.int64)
    offsets[1:] = np.cumsum(lens)
    n, N = int(offsets[-1]), len(lens)
    pool = synth.make_elt_pool(4, min(C // 2, 300), C, 33)
    ev = rng.integers(0, C, n, dtype=np.int32)
    if shape == "short-trials":
        ev[::3] = rng.choice(pool.event_ids, len(ev[::3]))
    if shape == "uneven":
        ev[::5] = pool.event_ids[0]
    yet = synth.YET(offsets, ev, C)
    layers = [(np.array(ids, np.int32), (10.0, 5e5, 1e2, 5e9), None) for ids in ([0, 1], [1, 2, 3])]
    for t0, t1 in {(0, N), (N // 3, N - N // 5)}:
        _assert_same_bits(_run_items(eng, yet, pool, layers, 2, t0, t1))
    assert eng.yet_index_info()["method"] == method


@pytest.mark.parametrize("shape,launches", [("few", 5), ("tile", 7), ("tile-and-one", 7), ("short-trials", 7),
                                            ("long-trials", 7), ("many-digits", 9)])
def test_yet_index_partition_edges(eng, shape, launches):
    """The partitions at the edges of their tiles (16,384 occurrences), of their
    trial lookup (many empty trials, trials longer than a tile) and of the line
    below which a YET has too few events for them (16 a catalogue id, which the
    launches of the build show): the dense item's bits."""
    rng = np.random.default_rng(len(shape))
    lens, C = {
        "few": ([16_000 // 64] * 64, 1_000),
        "tile": ([16_384 // 64] * 64, 1_000),
        "tile-and-one": ([16_384 // 64] * 64 + [1], 1_023),
        "short-trials": (list(rng.integers(0, 3, 30_000)) + [0] * 5_000 + list(rng.integers(0, 2, 20_000)), 1_025),
        "long-trials": ([3, 40_000, 0, 17_000, 20_011], 2_049),
        "many-digits": ([1_001] * 600, 16_385),
    }[shape]
    offsets = np.zeros(len(lens) + 1, np.int64)
    offsets[1:] = np.cumsum(lens)
    n, N = int(offsets[-1]), len(lens)
    pool = synth.make_elt_pool(5, 400, C, 33)
    ev = rng.integers(0, C, n, dtype=np.int32)
    yet = synth.YET(offsets, ev, C)
    layers = [(np.array(ids, np.int32), (10.0, 5e5, 1e2, 5e7), None) for ids in ([0, 1, 2], [2, 3, 4], [4])]
    for t0, t1 in {(0, N), (N // 3, N - N // 5), (N // 2, N // 2 + 1)}:
        _assert_same_bits(_run_items(eng, yet, pool, layers, 2, t0, t1))
    eng.load_yet(yet.offsets, yet.event_ids, C)
    eng.timing(reset=True)
    eng.build_yet_index()
    assert eng.timing()["kernel_launches"] == launches
