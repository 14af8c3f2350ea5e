"""GPU parity of the device quantizer (Section 6) against the CPU oracle on the same seeded weights: index
streams, outlier offsets, values and counts bit-exact; centroids equal up to one fp32 unit in the last place
(both sides round an fp64 mean once, the summation orders differ).  Every case runs through both methods of the
library (rank selection, the default, and the stable sort it falls back to)."""
import numpy as np
import pytest
import torch

import workloads as W
from workloads.shards import ATTN, FFN, make_unit_weights
from oracle import sti_quantizer_oracle as Q

pytestmark = pytest.mark.gpu

sti = pytest.importorskip("paper_2207_05022_b200")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2207_05022_b200 import build
    build.build_library()
    sti.load_library()


def _run(units, bits, max_out=4096, method=None, want_sorted=False):
    """units: [n_units][n] fp32 on the host -> (words, centroids, offsets, values, counts) from the device."""
    n_units, n = units.shape
    w = torch.from_numpy(units).cuda()
    K = 1 << bits
    codes = torch.zeros((n_units, n * bits // 32), dtype=torch.int32, device="cuda")
    cents = torch.zeros((n_units, K), dtype=torch.float32, device="cuda")
    off = torch.zeros((n_units, max_out), dtype=torch.int32, device="cuda")
    val = torch.zeros((n_units, max_out), dtype=torch.float32, device="cuda")
    cnt = torch.zeros(n_units, dtype=torch.int32, device="cuda")
    ws_bytes = sti.sti_quantize_workspace_bytes(n_units, n)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    by_sort = torch.full((n_units,), 7, dtype=torch.uint8, device="cuda")
    if method is None:
        sti.sti_quantize_units(w.data_ptr(), n_units, n, bits, codes.data_ptr(), cents.data_ptr(), off.data_ptr(),
                               val.data_ptr(), max_out, cnt.data_ptr(), ws.data_ptr(), ws_bytes)
    else:
        sti.sti_quantize_units_by(w.data_ptr(), n_units, n, bits, codes.data_ptr(), cents.data_ptr(), off.data_ptr(),
                                  val.data_ptr(), max_out, cnt.data_ptr(), ws.data_ptr(), ws_bytes, method,
                                  by_sort.data_ptr())
    torch.cuda.synchronize()
    res = (codes.cpu().numpy().view(np.uint32), cents.cpu().numpy(), off.cpu().numpy().view(np.uint32),
           val.cpu().numpy(), cnt.cpu().numpy())
    return res + (by_sort.cpu().numpy(),) if want_sorted else res


def _ulp_diff(a, b):
    ia, ib = a.view(np.int32).astype(np.int64), b.view(np.int32).astype(np.int64)
    ia = np.where(ia < 0, -(ia & 0x7FFFFFFF), ia)
    ib = np.where(ib < 0, -(ib & 0x7FFFFFFF), ib)
    return np.abs(ia - ib)


def _check(units, bits, max_out=4096):
    """Both methods against the oracle; returns which units the default method handed to the sort."""
    refs = [Q.quantize_unit(units[u], bits) for u in range(units.shape[0])]
    _check_one(units, bits, max_out, refs, sti.STI_QUANTIZE_SORT)
    return _check_one(units, bits, max_out, refs, sti.STI_QUANTIZE_SELECT)


def _check_one(units, bits, max_out, refs, method):
    words, cents, off, val, cnt, by_sort = _run(units, bits, max_out, method, want_sorted=True)
    assert set(np.unique(by_sort)) <= {0, 1}
    if method == sti.STI_QUANTIZE_SORT:
        assert by_sort.all()
    _compare(units, bits, max_out, refs, words, cents, off, val, cnt)
    return by_sort


def _compare(units, bits, max_out, refs, words, cents, off, val, cnt):
    for u in range(units.shape[0]):
        rw, rc, ro, rv = refs[u]
        assert cnt[u] == ro.size, (u, bits)
        m = min(ro.size, max_out)
        assert np.array_equal(off[u, :m], ro[:m]) and np.array_equal(val[u, :m].view(np.uint32), rv[:m].view(np.uint32))
        assert _ulp_diff(cents[u], rc).max() <= 1, (u, bits)
        if np.array_equal(cents[u].view(np.uint32), rc.view(np.uint32)):
            assert np.array_equal(words[u], rw), (u, bits)
        else:       # a centroid one unit off can only move an outlier's nearest-centroid index; everything else is exact
            codes = np.asarray(__import__("oracle.sti_oracle", fromlist=["x"]).unpack_codes(words[u], units.shape[1], bits))
            ref = np.asarray(__import__("oracle.sti_oracle", fromlist=["x"]).unpack_codes(rw, units.shape[1], bits))
            inl = np.ones(units.shape[1], bool)
            inl[ro] = False
            assert np.array_equal(codes[inl], ref[inl]), (u, bits)


@pytest.mark.parametrize("bits", [2, 3, 4, 5, 6])
def test_bert_base_units_every_bitwidth(bits):
    shape = W.BERT_BASE
    units = np.stack([np.concatenate([m.reshape(-1) for m in make_unit_weights(shape, 11, l, ATTN, i)])
                      for l, i in ((0, 0), (1, 5), (2, 11))])
    assert not _check(units, bits).any()                  # Gaussian-like weights never need the sort


def test_bert_large_ffn_unit_with_heavy_tails():
    shape = W.BERT_LARGE
    mats = make_unit_weights(shape, 12, 3, FFN, 7, outlier_stress=0.0015)       # 524,288 weights, ~0.15 % outliers
    units = np.concatenate([m.reshape(-1) for m in mats])[None, :]
    assert not _check(units, 3).any()
    assert not _check(units, 6).any()


def test_ties_constant_and_tiny_units():
    rng = np.random.default_rng(5)
    few_values = rng.choice(np.linspace(-0.05, 0.05, 9).astype(np.float32), size=8192)      # massive ties
    signed_zero = few_values.copy()
    signed_zero[::7] = np.float32(-0.0)
    signed_zero[3::7] = np.float32(0.0)
    const = np.full(8192, 0.0125, np.float32)
    ramp = np.arange(8192, dtype=np.float32) * np.float32(1e-5) - np.float32(0.04)
    units = np.stack([few_values, signed_zero, const, ramp])
    for bits in (2, 4, 6):
        by_sort = _check(units, bits)
        assert by_sort[2] == 1                             # zero variance: no value bins to select in
    _check(rng.standard_normal((2, 32)).astype(np.float32) * np.float32(0.02), 5)            # fewer weights than 2 clusters' worth
    _check(rng.standard_normal((1, 1056)).astype(np.float32) * np.float32(0.02), 3)          # ragged last chunk


def test_units_the_selection_hands_to_the_sort():
    """Many equal values: one value bin holds more members than the counting selection accepts.  Mixed in one launch
    with units that the selection does itself."""
    rng = np.random.default_rng(6)
    n = 65536
    ties = rng.choice(np.linspace(-0.05, 0.05, 9).astype(np.float32), size=n)
    normal = (rng.standard_normal(n) * 0.03).astype(np.float32)
    half = normal.copy()
    half[: n // 2] = np.float32(0.01)                     # half the unit is one value
    units = np.stack([normal, ties, half, normal[::-1].copy()])
    for bits in (2, 5):
        by_sort = _check(units, bits)
        assert list(by_sort) == [0, 1, 1, 0]


def test_selection_is_deterministic():
    shape = W.BERT_LARGE
    units = np.stack([np.concatenate([m.reshape(-1) for m in make_unit_weights(shape, 14, 0, ATTN, i)]) for i in range(3)])
    a = _run(units, 6)
    b = _run(units, 6)
    for x, y in zip(a, b):
        assert np.array_equal(x.view(np.uint32) if x.dtype == np.float32 else x, y.view(np.uint32) if y.dtype == np.float32 else y)


@pytest.mark.parametrize("n_units,n,bits", [
    (1, 16384 + 32, 6),          # two CTAs share a unit (a step of 512 weights for each of their warps), ragged end
    (1, 32768, 5), (1, 65536 + 480, 4), (1, 131072 + 1056, 3), (2, 131072 + 8192, 6),      # four, eight, sixteen
    (1, (1 << 18), 2), (1, (1 << 18) + 128, 2),      # the line between 8,192 and 16,384 value bins
    (40, 16384, 3), (80, 33 * 1024, 4)])             # clusters by the dozen
def test_units_shared_by_a_cluster_of_ctas(n_units, n, bits):
    rng = np.random.default_rng(n + bits)
    units = (rng.standard_normal((n_units, n)) * 0.02).astype(np.float32)
    units[rng.random((n_units, n)) < 0.002] *= 10
    ref = [Q.quantize_unit(units[u], bits) for u in range(n_units)]
    assert not _check_one(units, bits, 4096, ref, sti.STI_QUANTIZE_SELECT).any()


def test_units_whose_mean_is_far_off():
    """A mean of many deviations, and a unit whose evenly spaced weights - the fit's provisional centre - are outliers."""
    rng = np.random.default_rng(8)
    n = 65536
    shifted = (rng.standard_normal(n) * 0.001 + 3.0).astype(np.float32)
    misled = (rng.standard_normal(n) * 0.02).astype(np.float32)
    misled[:: n // 32] = 25.0
    for bits in (3, 6):
        _check(np.stack([shifted, misled]), bits)


def test_units_whose_inlier_range_holds_no_fp32_value():
    """A deviation of 16 gives a radius of 12.6; about 3.0e8 fp32 values are 32 apart, so every weight is an outlier and the
    search for the ends of the range has to give up.  Beside a unit of an equally large deviation that has its inliers."""
    rng = np.random.default_rng(9)
    n = 8192
    apart = np.where(rng.permutation(n) < n // 2, np.float32(3.0e8), np.float32(3.0e8 + 32)).astype(np.float32)
    wide = (rng.standard_normal(n) * 16).astype(np.float32)
    for bits in (2, 5):
        assert list(_check(np.stack([apart, wide, -apart]), bits)) == [1, 0, 1]


def test_units_without_an_inlier():
    """Half the weights at -16 and half at +16: the radius of 12.6 leaves a range with fp32 values, but none of the weights."""
    rng = np.random.default_rng(10)
    n = 131072                                             # a cluster of several CTAs
    sign = np.where(rng.permutation(n) < n // 2, np.float32(-16), np.float32(16)).astype(np.float32)
    one = sign.copy()
    one[777] = 0.25                                        # a single inlier: every boundary is that weight
    for bits in (3, 6):
        assert list(_check(np.stack([sign, one]), bits)) == [1, 0]


@pytest.mark.parametrize("n_units,n", [(1, 196608), (3, 65536 + 480), (1, 524288)])
def test_units_shared_by_ctas_that_leave_early(n_units, n):
    """No variance, or a range whose ends are not found: all CTAs of a cluster leave after they have read one another's histograms."""
    rng = np.random.default_rng(n)
    flat = np.zeros((n_units, n), np.float32)
    wide = (rng.standard_normal((n_units, n)) * 30).astype(np.float32)         # above a deviation of 21.8 every weight is an outlier
    apart = np.where(rng.random((n_units, n)) < 0.5, np.float32(3.0e8), np.float32(3.0e8 + 32)).astype(np.float32)
    normal = (rng.standard_normal((1, n)) * 0.02).astype(np.float32)
    for bits in (3, 4):
        for units in (flat, wide, apart):
            assert list(_check(np.concatenate([units, normal]), bits, max_out=n)) == [1] * n_units + [0]


def _long_bins_and_long_tails(n, seed, narrow):
    """Weights with 0.15 % of ten times the spread; with `narrow`, half of the others have a tenth of it.  A warp's run then has
    more tails than its list in shared memory takes, and boundary bins hold more than 256 weights."""
    rng = np.random.default_rng(seed)
    w = (rng.standard_normal(n) * 0.02).astype(np.float32)
    if narrow:
        w[rng.random(n) < 0.5] *= np.float32(0.1)
    else:
        w[rng.random(n) < 0.0015] *= 10
    return w


@pytest.mark.parametrize("n,bits", [(1 << 20, 2), (1 << 20, 3), (1 << 20, 6), (524288, 6), (524288, 2)])
def test_long_boundary_bins_beside_long_lists_of_tails(n, bits):
    units = _long_bins_and_long_tails(n, 1, narrow=True)[None, :]
    assert not _check(units, bits, max_out=n).any()


@pytest.mark.parametrize("n,narrow,bits", [(1 << 21, False, 3), (1 << 21, False, 2), (1 << 18, True, 2), (524288, True, 3)])
def test_long_boundary_bins_beside_long_lists_of_tails_one_cta_per_unit(n, narrow, bits):
    """As many units as the device holds at a time, all the same one."""
    unit = _long_bins_and_long_tails(n, 2, narrow)
    words, cents, off, val = Q.quantize_unit(unit, bits)
    n_units, max_out = 2 * torch.cuda.get_device_properties(0).multi_processor_count, off.size
    w = torch.from_numpy(unit).cuda().expand(n_units, n).contiguous()
    ws_bytes = sti.sti_quantize_workspace_bytes(n_units, n)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda")
    for method in (sti.STI_QUANTIZE_SELECT, sti.STI_QUANTIZE_SORT):
        some = n_units if method == sti.STI_QUANTIZE_SELECT else 1
        codes = torch.zeros((some, n * bits // 32), dtype=torch.int32, device="cuda")
        got_cents = torch.zeros((some, 1 << bits), device="cuda")
        got_off = torch.zeros((some, max_out), dtype=torch.int32, device="cuda")
        got_val = torch.zeros((some, max_out), device="cuda")
        count = torch.zeros(some, dtype=torch.int32, device="cuda")
        by_sort = torch.zeros(some, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        sti.sti_quantize_units_by(w.data_ptr(), some, n, bits, codes.data_ptr(), got_cents.data_ptr(), got_off.data_ptr(), got_val.data_ptr(),
                                  max_out, count.data_ptr(), ws.data_ptr(), ws_bytes, method, by_sort.data_ptr())
        torch.cuda.synchronize()
        assert (by_sort == (0 if method == sti.STI_QUANTIZE_SELECT else 1)).all()
        for out in (codes, got_cents, got_off, got_val, count):
            assert torch.equal(out, out[:1].expand_as(out))
        _compare(unit[None, :], bits, max_out, [(words, cents, off, val)], codes[:1].cpu().numpy().view(np.uint32), got_cents[:1].cpu().numpy(),
                 got_off[:1].cpu().numpy().view(np.uint32), got_val[:1].cpu().numpy(), count[:1].cpu().numpy())


def test_outlier_lists_shorter_than_the_outliers_found():
    shape = W.ModelShape(n_layers=1, hidden=256, n_heads=4, head_dim=64, ffn=1024, n_ffn_slices=4)
    mats = make_unit_weights(shape, 13, 0, FFN, 1, outlier_stress=0.01)
    units = np.concatenate([m.reshape(-1) for m in mats])[None, :]
    _check(units, 4, max_out=16)          # count reported in full, lists truncated, index stream complete


def test_argument_checks():
    w = torch.zeros(64, device="cuda")
    buf = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    p = buf.data_ptr()
    with pytest.raises(sti.StiError) as e:
        sti.sti_quantize_units(w.data_ptr(), 1, 64, 7, p, p, p, p, 4, p, p, 4096)
    assert e.value.status == 2
    with pytest.raises(sti.StiError) as e:
        sti.sti_quantize_units(w.data_ptr(), 1, 48, 4, p, p, p, p, 4, p, p, 4096)
    assert e.value.status == 3
    with pytest.raises(sti.StiError) as e:
        sti.sti_quantize_units(w.data_ptr(), 1, 64, 4, p, p, p, p, 4, p, p, 100)
    assert e.value.status == 4
    big = torch.zeros(1 << 16, dtype=torch.uint8, device="cuda")
    q = big.data_ptr()
    with pytest.raises(sti.StiError) as e:                               # no such method
        sti.sti_quantize_units_by(w.data_ptr(), 1, 64, 4, q, q, q, q, 4, q, q, 1 << 16, 2)
    assert e.value.status == 1
    with pytest.raises(sti.StiError) as e:                               # weights not 16-byte aligned
        sti.sti_quantize_units(w.data_ptr() + 4, 1, 32, 4, q, q, q, q, 4, q, q, 1 << 16)
    assert e.value.status == 1


def test_device_quantized_units_run_through_the_layer():
    """fp32 weights -> sti_quantize_units -> sti_shard_upload -> sti_layer_forward, against the oracle's forward
    on the oracle's own quantization of the same weights."""
    from gpu_util import run_layer, rel_err, REL_TOL
    from oracle import sti_oracle as O
    from workloads.shards import ShardBlob
    shape = W.ModelShape(n_layers=1, hidden=256, n_heads=4, head_dim=64, ffn=1024, n_ffn_slices=4)
    bits_of = {ATTN: [2, 3, 5, 6], FFN: [4, 6, 3, 2]}
    attn = [[W.UnitPlan(True, bits_of[ATTN][i], True) for i in range(4)]]
    ffn = [[W.UnitPlan(True, bits_of[FFN][i], True) for i in range(4)]]
    work = W.build_workload("quantized_on_device", shape, 1, 96, "f32", attn, ffn, seed=19, ring_slots=2)
    blobs = {}
    for (l, kind, idx), ref_blob in work.blobs.items():
        flat = np.concatenate([m.reshape(-1) for m in make_unit_weights(shape, 19, l, kind, idx)])[None, :]
        words, cents, off, val, cnt = _run(flat, ref_blob.bits)
        n_out = int(cnt[0])
        blobs[(l, kind, idx)] = ShardBlob(bits=ref_blob.bits, codes=words[0].copy(), centroids=cents[0].copy(),
                                          outlier_off=off[0, :n_out].copy(), outlier_val=val[0, :n_out].copy())
        assert np.array_equal(words[0], ref_blob.codes)          # the generator's blob is the same quantization
    import dataclasses
    work_dev = dataclasses.replace(work, blobs=blobs)
    ref = O.run_workload(work)
    with sti.Session(work_dev) as s:
        y = run_layer(s, work_dev, 0)
    assert rel_err(y, ref) <= REL_TOL


def _guess_positions(n):
    """Offsets of the weights that the selection looks at to place its bins: 64 groups of four spread over the unit."""
    first = (n // 4) * np.arange(64, dtype=np.int64) // 64 * 4
    return (first[:, None] + np.arange(4)).reshape(-1)


@pytest.mark.parametrize("n", [1024, 24576, 100096])
@pytest.mark.parametrize("what", ["wide", "narrow", "constant", "far", "heavy", "one_sided", "large", "ordered"])
def test_units_unlike_what_their_sample_says(what, n):
    """The bins and the tails that are listed come from 256 weights: whatever they say, the result is the oracle's."""
    rng = np.random.default_rng(n)
    w = rng.normal(0, 0.02, n).astype(np.float32)
    at = _guess_positions(n)
    if what == "wide":              # outliers lie inside the listed tails: they are listed again
        w[at] *= 3
    elif what == "narrow":          # most bins are wasted on a sliver of the range, boundaries lie outside them
        w[at] *= np.float32(0.05)
    elif what == "constant":        # no scale at all
        w[at] = np.float32(0.01)
    elif what == "far":             # the mean far from zero: squares about zero cancel
        w += np.float32(3)
    elif what == "heavy":           # more tails than a warp's list in shared memory holds
        heavy = rng.random(n) < 0.06
        w[heavy] = rng.normal(0, 0.2, int(heavy.sum())).astype(np.float32)
    elif what == "one_sided":       # outliers below the mean only: every rank is shifted
        w[rng.random(n) < 0.01] = np.float32(-0.5)
    elif what == "large":           # a deviation at which a tenth of a Gaussian's weights are outliers
        w *= np.float32(300)
    elif what == "ordered":         # from no weight of a group of 128 in the tails to all of them
        w = np.sort(w * np.float32(50))
    for bits in (2, 3, 5, 6):
        _check(np.stack([w, w[::-1].copy()]), bits)
