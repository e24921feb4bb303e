"""cfi_srigl_update (device) against the oracle of Sec. 3.1's seven steps: masks and weights bit for bit, k' and the
number of live neurons equal.  Index and integer work: no tolerance."""
import numpy as np
import pytest

from oracle.srigl_update import srigl_update
from paper_2305_02299_b200 import inputs

pytestmark = pytest.mark.gpu


def _layer(out_f, in_f, k, n_abl, seed):
    L = inputs.make_layer(in_f, out_f, k, n_ablated=n_abl, seed=seed, bias=False)
    g = inputs.make_x(out_f, in_f, seed=seed + 77)
    return L.w_dense.copy(), L.mask.copy(), g


def _run_device(w, m, g, K, gamma):
    import torch
    from paper_2305_02299_b200 import binding as cfi
    wd, md, gd = torch.from_numpy(w).cuda(), torch.from_numpy(m).cuda(), torch.from_numpy(g).cuda()
    k_new, n_act = cfi.cfi_srigl_update(wd, md, gd, K, gamma)
    torch.cuda.synchronize()
    return wd.cpu().numpy(), md.cpu().numpy(), k_new, n_act


def _compare(w, m, g, K, gamma):
    gamma = float(np.float32(gamma))
    w_ref, m_ref, k_ref, abl = srigl_update(w, m, g, K, gamma)
    w_dev, m_dev, k_dev, n_dev = _run_device(w, m, g, K, gamma)
    assert k_dev == k_ref
    assert n_dev == int((m_ref.sum(1) > 0).sum())
    assert np.array_equal(m_dev, m_ref)
    assert np.array_equal(w_dev, w_ref)
    return k_ref, abl


@pytest.mark.parametrize("out_f,in_f,k,n_abl,K,gamma", [
    (24, 40, 6, 0, 30, 0.3), (24, 40, 6, 3, 60, 0.5), (16, 16, 2, 0, 8, 1.0), (64, 96, 10, 5, 200, 0.3),
    (8, 8, 8, 0, 0, 0.3), (12, 30, 3, 0, 36, 0.0), (1, 5, 2, 0, 1, 0.5), (7, 4099, 33, 1, 100, 0.25),
    (768, 3072, 307, 38, 70_000, 0.3), (3072, 768, 77, 154, 60_000, 0.3), (300, 1000, 10, 0, 2990, 0.9),
    (6, 9000, 50, 1, 120, 0.25), (5, 9001, 40, 0, 199, 0.5)])   # rows too long for the shared-memory copy of the keys
def test_matches_oracle(out_f, in_f, k, n_abl, K, gamma):
    w, m, g = _layer(out_f, in_f, k, n_abl, seed=out_f + in_f)
    _compare(w, m, g, K, gamma)


def test_matches_oracle_at_the_benchmarked_size():
    """4096 x 4096 at 80 % sparsity with K = 30 % of the active weights (about 1.0 M): the size and K the benchmark's
    mask-update leg times."""
    w, m, g = _layer(4096, 4096, 819, 0, seed=11)
    _compare(w, m, g, int(0.3 * 4096 * 819), 0.3)


def test_ablation_case_and_chained_updates():
    """A neuron with tiny weights and gradients is ablated and k' rises; a second update on the result still matches."""
    w, m, g = _layer(64, 256, 16, 0, seed=9)
    w[5] *= 1e-6
    g[5] *= 1e-6
    w[40] *= 1e-6
    g[40] *= 1e-6
    k2, abl = _compare(w, m, g, 32, 0.3)
    assert set(abl) == {5, 40} and k2 == (16 * 64) // 62
    w2, m2, _, _ = srigl_update(w, m, g, 32, float(np.float32(0.3)))
    g2 = inputs.make_x(64, 256, seed=123)
    _compare(w2, m2, g2, 50, 0.3)


@pytest.mark.parametrize("seed", range(6))
def test_many_ties(seed):
    """Quantised magnitudes and gradients: most selections are decided by position."""
    rng = np.random.default_rng(seed)
    out_f, in_f, k = int(rng.integers(3, 40)), int(rng.integers(8, 300)), 0
    k = int(rng.integers(1, min(in_f, 20)))
    w, m, g = _layer(out_f, in_f, k, int(rng.integers(0, out_f // 3 + 1)), seed=200 + seed)
    w = (np.round(w * 2) / 2 * (m == 1)).astype(np.float32)
    g = np.round(g).astype(np.float32)
    _compare(w, m, g, int(rng.integers(0, out_f * k + 1)), float(rng.choice([0.0, 0.25, 0.5, 1.0])))


@pytest.mark.parametrize("levels", [3, 4096])
def test_ties_with_and_without_room_in_the_candidate_list(levels):
    """300 x 1024 with magnitudes and gradients quantised to `levels` values.  With 3 levels a third of the layer
    equals the cut key: far more than the list of the last digit's candidates holds (4800 entries), so ties are ranked
    by the counting path; with 4096 levels the ties at the cut fit the list and the marking takes them up to a position.
    Both must equal the oracle bit for bit."""
    w, m, g = _layer(300, 1024, 100, 7, seed=77)
    q = float(levels)
    w = (np.ceil(np.abs(w) * q / 4) * 4 / q * np.sign(w) * (m == 1)).astype(np.float32)
    g = (np.round(g * q / 8) * 8 / q).astype(np.float32)
    _compare(w, m, g, 9000, 0.3)


# Both load widths (rows a multiple of four columns or not) at the ends of each number of rows per step and of each row
# length that the per-neuron step keeps in registers, with distinct keys, with many equal ones and with all gradients
# equal (then the lists of open elements overflow and further digits, of the position too, are counted first).
@pytest.mark.parametrize("values", ["distinct", "coarse", "equal"])
@pytest.mark.parametrize("out_f,in_f", [(61, 255), (700, 257), (33, 512), (20, 513), (40, 1020), (37, 1024), (19, 1028), (24, 2047), (23, 2048),
                                        (18, 2049), (17, 4095), (16, 4096), (12, 4100), (9, 4101)])
def test_row_lengths(out_f, in_f, values):
    w, m, g = _layer(out_f, in_f, max(1, in_f // 9), out_f // 10, seed=out_f * 7 + in_f)
    if values != "distinct":
        w = (np.ceil(np.abs(w) * 8) / 8 * np.sign(w) * (m == 1)).astype(np.float32)
        g = np.round(g).astype(np.float32) if values == "coarse" else np.ones_like(g)
    _compare(w, m, g, int(0.25 * m.sum()), 0.3)


def test_equal_keys_fill_the_lists():
    """512 x 2048 in whose gradients 2 % of the positions tie at the cut: more than the ties have room for (16384) and fewer
    than the lists (126976), so that the listed elements take further digits before they are decided."""
    w, m, g = _layer(512, 2048, 200, 0, seed=5)
    g = (np.abs(g) * 1e-3).astype(np.float32)
    flat = np.random.default_rng(1).permutation(512 * 2048)[:24_000]
    g.ravel()[flat] = 0.5
    _compare(w, m, g, 9_000, 0.3)


def test_unaligned_arrays():
    """Arrays that start off a 16-byte boundary take the one-column loads; what comes out is the same."""
    import torch
    from paper_2305_02299_b200 import binding as cfi
    w, m, g = _layer(37, 512, 50, 3, seed=8)
    w_ref, m_ref, k_ref, _ = srigl_update(w, m, g, 300, float(np.float32(0.3)))
    dev = []
    for a in (w, m, g):
        t = torch.empty(a.size + 1, dtype=torch.from_numpy(a).dtype, device="cuda")[1:].view(a.shape)
        t.copy_(torch.from_numpy(a))
        dev.append(t)
    k_new, _ = cfi.cfi_srigl_update(*dev, 300, 0.3)
    assert k_new == k_ref and np.array_equal(dev[1].cpu().numpy(), m_ref) and np.array_equal(dev[0].cpu().numpy(), w_ref)
    v, ix, rows = cfi.cfi_pack_device(dev[0], dev[1])
    vh, ih, rh = cfi.cfi_pack(w_ref, m_ref)
    assert np.array_equal(v.cpu().numpy(), vh) and np.array_equal(ix.cpu().numpy(), ih) and np.array_equal(rows.cpu().numpy(), rh)


@pytest.mark.parametrize("out_f,in_f", [(1, 16), (9, 512), (8, 528), (2049, 32), (5000, 1040), (3, 8192)])
def test_pack_row_and_column_chunks(out_f, in_f):
    """Rows around the eight of a block and the 2048 of a ranking round, columns around the 512 of a warp's step."""
    import torch
    from paper_2305_02299_b200 import binding as cfi
    w, m, _ = _layer(out_f, in_f, max(1, in_f // 11), out_f // 3, seed=out_f)
    v, ix, rows = cfi.cfi_pack_device(torch.from_numpy(w).cuda(), torch.from_numpy(m).cuda())
    vh, ih, rh = cfi.cfi_pack(w, m)
    assert np.array_equal(v.cpu().numpy(), vh) and np.array_equal(ix.cpu().numpy(), ih) and np.array_equal(rows.cpu().numpy(), rh)


def test_workspace_and_argument_checks():
    import ctypes
    import torch
    from paper_2305_02299_b200 import binding as cfi
    w = torch.zeros((4, 8), device="cuda")
    m = torch.zeros((4, 8), device="cuda", dtype=torch.uint8)
    with pytest.raises(cfi.CfiError) as e:
        cfi.cfi_srigl_update(w, m, w, 1, -0.5)
    assert e.value.status == 2
    k_new, n_act = cfi.cfi_srigl_update(w, m, w, 3, 0.3)      # a layer with no active weight stays empty
    assert (k_new, n_act) == (0, 0) and int(m.sum()) == 0


def test_update_then_pack_create_forward():
    """The update's output is a constant-fan-in mask that the forward path accepts as is: cfi_pack (mask given, so grown
    weights with value 0 count), cfi_create, cfi_forward, against the oracle forward on the oracle's updated layer."""
    import torch
    import oracle
    from paper_2305_02299_b200 import binding as cfi
    from parity import TOL, scaled_error
    w, m, g = _layer(384, 512, 51, 20, seed=31)
    w[7] *= 1e-6
    g[7] *= 1e-6
    gamma = float(np.float32(0.3))
    w_ref, m_ref, k_ref, _ = srigl_update(w, m, g, 3000, gamma)
    w_dev, m_dev, k_dev, n_dev = _run_device(w, m, g, 3000, gamma)
    assert k_dev == k_ref and np.array_equal(m_dev, m_ref)
    v, ix, rows = cfi.cfi_pack(w_dev, m_dev)
    assert v.shape == (n_dev, k_dev) and np.any(v == 0.0)            # freshly grown weights are kept entries of value 0
    bias = inputs.make_layer(512, 384, 51, seed=32).bias
    x = inputs.make_x(40, 512, seed=33)
    vr, ir, rr = oracle.pack(w_ref, m_ref)
    y_ref, S = oracle.forward(vr, ir, rr, bias, 512, 384, x, want_scale=True)
    layer = cfi.cfi_create(v, ix, rows, bias, 512, 384)
    y = torch.empty((40, 384), device="cuda")
    cfi.cfi_forward(layer, torch.from_numpy(x).cuda(), y, 40)
    torch.cuda.synchronize()
    layer.close()
    assert scaled_error(y.cpu().numpy(), y_ref, S) <= TOL["f32"]


@pytest.mark.parametrize("out_f,in_f,k,n_abl", [(24, 40, 6, 0), (300, 1000, 10, 37), (7, 4099, 33, 1), (768, 3072, 307, 38), (5, 9, 9, 0)])
def test_pack_device_equals_host_pack(out_f, in_f, k, n_abl):
    """cfi_pack_device on device-resident w and mask gives exactly cfi_pack's arrays (and the oracle's)."""
    import torch
    import oracle
    from paper_2305_02299_b200 import binding as cfi
    w, m, _ = _layer(out_f, in_f, k, n_abl, seed=out_f)
    zr, zc = np.nonzero(m == 1)
    w[zr[::7], zc[::7]] = 0.0                                    # kept entries of value 0 still count (the mask decides)
    v, ix, rows = cfi.cfi_pack_device(torch.from_numpy(w).cuda(), torch.from_numpy(m).cuda())
    vh, ih, rh = cfi.cfi_pack(w, m)
    vo, io, ro = oracle.pack(w, m)
    assert np.array_equal(v.cpu().numpy(), vh) and np.array_equal(ix.cpu().numpy(), ih) and np.array_equal(rows.cpu().numpy(), rh)
    assert np.array_equal(vh, vo) and np.array_equal(ih, io) and np.array_equal(rh, ro)


@pytest.mark.parametrize("in_f", [1, 31, 511, 512, 513, 1025, 9001])
def test_pack_device_rows_without_wide_loads(in_f):
    """Rows whose mask cannot be read 16 bytes at a time (odd lengths; 512 from an odd address): around the 512 columns of a step."""
    import torch
    from paper_2305_02299_b200 import binding as cfi
    w, m, _ = _layer(9, in_f, max(1, in_f // 5), 1, seed=in_f)
    m_d = torch.empty(m.size + 1, dtype=torch.uint8, device="cuda")[1:].view(m.shape)
    m_d.copy_(torch.from_numpy(m))
    v, ix, rows = cfi.cfi_pack_device(torch.from_numpy(w).cuda(), m_d)
    vh, ih, rh = cfi.cfi_pack(w, m)
    assert np.array_equal(v.cpu().numpy(), vh) and np.array_equal(ix.cpu().numpy(), ih) and np.array_equal(rows.cpu().numpy(), rh)


def test_pack_device_errors_and_empty():
    import torch
    from paper_2305_02299_b200 import binding as cfi
    w, m, _ = _layer(10, 20, 4, 2, seed=3)
    m2 = m.copy()
    row = int(np.nonzero(m2.sum(1))[0][0])
    m2[row, np.nonzero(m2[row])[0][0]] = 0                        # one row keeps one entry fewer
    with pytest.raises(cfi.CfiError) as e:
        cfi.cfi_pack_device(torch.from_numpy(w).cuda(), torch.from_numpy(m2).cuda())
    assert e.value.status == 3
    v, ix, rows = cfi.cfi_pack_device(torch.zeros((4, 8), device="cuda"), torch.zeros((4, 8), device="cuda", dtype=torch.uint8))
    assert v.shape == (0, 0) and rows.shape == (0,)


def test_pack_device_fill_writes_only_what_was_counted():
    """The filling step takes the counts of the size query; with other counts it writes nothing and says so."""
    import ctypes
    import torch
    from paper_2305_02299_b200 import binding as cfi
    out_f, in_f, k = 40, 96, 7
    L = inputs.make_layer(in_f, out_f, k, n_ablated=3, seed=5)
    w, m = torch.from_numpy(L.w_dense).cuda(), torch.from_numpy(L.mask).cuda()
    ws = torch.empty(8 * out_f + 512, dtype=torch.uint8, device="cuda")
    base = (ws.data_ptr() + 255) & ~255
    kk, na = ctypes.c_int32(0), ctypes.c_int32(0)
    head = (w.data_ptr(), m.data_ptr(), out_f, in_f, base, 8 * out_f + 256)
    assert cfi._lib.cfi_pack_device(*head, ctypes.byref(kk), ctypes.byref(na), None, None, None, None) == 0
    assert (kk.value, na.value) == (k, out_f - 3)
    v = torch.full((out_f, in_f), -1.0, device="cuda")
    ix, rows = torch.full((out_f, in_f), -1, dtype=torch.int32, device="cuda"), torch.full((out_f,), -1, dtype=torch.int32, device="cuda")
    arrays = (v.data_ptr(), ix.data_ptr(), rows.data_ptr(), None)
    for wrong in ((k - 1, out_f - 3), (k, out_f - 4), (k + 1, out_f - 3)):
        assert cfi._lib.cfi_pack_device_fill(*head, *wrong, *arrays) == 2
        assert bool((v == -1).all()) and bool((ix == -1).all()) and bool((rows == -1).all())
    assert cfi._lib.cfi_pack_device_fill(*head, k, out_f - 3, *arrays) == 0
    hv, hix, hrows = cfi.cfi_pack(L.w_dense, L.mask)
    n = hv.size
    assert np.array_equal(v.flatten()[:n].cpu().numpy(), hv.ravel()) and np.array_equal(ix.flatten()[:n].cpu().numpy(), hix.ravel())
    assert np.array_equal(rows[:out_f - 3].cpu().numpy(), hrows) and bool((v.flatten()[n:] == -1).all())


@pytest.mark.parametrize("in_f", [96, 99])
@pytest.mark.parametrize("change", ["fewer", "more", "moved", "empty_row"])
def test_pack_device_fill_reports_a_mask_that_changed_since_the_query(in_f, change):
    """A mask that another stream changes between the two steps: never a success with arrays that were not filled."""
    import ctypes
    import torch
    from paper_2305_02299_b200 import binding as cfi
    out_f, k = 40, 7
    L = inputs.make_layer(in_f, out_f, k, n_ablated=3, seed=6)
    w, m = torch.from_numpy(L.w_dense).cuda(), torch.from_numpy(L.mask).cuda()
    ws = torch.empty(8 * out_f + 512, dtype=torch.uint8, device="cuda")
    base = (ws.data_ptr() + 255) & ~255
    kk, na = ctypes.c_int32(0), ctypes.c_int32(0)
    head = (w.data_ptr(), m.data_ptr(), out_f, in_f, base, 8 * out_f + 256)
    query = lambda: cfi._lib.cfi_pack_device(*head, ctypes.byref(kk), ctypes.byref(na), None, None, None, None)
    assert query() == 0 and (kk.value, na.value) == (k, out_f - 3)
    counts = m.sum(1)
    row, other, empty = (int(counts.nonzero()[0]), int(counts.nonzero()[1]), int((counts == 0).nonzero()[0]))
    if change != "more":
        m[row, m[row].nonzero()[0]] = 0
    if change != "fewer":
        to = {"more": row, "moved": other, "empty_row": empty}[change]
        m[to, (m[to] == 0).nonzero()[-1]] = 1
    guard = 64
    v = torch.full(((out_f - 3) * k + guard,), -1.0, device="cuda")
    ix, rows = torch.full(v.shape, -1, dtype=torch.int32, device="cuda"), torch.full((out_f - 3 + guard,), -1, dtype=torch.int32, device="cuda")
    assert cfi._lib.cfi_pack_device_fill(*head, k, out_f - 3, v.data_ptr(), ix.data_ptr(), rows.data_ptr(), None) == 3
    assert bool((v[-guard:] == -1).all()) and bool((ix[-guard:] == -1).all()) and bool((rows[-guard:] == -1).all())
    assert query() == 3                                           # as the rows are counted anew


@pytest.mark.parametrize("in_f", [132, 768, 1030, 4096])
@pytest.mark.parametrize("kind", ["wide", "equal", "inf"])
def test_regrowth_where_the_fine_histogram_cannot_part_the_gradients(in_f, kind):
    """Gradients over 60 binades, nearly all equal, and with infinities: the first histogram of a row's selection puts
    too many into one bin, and the leading bits decide."""
    rng = np.random.default_rng(in_f)
    w, m, _ = _layer(24, in_f, max(2, in_f // 12), 2, seed=in_f)
    g = rng.standard_normal(w.shape).astype(np.float32)
    if kind == "wide":
        g = (g * np.exp2(rng.uniform(-60, 0, w.shape))).astype(np.float32)
        g[:, 0] = 1.0
    elif kind == "equal":
        g = np.where(rng.random(w.shape) < 0.97, np.float32(0.25), g).astype(np.float32)
    else:
        g[:, 1] = np.inf
    _compare(w, m, g, int(0.3 * m.sum()), 0.3)
