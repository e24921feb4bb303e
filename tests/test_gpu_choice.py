"""The automatic kernel choice (cfi_forward) against every explicit variant that can run the shape: on the named workloads
the kernel it picks must be within 15 % (plus 0.3 us of timing noise) of the fastest one, on a grid of widths, sparsities,
batches, types and layouts within what the models of the choice leave open.  Times are CUDA events around replays of a CUDA
graph of 50 launches on one layer, 200 launches per figure."""
import numpy as np
import pytest

from paper_2305_02299_b200 import inputs

pytestmark = pytest.mark.gpu
W = inputs.workloads()
SHAPES = [("c1", ["c1", "c2"]), ("c3_b1", ["c3_b1", "c3_b64", "c3_b256"])] + \
         [(f"c4_s{sp}_b1", [f"c4_s{sp}_b{b}" for b in (1, 16, 256)]) for sp in (80, 90, 95, 99)]


def _time(cfi, torch, layer, x, y, batch, variant):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        for _ in range(3):
            cfi.cfi_forward_variant(layer, x, y, batch, variant=variant)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(50):
                cfi.cfi_forward_variant(layer, x, y, batch, variant=variant)
        g.replay()
        s.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(s)
        for _ in range(4):
            g.replay()
        b.record(s)
        b.synchronize()
    return a.elapsed_time(b) * 1e3 / 200


@pytest.mark.parametrize("base,names", SHAPES, ids=[b for b, _ in SHAPES])
def test_auto_is_close_to_the_best_variant(base, names):
    import torch
    from paper_2305_02299_b200 import binding as cfi
    L = W[base].layer()
    v, ix, rows = cfi.cfi_pack(L.w_dense, L.mask)
    layer = cfi.cfi_create(v, ix, rows, L.bias, W[base].in_features, W[base].out_features)
    report = {}
    for name in names:
        w = W[name]
        x = torch.from_numpy(w.x()).cuda()
        y = torch.empty((w.batch, w.out_features), device="cuda")
        times = {}
        for variant in ("splitk", "batch", "slab", "dense_tc"):
            try:
                times[variant] = _time(cfi, torch, layer, x, y, w.batch, variant)
            except cfi.CfiError as e:
                assert e.status == 2                            # the variant cannot run this shape
        t_auto = _time(cfi, torch, layer, x, y, w.batch, "auto")
        best = min(times.values())
        report[name] = (t_auto, times)
        assert t_auto <= 1.15 * best + 0.3, (name, t_auto, times)
    layer.close()


# Batches on both sides of every line of the choice above eight rows; fp32 and bf16; with the dense copy and without.
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("layouts", [7, 3])
@pytest.mark.parametrize("in_f,out_f", [(768, 3072), (3072, 768), (512, 2048), (2048, 2048)])
def test_auto_is_close_to_the_best_variant_on_a_grid(dtype, layouts, in_f, out_f):
    """The models are within 20 to 25 % of the times, so of two kernels the one that looks faster takes at most
    1.25 / 0.78 = 1.6 times as long as the other.  fp32: the tensor cores' split products are less exact and taken for a large gain only, so where
    the choice is a kernel with fp32 sums it is compared with those."""
    import torch
    from paper_2305_02299_b200 import binding as cfi
    from parity import torch_dtype
    slow, report = [], {}
    for k in (max(1, in_f // 100), in_f // 20, in_f // 10):
        L = inputs.make_layer(in_f, out_f, k, seed=k)
        layer = cfi.cfi_create(*cfi.cfi_pack(L.w_dense, L.mask), L.bias, in_f, out_f, dtype=dtype, layouts=layouts)
        for batch in (9, 16, 32, 64, 128, 256, 320):
            x = torch.from_numpy(inputs.make_x(batch, in_f, seed=batch)).cuda().to(torch_dtype(dtype))
            y = torch.empty((batch, out_f), device="cuda", dtype=x.dtype)
            times = {}
            for variant in ("splitk", "batch", "slab", "dense_tc"):
                if variant == "dense_tc" and dtype == "f32" and cfi.cfi_choose_variant(layer, batch) != 4:
                    continue
                if (variant, dtype) == ("slab", "bf16") or batch > {"splitk": 256, "slab": 64}.get(variant, batch):
                    continue                                    # no candidate there
                try:
                    times[variant] = _time(cfi, torch, layer, x, y, batch, variant)
                except cfi.CfiError as e:
                    assert e.status == 2
            t_auto = _time(cfi, torch, layer, x, y, batch, "auto")
            report[(k, batch)] = t_auto / min(times.values())
            if t_auto > 1.6 * min(times.values()) + 0.3:
                slow.append((k, batch, t_auto, times))
        layer.close()
    print(sorted(report.values())[-3:])
    assert not slow, slow


@pytest.mark.parametrize("in_f,out_f,k,batch", [(3072, 768, 61, 1576), (3072, 768, 92, 1576), (1536, 1536, 46, 2048), (4096, 4096, 82, 2048),
                                                 (4096, 4096, 123, 512), (768, 3072, 23, 600), (1024, 4096, 10, 320), (256, 256, 3, 2500)])
def test_calls_below_the_line_keep_fp32_sums(in_f, out_f, k, batch):
    """Sparse fp32 calls for which the gather kernel is not far behind the tensor cores.  fp32 sums of up to 123 terms, one after
    another, are within 123 * 2^-24 = 7e-6 of each term's size at worst and sqrt(123) * 2^-24 / 2 = 3.3e-7 where roundings are
    independent; the split products alone leave at least 3.6e-7 (2-norm, measured at k = 3)."""
    import torch
    from paper_2305_02299_b200 import binding as cfi
    L = inputs.make_layer(in_f, out_f, k, seed=k)
    layer = cfi.cfi_create(*cfi.cfi_pack(L.w_dense, L.mask), L.bias, in_f, out_f)
    x = torch.from_numpy(inputs.make_x(batch, in_f, seed=1)).cuda()
    y = torch.empty((batch, out_f), device="cuda")
    cfi.cfi_forward(layer, x, y, batch)
    ref = x.double() @ torch.from_numpy(L.w_dense).cuda().double().t() + torch.from_numpy(L.bias).cuda().double()
    err = float((y.double() - ref).norm() / ref.norm())
    variant = cfi.cfi_choose_variant(layer, batch)
    layer.close()
    assert err <= 3.3e-7 and variant != 4, (err, variant)
