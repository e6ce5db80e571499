"""GPU parity: the CUDA path, through the C boundary, against the fp64 CPU oracle
on the same seeded inputs.

Tolerances (stated by the benchmark definition):
  * routing index: bit-exact, except rows whose k-th and (k+1)-th oracle
    scores lie within 1e-3 relative of each other (counted and reported);
    attention is always compared using the GPU's own index
  * O: bf16 I/O max-abs <= 2e-2 and mean-abs <= 2e-3; fp32 I/O max-abs <= 1e-5
  * gradients: max-abs <= 5e-2
"""
import numpy as np
import pytest

from oracle import bra_oracle as orc
from paper_2303_08810_b200 import synthetic
from paper_2303_08810_b200.synthetic import BraConfig, CONFIGS

pytestmark = pytest.mark.gpu

TOL = {"bf16": dict(max=2e-2, mean=2e-3), "f32": dict(max=1e-5, mean=1e-6)}
GRAD_MAX = 5e-2
# d_lce_w / d_lce_b are sums over all B*H*W positions of products that are exact in fp32; with
# fp32 partial sums the rounding error is about sqrt(n) * 2^-24 of the running sum (n <= 2e5 here)
LCE_GRAD_REL = 1e-4


@pytest.fixture(scope="module")
def bra():
    import paper_2303_08810_b200 as pkg
    from paper_2303_08810_b200 import build
    build.build_library()
    pkg.load_library()
    return pkg


def to_dev(x, cfg):
    import torch
    out = {}
    for k, v in x.items():
        t = torch.from_numpy(np.ascontiguousarray(v)).cuda()
        if k != "w" and cfg.dtype == "bf16":
            t = t.to(torch.bfloat16)
        out[k] = t
    return out


def problem_of(bra, cfg, impl=0, **kw):
    return bra.make_problem(cfg.B, cfg.H, cfg.W, cfg.C, cfg.heads, cfg.S, cfg.topk, cfg.dtype,
                            impl=impl, **kw)


def f64(t):
    return t.detach().float().cpu().numpy().astype(np.float64)


def check_index(idx_gpu, idx_ref, gap, topk, R, A=None):
    """Rows whose k-th and (k+1)-th oracle scores are clearly apart must select
    exactly the oracle's regions.  The order inside a row must match too, except
    between neighbours whose oracle scores lie within 1e-3 relative (fp32 and
    fp64 may rank those either way).  Near-tie rows must still be valid."""
    clear = gap > 1e-3
    assert np.array_equal(np.sort(idx_gpu[clear], axis=-1), np.sort(idx_ref[clear], axis=-1))
    assert idx_gpu.min() >= 0 and idx_gpu.max() < R
    if topk > 1:
        assert (np.diff(np.sort(idx_gpu, axis=-1), axis=-1) > 0).all()
    order_diff = (idx_gpu != idx_ref).any(axis=-1) & clear
    if A is not None and order_diff.any():
        top = np.take_along_axis(A, idx_ref.astype(np.int64), axis=-1)     # descending scores
        rel = (top[..., :-1] - top[..., 1:]) / np.maximum(
            np.maximum(np.abs(top[..., :-1]), np.abs(top[..., 1:])), 1e-30)
        # a row may differ in order only where two neighbouring scores nearly tie
        assert (rel[order_diff].min(axis=-1) <= 1e-3).all()
        mism = idx_gpu[order_diff] != idx_ref[order_diff]
        tie = np.zeros_like(mism)
        close = rel[order_diff] <= 1e-3
        tie[:, :-1] |= close
        tie[:, 1:] |= close
        assert not (mism & ~tie).any()
    elif A is None:
        assert not order_diff.any()
    near = int((~clear).sum())
    flips = int((np.sort(idx_gpu[~clear], -1) != np.sort(idx_ref[~clear], -1)).any(axis=-1).sum()) if near else 0
    return near, flips


def oracle_affinity(x, cfg, shared=False):
    return orc.region_affinity(orc.region_means(x["Q"], cfg.S), orc.region_means(x["K"], cfg.S),
                               cfg.heads, shared)


def check_O(O_gpu, O_ref, dtype):
    err = np.abs(O_gpu - O_ref)
    assert err.max() <= TOL[dtype]["max"], f"max-abs {err.max():.3e}"
    assert err.mean() <= TOL[dtype]["mean"], f"mean-abs {err.mean():.3e}"


# ------------------------------------------------------------------ routing
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
def test_route_matches_oracle(bra, n):
    cfg = CONFIGS[n]
    x = synthetic.make_inputs(cfg, seed=1000 + n)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    qm, km, idx = bra.bra_route(p, t["Q"], t["K"], ws=ws)
    assert bra.last_launch_count() >= 2
    Qr, Kr, idx_ref, gap = orc.bra_route(x["Q"], x["K"], cfg.heads, cfg.S, cfg.topk)
    np.testing.assert_allclose(f64(qm), Qr, rtol=0, atol=2e-6)
    np.testing.assert_allclose(f64(km), Kr, rtol=0, atol=2e-6)
    near, flips = check_index(idx.cpu().numpy(), idx_ref, gap, cfg.topk, cfg.R, oracle_affinity(x, cfg))
    print(f"config {n}: {near} near-tie rows of {gap.size}, {flips} differ")
    assert near < 0.02 * gap.size + 5
    assert bra.bra_device_status(ws) == 0


def test_route_shared_and_odd_shapes(bra):
    import torch
    cases = [
        (BraConfig("shared", 2, 12, 20, 48, 3, 4, 5, "f32"), True),
        (BraConfig("k=R", 1, 9, 6, 32, 2, 3, 9, "bf16"), False),
        (BraConfig("S=1", 2, 5, 7, 16, 1, 1, 1, "f32"), False),
        (BraConfig("S=16", 1, 32, 32, 32, 1, 16, 12, "bf16"), False),
        (BraConfig("R=100", 1, 20, 30, 64, 2, 10, 7, "f32"), True),
        # many winners per row and many (image, head) pairs: the thread-per-row routing kernel
        (BraConfig("k=12-many-pairs", 130, 8, 8, 64, 2, 4, 12, "bf16"), False),
        (BraConfig("k=9-shared-wide-rows", 256, 6, 6, 48, 3, 3, 9, "bf16"), True),
        # small square regions: pooled by one CTA per row of regions
        (BraConfig("1x1-regions", 3, 5, 5, 64, 2, 5, 7, "bf16"), False),
        (BraConfig("2x2-regions-f32", 2, 8, 8, 32, 1, 4, 3, "f32"), False),
        (BraConfig("4x4-regions-wide-rows", 2, 12, 12, 512, 16, 3, 2, "bf16"), True),
        # a few winners per row, many pairs, 32 channels per routing head: one CTA per (image, head)
        (BraConfig("cta-per-pair", 130, 14, 14, 64, 2, 7, 5, "bf16"), False),
        (BraConfig("cta-per-pair-k=R", 160, 4, 6, 64, 2, 2, 4, "f32"), False),
        (BraConfig("cta-per-pair-shared", 300, 6, 6, 32, 1, 3, 4, "f32"), True),
    ]
    for cfg, shared in cases:
        x = synthetic.make_inputs(cfg, seed=77)
        t = to_dev(x, cfg)
        p = problem_of(bra, cfg, shared_routing=shared)
        qm, km, idx = bra.bra_route(p, t["Q"], t["K"])
        Qr, Kr, idx_ref, gap = orc.bra_route(x["Q"], x["K"], cfg.heads, cfg.S, cfg.topk, shared)
        assert idx.shape == idx_ref.shape
        np.testing.assert_allclose(f64(qm), Qr, rtol=0, atol=2e-6)
        check_index(idx.cpu().numpy(), idx_ref, gap, cfg.topk, cfg.R, oracle_affinity(x, cfg, shared))


def test_route_exact_ties_go_to_lower_region(bra):
    """Identical K in every region: all affinities of a row are equal."""
    import torch
    cfg = BraConfig("ties", 1, 8, 8, 32, 1, 4, 3, "f32")
    Q = torch.randn(1, 8, 8, 32, device="cuda")
    K = torch.ones(1, 8, 8, 32, device="cuda")
    p = problem_of(bra, cfg)
    _, _, idx = bra.bra_route(p, Q, K)
    assert (idx.cpu().numpy() == np.array([0, 1, 2])).all()
    # +0 / -0 affinities are the same score
    Q0 = torch.zeros_like(Q)
    K0 = torch.randn_like(K)
    _, _, idx0 = bra.bra_route(p, Q0, K0)
    assert (idx0.cpu().numpy() == np.array([0, 1, 2])).all()
    # the same through the thread-per-row kernel (k > 8, many image-head pairs)
    cfg = BraConfig("ties-rows", 256, 8, 8, 32, 1, 4, 10, "f32")
    p = problem_of(bra, cfg)
    Q = torch.randn(256, 8, 8, 32, device="cuda")
    _, _, idx = bra.bra_route(p, Q, torch.ones_like(Q))
    assert (idx.cpu().numpy() == np.arange(10)).all()
    # and through the kernel with one CTA per (image, head) (2 <= k <= 8, at least 256 pairs, 32 channels per head)
    cfg = BraConfig("ties-cta-per-pair", 256, 8, 8, 32, 1, 4, 5, "f32")
    p = problem_of(bra, cfg)
    _, _, idx = bra.bra_route(p, Q, torch.ones_like(Q))
    assert (idx.cpu().numpy() == np.arange(5)).all()
    _, _, idx0 = bra.bra_route(p, torch.zeros_like(Q), torch.randn_like(Q))
    assert (idx0.cpu().numpy() == np.arange(5)).all()


# ------------------------------------------------------------------ attention
IMPLS = {"simt": 1, "mma": 2, "tc": 3, "img": 4, "auto": 0}


def run_attend_case(bra, cfg, impl, seed, shared=False, lce=True, bias=False, scale=0.0,
                    index=None, clustered=False, mutate=None):
    """One bra_attend call of kernel family `impl` against the oracle.  A family that is
    named explicitly must take the shape: BRA_ERR_UNSUPPORTED fails the test (the cases
    where a family rightly refuses a shape are asserted in
    test_kernel_families_refuse_only_what_they_should)."""
    import torch
    x = synthetic.make_inputs(cfg, seed=seed, clustered=clustered)
    if mutate is not None:
        mutate(x)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg, impl=IMPLS[impl], shared_routing=shared, lce=lce, scale=scale)
    ws = bra.workspace(p)
    if index is None:
        _, _, idx = bra.bra_route(p, t["Q"], t["K"], ws=ws)
    else:
        idx = torch.from_numpy(index).cuda()
    b = None
    b_np = None
    if bias:
        b_np = np.linspace(-0.5, 0.5, cfg.C).astype(np.float32)
        b = torch.from_numpy(b_np).cuda()
    O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, t["w"] if lce else None, b, ws=ws)
    assert bra.last_launch_count() >= 1
    assert bra.bra_device_status(ws) == 0
    O_ref, lse_ref = orc.bra_attend(x["Q"], x["K"], x["V"], idx.cpu().numpy(),
                                    x["w"] if lce else None, cfg.heads, cfg.S,
                                    scale if scale > 0 else None, b_np)
    check_O(f64(O), O_ref, cfg.dtype)
    np.testing.assert_allclose(f64(lse), lse_ref, rtol=0, atol=1e-5 if cfg.dtype == "f32" else 2e-3)
    return O


# which benchmark configs each kernel family takes: fp32 (config 1) only the CUDA-core kernel;
# tcgen05 wants 8 x 8 or 16-wide regions (configs 2, 4); the image-resident kernel wants a head's
# K and V of a whole image in shared memory (configs 3, 5)
TAKES = {"simt": {1, 2, 3, 4, 5}, "mma": {2, 3, 4, 5}, "tc": {2, 4}, "img": {3, 5}, "auto": {1, 2, 3, 4, 5}}


@pytest.mark.parametrize("impl,n", [(i, n) for i in TAKES for n in sorted(TAKES[i])])
def test_attend_matches_oracle_on_benchmark_configs(bra, n, impl):
    run_attend_case(bra, CONFIGS[n], impl, seed=1000 + n)


@pytest.mark.parametrize("impl,n", [(i, n) for i in TAKES for n in range(1, 6) if n not in TAKES[i]])
def test_kernel_families_refuse_only_what_they_should(bra, n, impl):
    """A family asked for a shape outside its range answers BRA_ERR_UNSUPPORTED on the host,
    nothing launched; every other (family, config) pair is a parity case above."""
    import torch
    cfg = CONFIGS[n]
    x = synthetic.make_inputs(synthetic.with_batch(cfg, 1), seed=3)
    small = synthetic.with_batch(cfg, 1)
    t = to_dev(x, small)
    p = problem_of(bra, small, impl=IMPLS[impl])
    idx = torch.zeros(1, small.heads, small.R, small.topk, dtype=torch.int32, device="cuda")
    with pytest.raises(bra.BraError) as e:
        bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, t["w"])
    assert e.value.code == 7
    assert bra.last_launch_count() == 0


EDGE = [
    BraConfig("S1-n_r=90", 2, 9, 10, 32, 1, 1, 1, "f32"),
    BraConfig("rect-regions", 2, 12, 20, 64, 2, 4, 3, "bf16"),
    BraConfig("n_r=15", 1, 9, 15, 32, 2, 3, 2, "f32"),
    BraConfig("full-k=R", 1, 14, 14, 64, 2, 7, 49, "bf16"),
    BraConfig("S=1", 2, 6, 6, 32, 1, 1, 1, "bf16"),
    BraConfig("one-token-regions", 1, 4, 4, 32, 1, 4, 5, "f32"),
    BraConfig("d=64", 1, 16, 16, 128, 2, 4, 3, "bf16"),
    BraConfig("d=16", 1, 16, 16, 32, 2, 2, 2, "f32"),
    BraConfig("d=128", 1, 8, 8, 128, 1, 2, 2, "bf16"),
    BraConfig("vit-adapt-small", 1, 32, 32, 128, 2, 8, 12, "bf16"),
]


@pytest.mark.parametrize("impl", ["simt", "auto"])
@pytest.mark.parametrize("cfg", EDGE, ids=[c.name for c in EDGE])
def test_attend_edge_shapes(bra, cfg, impl):
    run_attend_case(bra, cfg, impl, seed=5)


# 8 x 8-token regions with head dim 32: the shapes of the persistent tensor-core kernel
TC_CASES = [
    BraConfig("tc-k3-two-head-pairs", 2, 32, 32, 128, 4, 4, 3, "bf16"),
    BraConfig("tc-k16-every-region", 1, 32, 32, 64, 2, 4, 16, "bf16"),
    BraConfig("tc-several-tiles-per-cta", 5, 56, 56, 64, 2, 7, 2, "bf16"),
    BraConfig("tc-single-region", 1, 8, 8, 64, 2, 1, 1, "bf16"),
    BraConfig("tc-k5-S8", 1, 64, 64, 64, 2, 8, 5, "bf16"),
]


@pytest.mark.parametrize("cfg", TC_CASES, ids=[c.name for c in TC_CASES])
def test_attend_tc_shapes(bra, cfg):
    run_attend_case(bra, cfg, "tc", seed=21)


# head dim 32, bf16, every region shape: the warp-level tensor-core kernel
MMA_CASES = TC_CASES + [
    BraConfig("mma-2x2-regions-k16", 2, 14, 14, 256, 8, 7, 16, "bf16"),
    BraConfig("mma-4x4-regions-k4", 2, 28, 28, 128, 4, 7, 4, "bf16"),
    BraConfig("mma-16x16-regions-two-chunks", 1, 32, 32, 64, 2, 2, 3, "bf16"),
    BraConfig("mma-3x5-regions-odd-width", 2, 12, 20, 64, 2, 4, 3, "bf16"),
    BraConfig("mma-last-block-partial", 1, 14, 14, 64, 2, 7, 49, "bf16"),
    BraConfig("mma-6x6-region-S1", 2, 6, 6, 32, 1, 1, 1, "bf16"),
    BraConfig("mma-7x7-regions-k3", 1, 56, 56, 64, 2, 8, 3, "bf16"),
    BraConfig("mma-one-token-regions", 1, 4, 4, 32, 1, 4, 5, "bf16"),
    BraConfig("mma-wide-regions-3-chunks", 1, 18, 64, 32, 1, 1, 1, "bf16"),
    # head dim 64: two 32-channel planes per head
    BraConfig("mma-d64-vit-adaptation", 1, 32, 32, 768, 12, 8, 12, "bf16"),
    BraConfig("mma-d64-8x8-regions-k2", 2, 16, 16, 128, 2, 2, 2, "bf16"),
    BraConfig("mma-d64-3x5-regions", 1, 12, 20, 192, 3, 4, 3, "bf16"),
    BraConfig("mma-d64-last-block-partial", 1, 14, 14, 64, 1, 7, 49, "bf16"),
]


@pytest.mark.parametrize("cfg", MMA_CASES, ids=[c.name for c in MMA_CASES])
def test_attend_mma_shapes(bra, cfg):
    run_attend_case(bra, cfg, "mma", seed=22)


def test_attend_mma_options(bra):
    cfg = BraConfig("mma-opts", 2, 16, 16, 64, 2, 4, 3, "bf16")
    run_attend_case(bra, cfg, "mma", seed=6, lce=False)
    run_attend_case(bra, cfg, "mma", seed=6, bias=True)
    run_attend_case(bra, cfg, "mma", seed=6, scale=0.5)
    run_attend_case(bra, cfg, "mma", seed=6, shared=True)
    rng = np.random.default_rng(3)
    idx = rng.integers(0, cfg.R, size=(cfg.B, cfg.heads, cfg.R, cfg.topk)).astype(np.int32)
    idx[0, 0, 0] = [5, 5, 5]
    run_attend_case(bra, cfg, "mma", seed=6, index=idx)


# head dim 32, bf16, maps small enough that one (image, head) of K and V fits in shared memory
IMG_CASES = [c for c in MMA_CASES if c.H * c.W <= 1500 and c.C // c.heads == 32] + [
    BraConfig("img-tail-tile-n_r=24", 2, 12, 16, 64, 2, 2, 3, "bf16"),
    BraConfig("img-5x5-regions-odd", 1, 15, 15, 32, 1, 3, 4, "bf16"),
    BraConfig("img-k-many-blocks", 1, 16, 16, 64, 2, 4, 16, "bf16"),
    BraConfig("img-many-images", 40, 14, 14, 64, 2, 7, 5, "bf16"),
]


@pytest.mark.parametrize("cfg", IMG_CASES, ids=[c.name for c in IMG_CASES])
def test_attend_img_shapes(bra, cfg):
    run_attend_case(bra, cfg, "img", seed=24)


def test_attend_img_options(bra):
    cfg = BraConfig("img-opts", 2, 16, 16, 64, 2, 4, 3, "bf16")
    run_attend_case(bra, cfg, "img", seed=6, lce=False)
    run_attend_case(bra, cfg, "img", seed=6, bias=True)
    run_attend_case(bra, cfg, "img", seed=6, scale=0.5)
    run_attend_case(bra, cfg, "img", seed=6, shared=True)
    run_attend_case(bra, cfg, "img", seed=6, clustered=True)
    rng = np.random.default_rng(3)
    idx = rng.integers(0, cfg.R, size=(cfg.B, cfg.heads, cfg.R, cfg.topk)).astype(np.int32)
    idx[0, 0, 0] = [5, 5, 5]
    run_attend_case(bra, cfg, "img", seed=6, index=idx)


# head dim 32, regions 16 tokens wide and a multiple of 8 high: the tcgen05 kernel for large regions
TC_WIDE_CASES = [
    BraConfig("wide-16x16-k4", 2, 32, 32, 64, 2, 2, 4, "bf16"),
    BraConfig("wide-16x16-k1-three-heads", 1, 32, 32, 96, 3, 2, 1, "bf16"),
    BraConfig("wide-8x16-regions-k3", 1, 16, 32, 32, 1, 2, 3, "bf16"),
    BraConfig("wide-24x16-regions", 1, 48, 32, 64, 2, 2, 2, "bf16"),
    BraConfig("wide-many-tiles", 3, 64, 64, 64, 2, 4, 5, "bf16"),
]


@pytest.mark.parametrize("cfg", TC_WIDE_CASES, ids=[c.name for c in TC_WIDE_CASES])
def test_attend_tc_wide_shapes(bra, cfg):
    run_attend_case(bra, cfg, "tc", seed=23)


def test_attend_tc_wide_options(bra):
    cfg = BraConfig("wide-opts", 1, 32, 32, 64, 2, 2, 2, "bf16")
    run_attend_case(bra, cfg, "tc", seed=6, lce=False)
    run_attend_case(bra, cfg, "tc", seed=6, bias=True)
    run_attend_case(bra, cfg, "tc", seed=6, scale=0.5)
    run_attend_case(bra, cfg, "tc", seed=6, shared=True)
    idx = np.array([[[[3, 3], [0, 1], [2, 0], [1, 1]]] * 2], dtype=np.int32)
    run_attend_case(bra, cfg, "tc", seed=6, index=idx)


@pytest.mark.parametrize("order", [[0, 1, 2, 3], [0, 3, 1, 2], [3, 0, 1, 2], [1, 2, 3, 3]])
@pytest.mark.parametrize("gain", [8.0, 64.0])
def test_attend_tc_wide_scores_that_grow_late(bra, order, gain):
    """The keys of one region are scaled up, so that the row maxima of its key blocks lie far above
    those of the blocks routed before it (by a few hundred at gain 64): whatever reference
    maximum the kernel carries from earlier blocks, the result must be the plain softmax."""
    cfg = BraConfig("wide-late-scores", 1, 32, 32, 64, 2, 2, 4, "bf16")

    def louder_region_3(x):
        x["K"][:, 16:, 16:, :] *= gain             # region 3 of the 2 x 2 partition

    idx = np.array([[[order] * 4] * 2], dtype=np.int32)
    run_attend_case(bra, cfg, "tc", seed=31, index=idx, mutate=louder_region_3)


OPT_CASES = [BraConfig("opts", 2, 16, 16, 64, 2, 4, 3, "bf16"),
             BraConfig("opts-8x8-regions", 2, 32, 32, 64, 2, 4, 3, "bf16")]


@pytest.mark.parametrize("cfg", OPT_CASES, ids=[c.name for c in OPT_CASES])
@pytest.mark.parametrize("impl", ["simt", "auto"])
def test_attend_options(bra, impl, cfg):
    run_attend_case(bra, cfg, impl, seed=6, lce=False)
    run_attend_case(bra, cfg, impl, seed=6, bias=True)
    run_attend_case(bra, cfg, impl, seed=6, scale=0.5)
    run_attend_case(bra, cfg, impl, seed=6, shared=True)
    run_attend_case(bra, cfg, impl, seed=6, clustered=True)
    # a caller's index: any order, duplicates count twice
    rng = np.random.default_rng(3)
    idx = rng.integers(0, cfg.R, size=(cfg.B, cfg.heads, cfg.R, cfg.topk)).astype(np.int32)
    idx[0, 0, 0] = [5, 5, 5]
    run_attend_case(bra, cfg, impl, seed=6, index=idx)


@pytest.mark.parametrize("hw", [16, 32])
@pytest.mark.parametrize("impl", ["simt", "img", "auto"])
def test_out_of_range_index_is_reported_not_fatal(bra, impl, hw):
    import torch
    cfg = BraConfig("bad-index", 1, hw, hw, 64, 2, 4, 2, "bf16")
    x = synthetic.make_inputs(cfg, seed=8)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg, impl=IMPLS[impl])
    ws = bra.workspace(p)
    idx = torch.zeros(cfg.B, cfg.heads, cfg.R, cfg.topk, dtype=torch.int32, device="cuda")
    idx[0, 1, 3, 1] = cfg.R          # one past the end
    idx[0, 0, 7, 0] = -4
    O, _ = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, t["w"], ws=ws)
    assert bra.bra_device_status(ws) == 9
    assert bra.bra_device_status(ws) == 0          # cleared by the read
    assert torch.isfinite(O.float()).all()
    # the context is still usable and a clean call reports no error
    idx.zero_()
    bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, t["w"], ws=ws)
    assert bra.bra_device_status(ws) == 0


# ------------------------------------------------------------------ fused forward
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
def test_forward_matches_oracle(bra, n):
    cfg = CONFIGS[n]
    x = synthetic.make_inputs(cfg, seed=1000 + n)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    O, idx, lse = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws)
    assert bra.last_launch_count() >= 1
    assert bra.bra_device_status(ws) == 0
    _, _, idx_ref, gap = orc.bra_route(x["Q"], x["K"], cfg.heads, cfg.S, cfg.topk)
    near, flips = check_index(idx.cpu().numpy(), idx_ref, gap, cfg.topk, cfg.R, oracle_affinity(x, cfg))
    O_ref, lse_ref = orc.bra_attend(x["Q"], x["K"], x["V"], idx.cpu().numpy(), x["w"], cfg.heads, cfg.S)
    check_O(f64(O), O_ref, cfg.dtype)
    # without the optional outputs the result is the same
    O2, _, _ = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws, want_index=False, want_lse=False)
    assert (O2 == O).all()
    print(f"config {n}: forward ok, {near} near-tie rows, {flips} differ")


def test_forward_is_deterministic(bra):
    cfg = CONFIGS[5]
    x = synthetic.make_inputs(cfg, seed=42)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    O1, i1, l1 = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws)
    O2, i2, l2 = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws)
    assert (O1 == O2).all() and (i1 == i2).all() and (l1 == l2).all()


@pytest.mark.parametrize("n", [2, 3, 4, 5])
def test_forward_orders_attention_after_routing(bra, n):
    """The library's kernels overlap (programmatic dependent launch): attention must still see the
    index the routing step of the SAME call wrote.  Each call starts from an index buffer full of
    out-of-range entries and another pair of Q, K, so a kernel that read the buffer too early would
    either report a bad index or attend to the regions of the call before."""
    import torch
    cfg = CONFIGS[n]
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    sets = [to_dev(synthetic.make_inputs(cfg, seed=77 + s), cfg) for s in range(2)]
    want = []
    for t in sets:
        _, _, idx = bra.bra_route(p, t["Q"], t["K"], ws=ws)
        O, _ = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, t["w"], ws=ws)
        want.append((idx.clone(), O.clone()))
    assert bra.bra_device_status(ws) == 0
    idx = torch.empty_like(want[0][0])
    for it in range(6):
        t, (idx_ref, O_ref) = sets[it % 2], want[it % 2]
        idx.fill_(-7)
        O, idx, _ = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], index=idx, ws=ws)
        assert bra.bra_device_status(ws) == 0, f"call {it}"
        assert (idx == idx_ref).all() and (O == O_ref).all(), f"call {it}"


# bf16, head dim 32, 8 x 8-token regions, topk = 1, per-head routing, <= 64 regions, C <= 128: with
# BRA_IMPL_TC_FUSED bra_forward is ONE launch (pooling, routing, attention: three phases of one grid)
FUSED = 5
ONE_LAUNCH_CASES = [
    BraConfig("fused-single-region", 1, 8, 8, 64, 2, 1, 1, "bf16"),
    BraConfig("fused-one-image", 1, 56, 56, 64, 2, 7, 1, "bf16"),
    BraConfig("fused-two-head-pairs", 3, 32, 32, 128, 4, 4, 1, "bf16"),
    BraConfig("fused-64-regions", 2, 64, 64, 64, 2, 8, 1, "bf16"),
    BraConfig("fused-nine-regions", 5, 24, 24, 64, 2, 3, 1, "bf16"),
    BraConfig("fused-more-images-than-lookahead", 40, 16, 16, 64, 2, 2, 1, "bf16"),
]


@pytest.mark.parametrize("cfg", ONE_LAUNCH_CASES, ids=[c.name for c in ONE_LAUNCH_CASES])
def test_forward_in_one_launch_equals_route_then_attend(bra, cfg):
    """The one-launch forward gives, bit for bit, the index of bra_route and the O / lse of bra_attend,
    call after call on the same scratch buffer (its barrier counters clean themselves), and matches
    the oracle."""
    import torch
    p = problem_of(bra, cfg, impl=FUSED)
    ws = bra.workspace(p)
    sets = [to_dev(synthetic.make_inputs(cfg, seed=300 + s, clustered=bool(s)), cfg) for s in range(2)]
    want = []
    for t in sets:
        _, _, idx = bra.bra_route(p, t["Q"], t["K"], ws=ws)
        O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, t["w"], ws=ws)
        want.append((idx.clone(), O.clone(), lse.clone()))
    for it in range(5):
        t, (idx_ref, O_ref, lse_ref) = sets[it % 2], want[it % 2]
        O, idx, lse = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws)
        assert bra.last_launch_count() == 1
        assert bra.bra_device_status(ws) == 0, f"call {it}"
        assert (idx == idx_ref).all(), f"call {it}"
        assert (O == O_ref).all() and (lse == lse_ref).all(), f"call {it}"
    x = synthetic.make_inputs(cfg, seed=300)
    _, _, idx_o, gap = orc.bra_route(x["Q"], x["K"], cfg.heads, cfg.S, cfg.topk)
    check_index(want[0][0].cpu().numpy(), idx_o, gap, cfg.topk, cfg.R, oracle_affinity(x, cfg))
    O_o, _ = orc.bra_attend(x["Q"], x["K"], x["V"], want[0][0].cpu().numpy(), x["w"], cfg.heads, cfg.S)
    check_O(f64(want[0][1]), O_o, cfg.dtype)


def test_bounded_wait_that_runs_out_is_reported_and_recoverable(bra):
    """Failure detection without a GPU fault: with the injection switch one pooled unit of the
    one-launch forward is never counted as done, so every CTA's bounded wait for the end of pooling runs
    out (no tile copy and no tensor-core work has been issued at that point), the kernel returns, and the
    status reads BRA_ERR_TIMEOUT.  Reading the status restores the scratch buffer: the next call is clean."""
    cfg = BraConfig("timeout", 3, 32, 32, 64, 2, 4, 1, "bf16")
    t = to_dev(synthetic.make_inputs(cfg, seed=9), cfg)
    p = problem_of(bra, cfg, impl=FUSED)
    ws = bra.workspace(p)
    O_ref, idx_ref, _ = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws)
    assert bra.bra_device_status(ws) == 0
    p_bad = problem_of(bra, cfg, impl=FUSED, inject=1)
    bra.bra_forward(p_bad, t["Q"], t["K"], t["V"], t["w"], ws=ws)
    assert bra.bra_device_status(ws) == 10
    assert bra.bra_device_status(ws) == 0          # cleared by the read
    for _ in range(2):
        O, idx, _ = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws)
        assert bra.bra_device_status(ws) == 0
        assert (O == O_ref).all() and (idx == idx_ref).all()


def test_workspace_init_makes_a_dirty_buffer_usable(bra):
    """A scratch buffer full of garbage: after bra_workspace_init an out-of-range index entry is still
    reported, and the one-launch forward (which needs its counters at zero) gives the right result."""
    import torch
    cfg = BraConfig("dirty-ws", 2, 32, 32, 64, 2, 4, 1, "bf16")
    t = to_dev(synthetic.make_inputs(cfg, seed=10), cfg)
    p = problem_of(bra, cfg, impl=FUSED)
    O_ref, idx_ref, _ = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"])
    ws = bra.workspace(p)
    ws.fill_(0xFF)
    bra.workspace_init(p, ws)
    bad = idx_ref.clone()
    bad[1, 0, 3, 0] = cfg.R
    bra.bra_attend(p, t["Q"], t["K"], t["V"], bad, t["w"], ws=ws)
    assert bra.bra_device_status(ws) == 9
    O, idx, _ = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws)
    assert bra.bra_device_status(ws) == 0
    assert (O == O_ref).all() and (idx == idx_ref).all()


# ------------------------------------------------------------------ maps S does not divide (Appendix C)
PADDED_CASES = [
    BraConfig("pad-8x8-regions-k1", 2, 30, 29, 64, 2, 4, 1, "bf16"),          # padded to 32 x 32: tcgen05, topk = 1
    BraConfig("pad-8x8-regions-k3", 1, 61, 63, 64, 2, 8, 3, "bf16"),          # padded to 64 x 64: tcgen05, any topk
    BraConfig("pad-small-map-many-images", 40, 13, 13, 64, 2, 7, 4, "bf16"),  # padded to 14 x 14: image-resident
    BraConfig("pad-small-map", 3, 13, 14, 64, 2, 7, 4, "bf16"),               # warp-level kernel
    BraConfig("pad-wide-regions", 1, 30, 31, 64, 2, 2, 2, "bf16"),            # padded to 32 x 32, 16 x 16 regions
    BraConfig("pad-fp32", 1, 15, 14, 32, 1, 4, 2, "f32"),
]


@pytest.mark.parametrize("cfg", PADDED_CASES, ids=[c.name for c in PADDED_CASES])
def test_maps_that_S_does_not_divide(bra, cfg):
    """Forward and backward on a map zero-padded (inside the library) to the next multiples of S, against
    the oracle's padded reading: index of the padded map's regions, O / lse / gradients of the caller's size."""
    x = synthetic.make_inputs(cfg, seed=77, with_do=True)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    O, idx, lse = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws)
    assert bra.bra_device_status(ws) == 0
    assert tuple(O.shape) == (cfg.B, cfg.H, cfg.W, cfg.C) and tuple(lse.shape) == (cfg.B, cfg.heads, cfg.H * cfg.W)
    Qr, Kr, idx_ref, gap = orc.bra_route(x["Q"], x["K"], cfg.heads, cfg.S, cfg.topk)
    A = orc.region_affinity(Qr, Kr, cfg.heads)
    check_index(idx.cpu().numpy(), idx_ref, gap, cfg.topk, cfg.R, A)
    idn = idx.cpu().numpy()
    O_ref, lse_ref = orc.bra_attend(x["Q"], x["K"], x["V"], idn, x["w"], cfg.heads, cfg.S)
    check_O(f64(O), O_ref, cfg.dtype)
    np.testing.assert_allclose(f64(lse), lse_ref, rtol=0, atol=1e-5 if cfg.dtype == "f32" else 2e-3)
    # the two-call form gives the same
    qm, km, idx2 = bra.bra_route(p, t["Q"], t["K"], ws=ws)
    O2, lse2 = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx2, t["w"], ws=ws)
    assert (idx2 == idx).all() and (O2 == O).all()
    np.testing.assert_allclose(f64(qm), Qr, rtol=0, atol=2e-6)
    g = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, t["w"], lse, t["dO"], ws=ws, want_bias_grad=True)
    assert bra.bra_device_status(ws) == 0
    ref = orc.bra_backward(x["Q"], x["K"], x["V"], idn, x["w"], x["dO"], cfg.heads, cfg.S)
    tol = GRAD_MAX if cfg.dtype == "bf16" else 2e-4
    for name, a, r in zip(("dQ", "dK", "dV", "d_lce_w", "d_lce_b"), g, ref):
        assert tuple(a.shape) == r.shape, name
        assert np.abs(f64(a) - r).max() <= tol, f"{cfg.name} {name}"


# ------------------------------------------------------------------ backward
def run_backward_case(bra, cfg, seed, clustered=False, shared=False, index=None, impl="auto"):
    import torch
    x = synthetic.make_inputs(cfg, seed=seed, with_do=True, clustered=clustered)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg, impl=IMPLS[impl], shared_routing=shared)
    ws = bra.workspace(p)
    if index is None:
        O, idx, lse = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws)
    else:
        idx = torch.from_numpy(index).cuda()
        O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, t["w"], ws=ws)
    g1 = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, t["w"], lse, t["dO"], ws=ws, want_bias_grad=True)
    assert bra.last_launch_count() >= 3
    g2 = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, t["w"], lse, t["dO"], ws=ws, want_bias_grad=True)
    assert bra.bra_device_status(ws) == 0
    for a, b in zip(g1, g2):
        assert (a == b).all(), "backward is not bit-reproducible"
    ref = orc.bra_backward(x["Q"], x["K"], x["V"], idx.cpu().numpy(), x["w"], x["dO"], cfg.heads, cfg.S)
    names = ("dQ", "dK", "dV", "d_lce_w", "d_lce_b")
    tol = GRAD_MAX if cfg.dtype == "bf16" else 2e-4
    for name, g, r in zip(names, g1, ref):
        err = np.abs(f64(g) - r).max()
        assert err <= tol, f"{cfg.name} {name}: max-abs {err:.3e}"
        if name.startswith("d_lce"):
            # sums of B*H*W exact products accumulated in fp32: besides the stated absolute
            # bound, the error stays a small fraction of the largest entry
            assert err <= LCE_GRAD_REL * max(1.0, np.abs(r).max()), f"{cfg.name} {name}: {err:.3e} rel"


def test_backward_tiny_fp32(bra):
    run_backward_case(bra, CONFIGS[1], seed=1001)


def test_backward_training_config(bra):
    run_backward_case(bra, CONFIGS[5], seed=1005)


BWD_MMA_CASES = [
    BraConfig("bwd-2x2-regions-k16", 2, 14, 14, 256, 8, 7, 16, "bf16"),
    BraConfig("bwd-8x8-regions-k2", 2, 32, 32, 64, 2, 4, 2, "bf16"),
    BraConfig("bwd-16x16-regions-multi-block", 1, 32, 32, 64, 2, 2, 3, "bf16"),
    BraConfig("bwd-last-block-partial", 1, 14, 14, 64, 2, 7, 49, "bf16"),
    BraConfig("bwd-one-token-regions", 1, 4, 4, 32, 1, 4, 5, "bf16"),
    BraConfig("bwd-3x5-regions", 2, 12, 20, 64, 2, 4, 3, "bf16"),
]


@pytest.mark.parametrize("cfg", BWD_MMA_CASES, ids=[c.name for c in BWD_MMA_CASES])
def test_backward_tensor_core_shapes(bra, cfg):
    run_backward_case(bra, cfg, seed=31)


# maps small enough for the kernels that keep a whole (image, head) slice in shared memory
BWD_IMG_CASES = [c for c in BWD_MMA_CASES if c.H * c.W <= 1500] + [
    BraConfig("bwd-img-4x4-regions-k4", 3, 28, 28, 128, 4, 7, 4, "bf16"),
    BraConfig("bwd-img-tail-tile-n_r=24", 2, 12, 16, 64, 2, 2, 3, "bf16"),
    BraConfig("bwd-img-many-images", 40, 14, 14, 64, 2, 7, 5, "bf16"),
]


@pytest.mark.parametrize("cfg", BWD_IMG_CASES, ids=[c.name for c in BWD_IMG_CASES])
def test_backward_image_resident_shapes(bra, cfg):
    run_backward_case(bra, cfg, seed=33, impl="img")


def test_backward_image_resident_options(bra):
    cfg = BraConfig("bwd-img-opts", 2, 16, 16, 64, 2, 4, 3, "bf16")
    run_backward_case(bra, cfg, seed=34, impl="img", shared=True)
    run_backward_case(bra, cfg, seed=34, impl="img", clustered=True)
    idx = np.zeros((cfg.B, cfg.heads, cfg.R, cfg.topk), dtype=np.int32)
    idx[..., 1] = np.arange(cfg.R)[None, None, :] % 5
    idx[..., 2] = 3
    run_backward_case(bra, cfg, seed=35, impl="img", index=idx)


def test_backward_tensor_core_duplicates_and_fan_in(bra):
    cfg = BraConfig("bwd-dup-bf16", 1, 8, 8, 32, 1, 2, 3, "bf16")
    idx = np.array([[[[0, 0, 3], [1, 2, 1], [3, 3, 3], [2, 0, 1]]]], dtype=np.int32)
    run_backward_case(bra, cfg, seed=12, index=idx)
    # every query region routes to region 0 (largest fan-in) and region 5 is never routed to
    cfg = BraConfig("bwd-fan-in", 2, 16, 16, 64, 2, 4, 2, "bf16")
    idx = np.zeros((cfg.B, cfg.heads, cfg.R, cfg.topk), dtype=np.int32)
    idx[..., 1] = np.arange(cfg.R)[None, None, :] % 5
    run_backward_case(bra, cfg, seed=13, index=idx)


def test_backward_edge_cases(bra):
    run_backward_case(bra, synthetic.with_batch(CONFIGS[5], 4), seed=9, clustered=True)
    run_backward_case(bra, BraConfig("bwd-shared", 2, 12, 20, 64, 2, 4, 3, "bf16"), seed=10, shared=True)
    run_backward_case(bra, BraConfig("bwd-full", 1, 8, 8, 32, 2, 2, 4, "f32"), seed=11)
    cfg = BraConfig("bwd-dup", 1, 8, 8, 32, 1, 2, 3, "f32")
    idx = np.array([[[[0, 0, 3], [1, 2, 1], [3, 3, 3], [2, 0, 1]]]], dtype=np.int32)
    run_backward_case(bra, cfg, seed=12, index=idx)


# ------------------------------------------------------------------ random shapes
@pytest.mark.parametrize("seed", [11, 12])
def test_random_shapes_forward_and_backward(bra, seed):
    """Seeded random problems (head dim 32, bf16): region shapes from 1 x 1 to 8 x 8 and 16-wide, any S in
    {1, 2, 3, 4, 7}, 1-4 heads, k up to 12, every kernel family that accepts the shape, per-head and
    shared routing.  Forward against the oracle on the GPU's own index, then every gradient."""
    rng = np.random.default_rng(seed)
    ran = 0
    for it in range(16):
        S = int(rng.choice([1, 2, 3, 4, 7]))
        hs, ws = int(rng.integers(1, 9)), int(rng.integers(1, 9))
        if rng.random() < 0.3:
            ws, hs = 16, 8 * int(rng.integers(1, 3))
        heads = int(rng.choice([1, 2, 3, 4]))
        B = int(rng.choice([1, 2, 3, 40]))
        if B == 40 and S * S * hs * ws > 300:
            B = 3
        k = int(rng.integers(1, min(S * S, 12) + 1))
        cfg = BraConfig(f"rnd{seed}-{it}", B, S * hs, S * ws, 32 * heads, heads, S, k, "bf16")
        impl = str(rng.choice(["auto", "img", "mma", "tc"]))
        shared = bool(rng.random() < 0.2)
        x = synthetic.make_inputs(cfg, seed=100 * seed + it, with_do=True)
        t = to_dev(x, cfg)
        p = problem_of(bra, cfg, impl=IMPLS[impl], shared_routing=shared)
        ws_buf = bra.workspace(p)
        try:
            O, idx, lse = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws_buf)
        except bra.BraError as e:
            assert e.code == 7 and impl != "auto"        # that kernel family does not take the shape
            continue
        assert bra.bra_device_status(ws_buf) == 0
        idn = idx.cpu().numpy()
        O_ref, lse_ref = orc.bra_attend(x["Q"], x["K"], x["V"], idn, x["w"], cfg.heads, cfg.S)
        check_O(f64(O), O_ref, cfg.dtype)
        np.testing.assert_allclose(f64(lse), lse_ref, rtol=0, atol=2e-3)
        g = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, t["w"], lse, t["dO"], ws=ws_buf, want_bias_grad=True)
        assert bra.bra_device_status(ws_buf) == 0
        ref = orc.bra_backward(x["Q"], x["K"], x["V"], idn, x["w"], x["dO"], cfg.heads, cfg.S)
        for name, a, r in zip(("dQ", "dK", "dV", "d_lce_w", "d_lce_b"), g, ref):
            assert np.abs(f64(a) - r).max() <= GRAD_MAX, f"{cfg} {impl} {name}"
        ran += 1
    assert ran >= 8


# ------------------------------------------------------------------ edges of the kernels and of their dispatch rules
# The bounds are those at the top of this file: one rounding of P and of O to bf16 (2^-9 of values of order 1 to 4), fp32 sums
# otherwise.  `kind` of the index: "route" (bra_route's), "repeats" (random, one row names a single region).
def run_edge(bra, cfg, impl, kind="route", seed=51, **kw):
    index = None
    if kind == "repeats":
        rng = np.random.default_rng(seed)
        heads_i = 1 if kw.get("shared") else cfg.heads
        index = rng.integers(0, cfg.R, size=(cfg.B, heads_i, cfg.R, cfg.topk)).astype(np.int32)
        index[0, 0, 0] = cfg.R - 1
    run_attend_case(bra, cfg, impl, seed, index=index, **kw)
    if cfg.d <= 64:                         # no gradients at head dim 128
        run_backward_case(bra, cfg, seed, index=index, impl=impl, shared=kw.get("shared", False))


# every token of the map a key: topk * 16 rows (n_r rounded up) > tokens; above 64 tokens from 64 pairs on, gradients 296
DENSE_EDGES = [
    (BraConfig("dense-one-token-map", 1, 1, 1, 32, 1, 1, 1, "bf16"), "route"),
    (BraConfig("dense-1-token-regions-k=R", 2, 7, 7, 64, 2, 7, 49, "bf16"), "route"),
    (BraConfig("dense-64-regions", 2, 8, 8, 32, 1, 8, 5, "bf16"), "route"),          # the mask's last bit; repeats: counts
    (BraConfig("dense-64-regions-repeats", 2, 8, 8, 64, 2, 8, 5, "bf16"), "repeats"),
    (BraConfig("dense-1x2-regions", 3, 4, 8, 64, 2, 4, 3, "bf16"), "route"),
    (BraConfig("dense-3x3-regions", 2, 6, 6, 64, 2, 2, 3, "bf16"), "repeats"),
    (BraConfig("dense-3x5-regions-k=R", 2, 6, 10, 64, 2, 2, 4, "bf16"), "route"),
    (BraConfig("dense-2x2-regions-63-pairs", 63, 12, 12, 32, 1, 6, 13, "bf16"), "route"),
    (BraConfig("dense-2x2-regions-64-pairs", 64, 12, 12, 32, 1, 6, 13, "bf16"), "route"),
    (BraConfig("dense-256-tokens-296-pairs", 148, 16, 16, 64, 2, 8, 17, "bf16"), "route"),
    (BraConfig("dense-135-tokens-296-pairs", 148, 9, 15, 64, 2, 3, 9, "bf16"), "repeats"),
    (BraConfig("dense-padded-64-tokens", 2, 7, 6, 64, 2, 4, 5, "bf16"), "route"),
    (BraConfig("dense-padded-whole-regions", 2, 5, 5, 64, 2, 4, 5, "bf16"), "repeats"),
    (BraConfig("dense-padded-k=R-64-pairs", 32, 13, 13, 64, 2, 7, 49, "bf16"), "route"),
]


@pytest.mark.parametrize("cfg,kind", DENSE_EDGES, ids=[c.name for c, _ in DENSE_EDGES])
def test_dense_kernels_at_their_edges(bra, cfg, kind):
    run_edge(bra, cfg, "auto", kind)
    if cfg.B <= 3:
        run_edge(bra, cfg, "auto", "repeats", seed=52, shared=True)
        run_attend_case(bra, cfg, "auto", 53, lce=False)
        run_attend_case(bra, cfg, "auto", 54, bias=True, scale=0.5)
    if cfg.topk == cfg.R:                   # no index asked for: nothing needs to be routed
        x = synthetic.make_inputs(cfg, seed=55)
        t = to_dev(x, cfg)
        p = problem_of(bra, cfg)
        O, _, lse = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], want_index=False)
        every = np.broadcast_to(np.arange(cfg.R, dtype=np.int32), (cfg.B, cfg.heads, cfg.R, cfg.R))
        O_ref, lse_ref = orc.bra_attend(x["Q"], x["K"], x["V"], every, x["w"], cfg.heads, cfg.S)
        check_O(f64(O), O_ref, cfg.dtype)
        np.testing.assert_allclose(f64(lse), lse_ref, rtol=0, atol=2e-3)


# operands straight from global memory: any region and map, head dim 32 or 64; two tiles per warp from 1184 warps on
DIRECT_EDGES = [
    (BraConfig("direct-6x7-1152-warps", 18, 24, 28, 64, 2, 4, 3, "bf16"), "route"),
    (BraConfig("direct-6x7-1216-warps", 19, 24, 28, 64, 2, 4, 3, "bf16"), "route"),
    (BraConfig("direct-d64-6x7-1216-warps", 19, 24, 28, 128, 2, 4, 3, "bf16"), "repeats"),
    (BraConfig("direct-10x2-two-tiles", 37, 40, 8, 64, 2, 4, 2, "bf16"), "route"),
    (BraConfig("direct-7x3-two-tiles", 37, 28, 12, 64, 2, 4, 2, "bf16"), "route"),
    (BraConfig("direct-11x12-one-tile", 1, 22, 24, 64, 2, 2, 3, "bf16"), "repeats"),      # more than 128 tokens, 12-wide rows
    (BraConfig("direct-11x12-two-tiles", 30, 22, 24, 64, 2, 2, 3, "bf16"), "route"),
    (BraConfig("direct-2x128-row-of-a-chunk", 1, 4, 128, 32, 1, 1, 1, "bf16"), "route"),
    (BraConfig("direct-4x4-two-passes-of-a-table", 2, 28, 28, 64, 2, 7, 20, "bf16"), "repeats"),
    (BraConfig("direct-16x16-two-passes-of-a-table", 1, 32, 32, 64, 2, 2, 4, "bf16"), "route"),
    (BraConfig("direct-d64-one-token-regions", 1, 7, 7, 128, 2, 7, 49, "bf16"), "route"),
    (BraConfig("direct-d64-16x16", 1, 32, 32, 64, 1, 2, 3, "bf16"), "repeats"),
    (BraConfig("direct-padded-8x7", 2, 29, 27, 64, 2, 4, 3, "bf16"), "route"),
    (BraConfig("direct-padded-d64-8x7", 2, 29, 27, 128, 2, 4, 3, "bf16"), "route"),
    (BraConfig("direct-padded-two-tiles", 19, 21, 25, 64, 2, 4, 3, "bf16"), "route"),
    (BraConfig("direct-padded-rows-of-whole-regions", 2, 9, 9, 64, 2, 8, 6, "bf16"), "repeats"),
    (BraConfig("direct-529-regions", 1, 23, 23, 32, 1, 23, 3, "bf16"), "repeats"),          # inverse index: bits / comparisons
    (BraConfig("direct-576-regions", 1, 24, 24, 32, 1, 24, 3, "bf16"), "repeats"),
    (BraConfig("direct-961-regions", 1, 31, 31, 64, 2, 31, 5, "bf16"), "repeats"),
    # head dim 64, regions in chunks: one round of tiles per CTA below 148 CTAs
    (BraConfig("direct-d64-16x16-144-ctas", 18, 32, 32, 64, 1, 2, 3, "bf16"), "route"),
    (BraConfig("direct-d64-16x16-152-ctas", 19, 32, 32, 64, 1, 2, 3, "bf16"), "repeats"),
    (BraConfig("direct-d64-3x64", 1, 6, 128, 64, 1, 2, 2, "bf16"), "route"),
    (BraConfig("direct-d64-padded-9x17", 1, 17, 33, 64, 1, 2, 2, "bf16"), "repeats"),
]


@pytest.mark.parametrize("cfg,kind", DIRECT_EDGES, ids=[c.name for c, _ in DIRECT_EDGES])
def test_direct_kernels_at_their_edges(bra, cfg, kind):
    run_edge(bra, cfg, "mma", kind)
    if cfg.B <= 2:
        run_edge(bra, cfg, "mma", "repeats", seed=52, shared=True)
        run_attend_case(bra, cfg, "mma", 53, lce=False, index=np.zeros((cfg.B, cfg.heads, cfg.R, cfg.topk), np.int32))


# CUDA cores: two rows per lane up to head dim 32, 1 to 8 lanes per row, rows resident / staged / counted, chunks
SIMT_EDGES = [
    (BraConfig("simt-one-token-map", 1, 1, 1, 16, 1, 1, 1, "f32"), "route"),
    (BraConfig("simt-d16-8-lanes-per-row", 1, 8, 8, 16, 1, 2, 2, "f32"), "repeats"),
    (BraConfig("simt-d64-staged", 1, 24, 24, 64, 1, 3, 3, "f32"), "route"),
    (BraConfig("simt-d128", 1, 8, 12, 256, 2, 2, 3, "f32"), "repeats"),
    (BraConfig("simt-d128-odd-regions", 1, 9, 15, 128, 1, 3, 2, "f32"), "route"),
    (BraConfig("simt-one-lane-per-row", 32, 28, 28, 128, 4, 7, 1, "f32"), "route"),
    (BraConfig("simt-2x600-region", 1, 2, 600, 32, 1, 1, 1, "f32"), "route"),
    (BraConfig("simt-40x9-regions", 1, 80, 18, 32, 1, 2, 2, "f32"), "repeats"),
    (BraConfig("simt-every-region-counts", 1, 14, 14, 64, 2, 7, 49, "f32"), "repeats"),
    (BraConfig("simt-every-region", 2, 6, 6, 32, 1, 3, 9, "f32"), "route"),
    (BraConfig("simt-padded-d16", 2, 37, 26, 32, 2, 5, 4, "f32"), "route"),
    (BraConfig("simt-padded-resident", 1, 9, 9, 64, 2, 8, 6, "f32"), "repeats"),
    (BraConfig("simt-bf16-d16", 1, 14, 13, 32, 2, 7, 4, "bf16"), "route"),
    (BraConfig("simt-576-regions", 1, 24, 24, 32, 1, 24, 3, "f32"), "repeats"),
    # regions of one and two tokens with wide rows: one stage, as many regions as fit
    (BraConfig("simt-d64-1x1-k1", 1, 4, 4, 64, 1, 4, 1, "f32"), "route"),
    (BraConfig("simt-d64-1x1", 1, 14, 14, 64, 1, 14, 4, "f32"), "repeats"),
    (BraConfig("simt-d64-1x1-one-lane", 64, 16, 16, 192, 3, 16, 4, "f32"), "route"),
    (BraConfig("simt-d128-1x1", 1, 14, 14, 128, 1, 14, 4, "f32"), "repeats"),
    (BraConfig("simt-d128-1x1-one-lane", 64, 16, 16, 384, 3, 16, 3, "f32"), "route"),
    (BraConfig("simt-d128-1x2", 2, 14, 28, 256, 2, 14, 3, "f32"), "route"),
    (BraConfig("simt-d128-2x1-bf16", 2, 28, 14, 256, 2, 14, 3, "bf16"), "repeats"),
    (BraConfig("simt-d128-1x1-bf16", 2, 14, 14, 256, 2, 14, 3, "bf16"), "route"),
    (BraConfig("simt-d16-1x1", 64, 14, 14, 32, 2, 14, 8, "f32"), "route"),
    (BraConfig("simt-padded-1x2", 2, 6, 11, 32, 1, 6, 5, "f32"), "route"),
    (BraConfig("simt-padded-1x1-d64", 2, 5, 6, 64, 1, 6, 5, "f32"), "repeats"),
]


@pytest.mark.parametrize("cfg,kind", SIMT_EDGES, ids=[c.name for c, _ in SIMT_EDGES])
def test_cuda_core_kernels_at_their_edges(bra, cfg, kind):
    run_edge(bra, cfg, "simt", kind)
    if cfg.B <= 2:
        run_edge(bra, cfg, "simt", "repeats", seed=52, shared=True)
        run_attend_case(bra, cfg, "simt", 53, bias=True, index=np.zeros((cfg.B, cfg.heads, cfg.R, cfg.topk), np.int32))


@pytest.mark.parametrize("B,H,W,C,d,dtype", [
    (1, 1, 1, 32, 32, "bf16"), (2, 1, 70, 32, 32, "bf16"), (1, 70, 1, 96, 32, "f32"), (2, 33, 17, 96, 32, "bf16"),
    (1, 31, 65, 64, 64, "bf16"), (1, 5, 33, 16, 16, "f32"), (3, 17, 35, 80, 16, "f32"), (40, 12, 20, 128, 64, "bf16")])
def test_lce_weight_gradient_at_the_edges_of_its_tiles(bra, B, H, W, C, d, dtype):
    """Maps of one row or column, widths next to a tile's, channel counts that leave part of a block: d_lce_w and d_lce_b
    to the rounding of their fp32 sums (the attention gradients beside them have their own tests)."""
    import torch
    cfg = BraConfig("lce-grad", B, H, W, C, C // d, 1, 1, dtype)
    x = synthetic.make_inputs(cfg, seed=61, with_do=True)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    idx = torch.zeros(B, cfg.heads, 1, 1, dtype=torch.int32, device="cuda")
    _, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, t["w"], ws=ws)
    g = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, t["w"], lse, t["dO"], ws=ws, want_bias_grad=True)
    assert bra.bra_device_status(ws) == 0
    Vp = np.pad(x["V"].astype(np.float64), ((0, 0), (2, 2), (2, 2), (0, 0)))
    G = x["dO"].astype(np.float64)
    ref_w = np.stack([np.stack([(G * Vp[:, i:i + H, j:j + W]).sum((0, 1, 2)) for j in range(5)], -1) for i in range(5)], -2)
    ref_b = G.sum((0, 1, 2))
    for a, r in ((g[3], ref_w), (g[4], ref_b)):
        assert np.abs(f64(a) - r).max() <= LCE_GRAD_REL * max(1.0, np.abs(r).max())


@pytest.mark.parametrize("B,H,W,S,dtype", [
    (2, 30, 29, 4, "bf16"), (2, 13, 13, 7, "bf16"), (1, 6, 5, 7, "f32"), (2, 27, 26, 7, "f32"), (1, 23, 17, 4, "bf16"), (1, 5, 5, 4, "bf16")])
def test_pooling_of_maps_that_S_does_not_divide(bra, B, H, W, S, dtype):
    """Regions of 8 x 8, 2 x 2, 1 x 1, 4 x 4, 6 x 5 tokens that the map's edge cuts, and regions wholly outside."""
    cfg = BraConfig("pool", B, H, W, 64, 2, S, 2, dtype)
    x = synthetic.make_inputs(cfg, seed=71)
    t = to_dev(x, cfg)
    qm, km, idx = bra.bra_route(problem_of(bra, cfg), t["Q"], t["K"])
    Qr, Kr, idx_ref, gap = orc.bra_route(x["Q"], x["K"], cfg.heads, S, 2)
    np.testing.assert_allclose(f64(qm), Qr, rtol=0, atol=2e-6)
    np.testing.assert_allclose(f64(km), Kr, rtol=0, atol=2e-6)
    check_index(idx.cpu().numpy(), idx_ref, gap, 2, cfg.R, orc.region_affinity(Qr, Kr, cfg.heads))


# ------------------------------------------------------------------ large regions
@pytest.mark.parametrize("dtype,impl", [("f32", "simt"), ("bf16", "mma")])
def test_lists_with_repeats_of_large_regions(bra, dtype, impl):
    """Four regions of 22 500 tokens, every query region lists region 0 four times: the list of region 0 has 360 000 queries,
    and the last of them is the only one with a gradient.  The softmax over four copies of the keys is the softmax over one
    with every probability divided by four (exactly: a power of two), so O, and dK, dV summed over the copies, equal those
    of topk = 1 up to the rounding of sums in another order."""
    import torch
    H, W = 360, 250
    gen = torch.Generator(device="cuda")
    gen.manual_seed(91)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    Q, K, V = (torch.randn(1, H, W, 32, device="cuda", generator=gen).to(dt) for _ in range(3))
    dO = torch.zeros_like(Q)
    dO[0, -1, -1] = 1000.0 * torch.randn(32, device="cuda", generator=gen).to(dt)
    got = []
    for topk in (4, 1):
        p = bra.make_problem(1, H, W, 32, 1, 2, topk, dtype, lce=False, impl=IMPLS[impl])
        ws = bra.workspace(p)
        idx = torch.zeros(1, 1, 4, topk, dtype=torch.int32, device="cuda")
        O, lse = bra.bra_attend(p, Q, K, V, idx, ws=ws)
        dQ, dK, dV, _, _ = bra.bra_backward(p, Q, K, V, idx, None, lse, dO, ws=ws)
        assert bra.bra_device_status(ws) == 0
        got.append([f64(x) for x in (O, dQ, dK, dV)])
    # fp32: sums of up to 90 000 terms, sqrt(n) 2^-24 of them; bf16: two results rounded to 2^-9 each
    tol = 1e-4 if dtype == "f32" else 8e-3
    for name, a, r in zip(("O", "dQ", "dK", "dV"), *got):
        assert np.linalg.norm(a - r) <= tol * np.linalg.norm(r), name
    for a in got[0][2:]:
        assert np.abs(a[0, :180, :125]).max() > 0 and (a[0, 180:] == 0).all()       # region 0 only


# ------------------------------------------------------------------ problems that are more precise than one bf16 product
def rounding_ratio(got, ref):
    """Root mean square error of a bf16 result over that of the exact result rounded to bf16 once: 1 for a kernel whose own
    errors are small beside that rounding."""
    import torch
    ideal = torch.from_numpy(ref).to(torch.bfloat16).double().numpy()
    return np.sqrt(((f64(got) - ref) ** 2).mean() / ((ideal - ref) ** 2).mean())


# Regions of more than 128 tokens whose rows do not divide 128: P and dS enter their products with 16 bits of mantissa.  What
# that leaves, 2^-17 of each term, is 2^-8 of the result's own rounding (both add up over the same terms), which moves the
# ratio by about 2^-16; fp32 sums and ex2.approx are smaller still.  P and dS of 8 bits (2^-9 of each term) come out at 1.3
# to 1.5.  2 %: the ratio of 25 600 and more samples, few of which can differ.
RATIO_MAX = 1.02


@pytest.mark.parametrize("cfg", [
    BraConfig("exact-2x100", 1, 4, 200, 64, 2, 2, 2, "bf16"),
    BraConfig("exact-2x65", 2, 4, 130, 64, 2, 2, 3, "bf16"),
    BraConfig("exact-12x12", 1, 24, 24, 64, 2, 2, 3, "bf16"),
    BraConfig("exact-d64-2x100", 1, 4, 200, 128, 2, 2, 2, "bf16"),
], ids=lambda c: c.name)
def test_gradients_of_wide_regions_keep_their_precision(bra, cfg):
    x = synthetic.make_inputs(cfg, seed=93, with_do=True)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg, lce=False)
    ws = bra.workspace(p)
    O, idx, lse = bra.bra_forward(p, t["Q"], t["K"], t["V"], ws=ws)
    g = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, None, lse, t["dO"], ws=ws)
    assert bra.bra_device_status(ws) == 0
    ref = orc.bra_backward(x["Q"], x["K"], x["V"], idx.cpu().numpy(), np.zeros_like(x["w"]), x["dO"], cfg.heads, cfg.S)
    ratios = {name: rounding_ratio(a, r) for name, a, r in zip(("dQ", "dK", "dV"), g, ref)}
    print(cfg.name, ratios)
    assert max(ratios.values()) <= RATIO_MAX, ratios


@pytest.mark.parametrize("cfg", [
    BraConfig("exact-d64-12x12", 1, 24, 24, 128, 2, 2, 2, "bf16"),
    BraConfig("exact-d64-2x100", 1, 4, 200, 128, 2, 2, 2, "bf16"),
    BraConfig("exact-d64-12x12-two-tiles", 33, 24, 24, 128, 2, 2, 2, "bf16"),
    BraConfig("exact-12x12", 1, 24, 24, 64, 2, 2, 2, "bf16"),
], ids=lambda c: c.name)
def test_attention_of_wide_regions_keeps_its_precision(bra, cfg):
    x = synthetic.make_inputs(cfg, seed=94)
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg, lce=False)
    O, idx, _ = bra.bra_forward(p, t["Q"], t["K"], t["V"])
    ref, _ = orc.bra_attend(x["Q"], x["K"], x["V"], idx.cpu().numpy(), None, cfg.heads, cfg.S)
    assert rounding_ratio(O, ref) <= RATIO_MAX


@pytest.mark.parametrize("C", [32, 64])
def test_long_lists_keep_their_precision(bra, C):
    """More than 256 regions on a list (a caller's own index): 17 x 17 regions of one token, 257 of 289 listed."""
    import torch
    cfg = BraConfig("exact-long-lists", 2, 17, 17, C, 1, 17, 257, "bf16")
    x = synthetic.make_inputs(cfg, seed=95, with_do=True)
    t = to_dev(x, cfg)
    rng = np.random.default_rng(96)
    index = rng.permuted(np.tile(np.arange(cfg.R, dtype=np.int32), (cfg.B, 1, cfg.R, 1)), axis=-1)[..., :cfg.topk]
    idx = torch.from_numpy(np.ascontiguousarray(index)).cuda()
    p = problem_of(bra, cfg, lce=False)
    ws = bra.workspace(p)
    O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, ws=ws)
    g = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, None, lse, t["dO"], ws=ws)
    assert bra.bra_device_status(ws) == 0
    ref, _ = orc.bra_attend(x["Q"], x["K"], x["V"], index, None, cfg.heads, cfg.S)
    refs = (ref,) + orc.bra_backward(x["Q"], x["K"], x["V"], index, np.zeros_like(x["w"]), x["dO"], cfg.heads, cfg.S)[:3]
    ratios = {name: rounding_ratio(a, r) for name, a, r in zip(("O", "dQ", "dK", "dV"), (O,) + tuple(g[:3]), refs)}
    assert max(ratios.values()) <= RATIO_MAX, ratios


# ------------------------------------------------------------------ infinities and NaN stay where they are routed
def closed_lists(cfg, seed, bad=False, repeats=False):
    """Regions 0 .. topk - 1 list one another and nothing else lists them: what is in region 0 concerns no other region."""
    rng = np.random.default_rng(seed)
    idx = np.empty((cfg.B, cfg.heads, cfg.R, cfg.topk), np.int32)
    for b in range(cfg.B):
        for h in range(cfg.heads):
            for r in range(cfg.R):
                pool = np.arange(cfg.topk) if r < cfg.topk else np.arange(cfg.topk, cfg.R)
                idx[b, h, r] = rng.permutation(pool)[:cfg.topk]
    if repeats:
        idx[..., -1] = idx[..., 0]
    if bad:
        idx[0, 0, -1, -1] = cfg.R
        idx[-1, -1, cfg.topk, 0] = -1
    return idx


def region_mask(cfg, first, last):
    """[H, W]: tokens of regions first .. last - 1 of the (padded) map."""
    hs, ws = -(-cfg.H // cfg.S), -(-cfg.W // cfg.S)
    r = (np.arange(cfg.H) // hs)[:, None] * cfg.S + (np.arange(cfg.W) // ws)[None, :]
    return (r >= first) & (r < last)


def run_isolation_case(bra, cfg, impl, value, bad=False, repeats=False):
    """Region 0 of every tensor is `value`: O, lse and the gradients of the regions that do not list it are what they are
    with a finite region 0 (bf16: one rounding apart, in case the sums are taken in another order).  LCE off: it spreads
    over borders, rightly."""
    import torch
    x = synthetic.make_inputs(cfg, seed=97, with_do=True)
    idx = torch.from_numpy(closed_lists(cfg, 98, bad, repeats)).cuda()
    if repeats:
        idx[:, :, 0, 0] = 0                     # region 0 still lists itself
    p = problem_of(bra, cfg, impl=IMPLS[impl], lce=False)
    ws = bra.workspace(p)
    where = torch.from_numpy(region_mask(cfg, 0, 1)).cuda()
    outs = []
    for v in (None, value):
        t = to_dev(x, cfg)
        if v is not None:
            for n in ("Q", "K", "V", "dO"):
                t[n][:, where] = v
        O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, ws=ws)
        g = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, None, lse, t["dO"], ws=ws)
        assert bra.bra_device_status(ws) == (9 if bad else 0)
        outs.append((O,) + tuple(g[:3]) + (lse,))
    others = region_mask(cfg, cfg.topk, cfg.R)
    for name, clean, got in zip(("O", "dQ", "dK", "dV", "lse"), *outs):
        if name == "lse":
            a, r = f64(got)[..., others.ravel()], f64(clean)[..., others.ravel()]
        else:
            a, r = f64(got)[:, others], f64(clean)[:, others]
            assert not np.isfinite(f64(got)[:, where.cpu().numpy()]).any(), name       # region 0 lists itself
        assert np.isfinite(a).all(), f"{cfg.name} {name}: {np.count_nonzero(~np.isfinite(a))} of {a.size}"
        assert np.linalg.norm(a - r) <= (4e-3 if cfg.dtype == "bf16" else 1e-6) * np.linalg.norm(r), name


DIRECT_ISOLATION = [
    BraConfig("alone-one-block-of-keys", 2, 12, 20, 64, 2, 4, 3, "bf16"),           # 45 keys
    BraConfig("alone-tail", 2, 12, 20, 64, 2, 4, 7, "bf16"),                        # 105 keys
    BraConfig("alone-two-tables-of-a-warp", 1, 21, 35, 64, 2, 7, 20, "bf16"),       # 300 keys
    BraConfig("alone-two-tables-of-a-cta", 1, 30, 35, 64, 2, 5, 12, "bf16"),        # 504 keys of 42 tokens; lists up to 13 x 42
    BraConfig("alone-two-tiles-per-warp", 19, 24, 28, 64, 2, 4, 3, "bf16"),
    BraConfig("alone-d64", 1, 12, 20, 128, 2, 4, 3, "bf16"),
    BraConfig("alone-d64-two-tables", 1, 21, 35, 128, 2, 7, 20, "bf16"),
    BraConfig("alone-cut-map", 2, 29, 27, 64, 2, 4, 3, "bf16"),
    BraConfig("alone-cut-map-d64", 2, 29, 27, 128, 2, 4, 3, "bf16"),
    BraConfig("alone-11x12", 1, 33, 36, 64, 2, 3, 4, "bf16"),
    BraConfig("alone-cut-lists", 1, 64, 32, 64, 2, 8, 12, "bf16"),                  # parts of 8 entries, lists of up to 20
    BraConfig("alone-cut-lists-d64-five-tiles", 1, 64, 80, 64, 1, 8, 12, "bf16"),
]


@pytest.mark.parametrize("value", [float("inf"), float("nan")], ids=["inf", "nan"])
@pytest.mark.parametrize("cfg", DIRECT_ISOLATION, ids=lambda c: c.name)
def test_direct_kernels_keep_infinities_in_their_regions(bra, cfg, value):
    run_isolation_case(bra, cfg, "mma", value)
    run_isolation_case(bra, cfg, "mma", value, bad=True)


SIMT_ISOLATION = [
    BraConfig("alone-resident", 2, 8, 12, 64, 2, 4, 8, "f32"),
    BraConfig("alone-resident-d16", 2, 8, 12, 32, 2, 4, 7, "f32"),
    BraConfig("alone-staged-d64", 1, 12, 20, 64, 1, 4, 3, "f32"),
    BraConfig("alone-staged", 1, 21, 70, 64, 2, 7, 5, "f32"),
    BraConfig("alone-staged-d16", 1, 35, 35, 16, 1, 7, 9, "f32"),
    BraConfig("alone-staged-one-lane", 40, 21, 35, 64, 2, 7, 3, "f32"),
    BraConfig("alone-staged-d64-chunks", 1, 51, 51, 64, 1, 3, 2, "f32"),
    BraConfig("alone-cut-map-f32", 2, 29, 27, 64, 2, 4, 3, "f32"),
    BraConfig("alone-bf16-d16", 2, 12, 20, 32, 2, 4, 5, "bf16"),
    BraConfig("alone-1x1", 2, 6, 6, 64, 2, 6, 7, "f32"),
    BraConfig("alone-cut-1x2", 2, 6, 11, 64, 1, 6, 6, "f32"),
]


@pytest.mark.parametrize("value", [float("inf"), float("nan")], ids=["inf", "nan"])
@pytest.mark.parametrize("cfg", SIMT_ISOLATION, ids=lambda c: c.name)
def test_cuda_core_kernels_keep_infinities_in_their_regions(bra, cfg, value):
    run_isolation_case(bra, cfg, "simt", value)
    run_isolation_case(bra, cfg, "simt", value, bad=True)


@pytest.mark.parametrize("value", [float("inf"), float("nan")], ids=["inf", "nan"])
def test_cuda_core_kernels_keep_infinities_out_of_weighted_walks(bra, value):
    """topk = R with repeats: every region is walked, weighed by how often it is listed, region 0 not at all."""
    import torch
    cfg = BraConfig("alone-weighted", 2, 6, 6, 32, 1, 3, 9, "f32")
    x = synthetic.make_inputs(cfg, seed=97, with_do=True)
    idx = torch.randint(1, 9, (2, 1, 9, 9), dtype=torch.int32, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    idx[:, :, 0] = 0
    p = problem_of(bra, cfg, impl=IMPLS["simt"], lce=False)
    ws = bra.workspace(p)
    where = torch.from_numpy(region_mask(cfg, 0, 1)).cuda()
    outs = []
    for v in (None, value):
        t = to_dev(x, cfg)
        if v is not None:
            for n in ("Q", "K", "V", "dO"):
                t[n][:, where] = v
        O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, ws=ws)
        outs.append((O,) + tuple(bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, None, lse, t["dO"], ws=ws)[:3]))
    for clean, got in zip(*outs):
        assert (clean[:, ~where] == got[:, ~where]).all()


DENSE_ISOLATION = [
    BraConfig("alone-7x7", 20, 7, 7, 64, 2, 7, 10, "bf16"),
    BraConfig("alone-64-regions", 20, 8, 8, 64, 2, 8, 9, "bf16"),
    BraConfig("alone-2x2-regions", 60, 8, 8, 64, 2, 4, 5, "bf16"),
    BraConfig("alone-2x2-regions-64-pairs", 64, 12, 12, 32, 1, 6, 13, "bf16"),
    BraConfig("alone-256-tokens", 148, 16, 16, 64, 2, 8, 17, "bf16"),
    BraConfig("alone-cut-64-tokens", 60, 7, 6, 64, 2, 4, 5, "bf16"),
]


@pytest.mark.parametrize("value", [float("inf"), float("nan")], ids=["inf", "nan"])
@pytest.mark.parametrize("cfg", DENSE_ISOLATION, ids=lambda c: c.name)
def test_dense_kernels_keep_infinities_in_their_regions(bra, cfg, value):
    run_isolation_case(bra, cfg, "auto", value)
    run_isolation_case(bra, cfg, "auto", value, bad=True)
    run_isolation_case(bra, cfg, "auto", value, repeats=True)


@pytest.mark.parametrize("cfg", DENSE_ISOLATION, ids=lambda c: c.name)
def test_dense_kernels_by_token_match_the_oracle(bra, cfg):
    """One NaN makes a CTA work token by token: the tokens that it does not concern, LCE included, against the oracle."""
    import torch
    x = synthetic.make_inputs(cfg, seed=99, with_do=True)
    t = to_dev(x, cfg)
    index = closed_lists(cfg, 98)
    idx = torch.from_numpy(index).cuda()
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    bias = np.linspace(-0.5, 0.5, cfg.C).astype(np.float32)
    ref, _ = orc.bra_attend(x["Q"], x["K"], x["V"], index, x["w"], cfg.heads, cfg.S, None, bias)
    grads = orc.bra_backward(x["Q"], x["K"], x["V"], index, x["w"], x["dO"], cfg.heads, cfg.S)
    for n in ("Q", "K"):                        # (a NaN in V or dO spreads through the LCE)
        t[n][:, 0, 0] = float("nan")
    t["V"][:, 0, 0] = t["dO"][:, 0, 0] = float("inf")
    O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, t["w"], torch.from_numpy(bias).cuda(), ws=ws)
    g = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, t["w"], lse, t["dO"], ws=ws)
    assert bra.bra_device_status(ws) == 0
    far = region_mask(cfg, cfg.topk, cfg.R)
    far[:3, :3] = False
    check_O(f64(O)[:, far], ref[:, far], "bf16")
    for name, a, r in zip(("dQ", "dK", "dV"), g, grads):
        assert np.abs(f64(a)[:, far] - r[:, far]).max() <= GRAD_MAX, name


# ------------------------------------------------------------------ more images or heads than a grid holds in y or z
@pytest.mark.parametrize("dtype,impl,d", [("f32", "simt", 16), ("bf16", "mma", 32), ("bf16", "auto", 32)])
@pytest.mark.parametrize("many", ["images", "heads"])
def test_more_images_or_heads_than_a_grid_extent(bra, dtype, impl, d, many):
    """65 600 of them, 2 x 2 tokens each: the first and the last ones equal those of a problem of their own (another batch
    size may share rows between lanes otherwise: sums in another order)."""
    import torch
    n, part = 65600, 40
    B, heads = (n, 1) if many == "images" else (1, n)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    full = [torch.randn(B, 2, 2, heads * d, device="cuda", generator=gen).to(dt) for _ in range(4)]
    idx = torch.randint(0, 4, (B, heads, 4, 2), dtype=torch.int32, device="cuda", generator=gen)

    def run(x, idx):
        B, heads = idx.shape[:2]
        p = bra.make_problem(B, 2, 2, heads * d, heads, 2, 2, dtype, lce=False, impl=IMPLS[impl])
        ws = bra.workspace(p)
        O, lse = bra.bra_attend(p, x[0], x[1], x[2], idx, ws=ws)
        g = bra.bra_backward(p, x[0], x[1], x[2], idx, None, lse, x[3], ws=ws)
        assert bra.bra_device_status(ws) == 0
        return (O,) + tuple(g[:3])

    got = run(full, idx)
    for cut in (slice(0, part), slice(n - part, n)):
        if many == "images":
            ref = run([t[cut].contiguous() for t in full], idx[cut].contiguous())
            mine = [t[cut] for t in got]
        else:
            ch = slice(cut.start * d, cut.stop * d)
            ref = run([t[..., ch].contiguous() for t in full], idx[:, cut].contiguous())
            mine = [t[..., ch] for t in got]
        for a, r in zip(mine, ref):
            assert (a - r).float().norm() <= (4e-3 if dtype == "bf16" else 1e-6) * r.float().norm()


# ------------------------------------------------------------------ both sides of the dispatch rules
RULE_EDGES = [
    # maps of up to 64 tokens, attention: the direct kernel up to 1776 regions in the batch, the dense one from there on
    (BraConfig("rule-64-regions-27-pairs", 27, 8, 8, 32, 1, 8, 5, "bf16"), "route"),
    (BraConfig("rule-64-regions-28-pairs", 28, 8, 8, 32, 1, 8, 5, "bf16"), "repeats"),
    (BraConfig("rule-1x2-regions-111-pairs", 111, 4, 8, 32, 1, 4, 3, "bf16"), "repeats"),
    (BraConfig("rule-1x2-regions-112-pairs", 112, 4, 8, 32, 1, 4, 3, "bf16"), "route"),
    (BraConfig("rule-3x3-regions-446-pairs", 223, 6, 6, 64, 2, 2, 3, "bf16"), "route"),
    (BraConfig("rule-padded-112-pairs", 56, 7, 6, 64, 2, 4, 5, "bf16"), "repeats"),
    # regions of 4 x 4 and 2 x 2: resident slices from 190 pairs with enough to walk, gradients from 237
    (BraConfig("rule-2x2-188-pairs", 94, 20, 20, 64, 2, 10, 8, "bf16"), "route"),
    (BraConfig("rule-2x2-190-pairs", 95, 20, 20, 64, 2, 10, 8, "bf16"), "route"),
    (BraConfig("rule-4x4-236-pairs", 118, 8, 8, 64, 2, 2, 2, "bf16"), "repeats"),
    (BraConfig("rule-4x4-238-pairs", 119, 8, 8, 64, 2, 2, 2, "bf16"), "repeats"),
    (BraConfig("rule-4x4-15000-blocks", 200, 20, 20, 32, 1, 5, 6, "bf16"), "route"),
    (BraConfig("rule-4x4-14925-blocks", 199, 20, 20, 32, 1, 5, 6, "bf16"), "route"),
    # topk = 1, gradients: one launch up to 64 regions and from 32 pairs on, in between the direct kernels, which cut the long lists
    (BraConfig("rule-one-64-regions", 1, 40, 32, 64, 2, 8, 1, "bf16"), "repeats"),
    (BraConfig("rule-one-81-regions-31-pairs", 31, 45, 36, 32, 1, 9, 1, "bf16"), "route"),
    (BraConfig("rule-one-81-regions-32-pairs", 16, 45, 36, 64, 2, 9, 1, "bf16"), "route"),
    (BraConfig("rule-one-256-regions-3-pairs", 1, 80, 80, 96, 3, 16, 1, "bf16"), "repeats"),
]


@pytest.mark.parametrize("cfg,kind", RULE_EDGES, ids=[c.name for c, _ in RULE_EDGES])
def test_both_sides_of_the_dispatch_rules(bra, cfg, kind):
    run_edge(bra, cfg, "auto", kind)


# every region on every list, no index asked for: the dense attention masks nothing but what is behind the map's last token
ALL_LISTED = [
    BraConfig("all-1-token", 1, 1, 1, 32, 1, 1, 1, "bf16"),
    BraConfig("all-36-tokens", 2, 6, 6, 64, 2, 2, 4, "bf16"),
    BraConfig("all-49-tokens", 2, 7, 7, 64, 2, 7, 49, "bf16"),
    BraConfig("all-64-tokens", 3, 8, 8, 32, 1, 8, 64, "bf16"),
    BraConfig("all-100-tokens", 80, 10, 10, 32, 1, 5, 25, "bf16"),
    BraConfig("all-135-tokens", 32, 9, 15, 64, 2, 3, 9, "bf16"),
    BraConfig("all-padded-196", 40, 9, 11, 64, 2, 7, 49, "bf16"),
    BraConfig("all-256-tokens", 40, 16, 16, 64, 2, 8, 64, "bf16"),
]


@pytest.mark.parametrize("value", [None, float("inf"), float("nan")], ids=["finite", "inf", "nan"])
@pytest.mark.parametrize("cfg", ALL_LISTED, ids=lambda c: c.name)
def test_every_region_listed_without_an_index(bra, cfg, value):
    import torch
    x = synthetic.make_inputs(cfg, seed=109)
    t = to_dev(x, cfg)
    if value is not None:
        t["V"][0, 0, 0, 5] = value
        t["K"][-1, -1, -1, 7] = value
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    O, _, lse = bra.bra_forward(p, t["Q"], t["K"], t["V"], t["w"], ws=ws, want_index=False)
    assert bra.last_launch_count() == 1
    every = torch.arange(cfg.R, dtype=torch.int32, device="cuda").expand(cfg.B, cfg.heads, cfg.R, cfg.R).contiguous()
    O2, lse2 = bra.bra_attend(p, t["Q"], t["K"], t["V"], every, t["w"], ws=ws)
    assert bra.bra_device_status(ws) == 0
    assert torch.equal(O.nan_to_num(1e4, 1e5, -1e5), O2.nan_to_num(1e4, 1e5, -1e5))        # (the same sums in the same order)
    assert torch.equal(lse.nan_to_num(1e4, 1e5, -1e5), lse2.nan_to_num(1e4, 1e5, -1e5))
    if value is None:
        O_ref, lse_ref = orc.bra_attend(x["Q"], x["K"], x["V"], every.cpu().numpy(), x["w"], cfg.heads, cfg.S)
        check_O(f64(O), O_ref, cfg.dtype)
        np.testing.assert_allclose(f64(lse), lse_ref, rtol=0, atol=2e-3)


# ------------------------------------------------------------------ bad routing entries in every kernel, gradients among them
BAD_INDEX = [
    ("simt", BraConfig("bad-staged", 2, 12, 20, 64, 2, 4, 4, "f32")),
    ("simt", BraConfig("bad-resident", 2, 8, 12, 64, 2, 4, 8, "f32")),
    ("simt", BraConfig("bad-every-region", 2, 6, 6, 64, 2, 3, 9, "f32")),
    ("simt", BraConfig("bad-1x1", 2, 6, 6, 64, 2, 6, 7, "f32")),
    ("mma", BraConfig("bad-direct-one-block", 2, 12, 20, 64, 2, 4, 3, "bf16")),
    ("mma", BraConfig("bad-direct", 2, 21, 35, 64, 2, 7, 9, "bf16")),
    ("mma", BraConfig("bad-direct-d64", 2, 12, 20, 128, 2, 4, 4, "bf16")),
    ("mma", BraConfig("bad-direct-cut-lists", 1, 64, 32, 64, 2, 8, 12, "bf16")),           # parts of 8 entries
    ("mma", BraConfig("bad-direct-cut-lists-d64", 1, 64, 80, 64, 1, 8, 12, "bf16")),
    ("auto", BraConfig("bad-dense-7x7", 20, 7, 7, 64, 2, 7, 10, "bf16")),
    ("auto", BraConfig("bad-dense-k=R", 20, 7, 7, 64, 2, 7, 49, "bf16")),
    ("auto", BraConfig("bad-dense-2x2", 148, 16, 16, 64, 2, 8, 17, "bf16")),
    ("img", BraConfig("bad-resident-bf16", 2, 16, 16, 64, 2, 4, 4, "bf16")),
    ("tc", BraConfig("bad-tc", 2, 32, 32, 64, 2, 4, 4, "bf16")),
]


@pytest.mark.parametrize("impl,cfg", BAD_INDEX, ids=[c.name for _, c in BAD_INDEX])
def test_bad_entries_count_for_nothing(bra, impl, cfg):
    """Every row's last entry is out of range, every entry of one row is: the results are those of lists without these entries,
    a query without any gets the attention term 0, and the call reports BRA_ERR_INDEX."""
    import torch
    x = synthetic.make_inputs(cfg, seed=101, with_do=True)
    rng = np.random.default_rng(102)
    good = rng.permuted(np.tile(np.arange(cfg.R, dtype=np.int32), (cfg.B, cfg.heads, cfg.R, 1)), axis=-1)[..., :cfg.topk]
    bad = good.copy()
    bad[..., -1] = np.where(rng.random(bad[..., -1].shape) < 0.5, -1, cfg.R)
    lost = cfg.R // 2
    bad[0, 0, lost] = cfg.R + 3
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg, impl=IMPLS[impl], lce=False)
    ws = bra.workspace(p)
    idx = torch.from_numpy(bad).cuda()
    O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], idx, ws=ws)
    assert bra.bra_device_status(ws) == 9
    g = bra.bra_backward(p, t["Q"], t["K"], t["V"], idx, None, lse, t["dO"], ws=ws)
    assert bra.bra_device_status(ws) in (0, 9)       # (a gradient call may leave it to the forward call to say so)
    ref, _ = orc.bra_attend(x["Q"], x["K"], x["V"], good[..., :-1], None, cfg.heads, cfg.S)
    where = region_mask(cfg, lost, lost + 1)
    ref[0][where, :cfg.d] = 0
    dO = x["dO"].copy()
    dO[0][where, :cfg.d] = 0
    grads = orc.bra_backward(x["Q"], x["K"], x["V"], good[..., :-1], np.zeros_like(x["w"]), dO, cfg.heads, cfg.S)
    check_O(f64(O), ref, cfg.dtype)
    tol = GRAD_MAX if cfg.dtype == "bf16" else 2e-4
    for name, a, r in zip(("dQ", "dK", "dV"), g, grads):
        assert np.abs(f64(a) - r).max() <= tol, f"{name} {np.abs(f64(a) - r).max():.3e}"


# gradients of lists cut in parts (64 regions and more, parts of eight entries and more): every part of a region adds its sums
CUT_CASES = [
    BraConfig("cut-8x4", 2, 64, 32, 64, 2, 8, 2, "bf16"),
    BraConfig("cut-one-warp-regions", 1, 32, 32, 64, 2, 8, 3, "bf16"),                     # parts of 16
    BraConfig("cut-one-warp-regions-d64", 1, 32, 32, 128, 2, 8, 3, "bf16"),
    BraConfig("cut-odd-map", 1, 59, 61, 64, 2, 8, 2, "bf16"),
    BraConfig("cut-d64", 1, 48, 40, 128, 2, 8, 2, "bf16"),
    BraConfig("cut-12x12-chunks", 1, 96, 96, 32, 1, 8, 1, "bf16"),
    BraConfig("cut-8x16-two-rounds-d64", 1, 64, 128, 64, 1, 8, 2, "bf16"),
    BraConfig("cut-576-regions", 1, 96, 96, 32, 1, 24, 2, "bf16"),                         # inverse index without bits
    # two rounds of a CTA's four warps that have no tile for all of them: 5, 6 and 7 tiles, two chunks of 6, of 7 and 4
    BraConfig("cut-8x10-five-tiles-d64", 1, 64, 80, 128, 2, 8, 2, "bf16"),
    BraConfig("cut-9x10-six-tiles-d64", 1, 72, 80, 128, 2, 8, 4, "bf16"),
    BraConfig("cut-10x10-seven-tiles-d64", 1, 80, 80, 128, 2, 8, 2, "bf16"),
    BraConfig("cut-12x12-chunks-d64", 2, 96, 96, 192, 3, 8, 2, "bf16"),
    BraConfig("cut-18x9-chunks-d64", 2, 144, 72, 64, 1, 8, 2, "bf16"),
    BraConfig("cut-18x9-chunks", 2, 144, 72, 32, 1, 8, 2, "bf16"),
    # parts of the fair share, the last one shorter: 64 x 6 entries of 4 heads in two chunks over 296 CTAs, 11
    BraConfig("cut-fair-share", 1, 96, 96, 128, 4, 8, 6, "bf16"),
]


@pytest.mark.parametrize("cfg", CUT_CASES, ids=lambda c: c.name)
def test_gradients_of_lists_cut_in_parts(bra, cfg):
    rng = np.random.default_rng(71)
    shape = (cfg.B, cfg.heads, cfg.R, cfg.topk)
    # a few regions hold every list.  (dK and dV leave in bf16: a sum over n queries is about sqrt(n) times a query's share, and its
    # rounding alone |dK| 2^-9.  Five regions of 64 are listed some 40 times; so are 28 of 576, where |dK| of 25 would round by 0.05.)
    n = max(5, cfg.R // 20)
    few = rng.integers(0, n, size=shape).astype(np.int32) * (cfg.R // n)
    run_backward_case(bra, cfg, seed=72, index=few)
    # lists of every length around one, two and three parts, the other regions topk times or topk - 1 times.  (All columns of the index
    # but the first name every region once; what the first column has no room for comes in the next (image, head) or call.)
    part = max(8, -(-256 // (-(-cfg.H // cfg.S) * -(-cfg.W // cfg.S))))                   # entries: 256 queries, or 8, or a fair share
    part = 11 if cfg.name == "cut-fair-share" else part
    lengths = [part - 1, part, part + 1, 2 * part, 2 * part + 1, 3 * part, 3 * part + 1]
    firsts = [[]]
    for n in lengths:
        if sum(firsts[-1]) + n - (cfg.topk - 1) > cfg.R:
            firsts.append([])
        firsts[-1].append(n - (cfg.topk - 1))
    pairs = cfg.B * cfg.heads
    firsts += [firsts[0]] * (-len(firsts) % pairs)
    seen = set()
    for i in range(0, len(firsts), pairs):
        edge = np.broadcast_to(np.arange(cfg.R, dtype=np.int32)[::-1][:, None], (pairs, cfg.R, cfg.topk)).copy()
        for col, first in zip(edge[..., 0], firsts[i:i + pairs]):
            col[:] = np.arange(cfg.R)
            col[:sum(first)] = np.repeat(np.arange(len(first)), first)
        for rows in edge:
            seen |= set(np.bincount(rows.ravel()).tolist())
        run_backward_case(bra, cfg, seed=73, index=edge.reshape(shape))
    assert seen.issuperset(lengths)
    # the lists of this shape are cut: the scratch for the sums of the parts grows with topk, by far more than the index does (with a
    # fair share its parts grow instead: 4 heads, up to 2 * 384 / 11 parts, 12 tiles of 4 KB are most of the scratch)
    more = [bra.workspace_bytes(bra.make_problem(cfg.B, cfg.H, cfg.W, cfg.C, cfg.heads, cfg.S, k, cfg.dtype)) for k in (cfg.topk, cfg.topk + 1)]
    if cfg.name == "cut-fair-share":
        assert more[0] > 4 * 69 * 12 * 4096
    else:
        assert more[1] - more[0] > 10 * 8 * cfg.B * cfg.heads * cfg.R
    run_backward_case(bra, cfg, seed=74, index=few[:, :1].copy(), shared=True)
    if cfg.R <= 256:                                                                       # (as many as bra_forward routes)
        run_backward_case(bra, cfg, seed=75)


# topk = 1 in one launch: tiles of a region (17 .. 64 tokens), rows behind its last token, cut maps, every list length
ONE_EDGES = [
    (BraConfig("one-1x17", 1, 2, 34, 32, 1, 2, 1, "bf16"), "route"),
    (BraConfig("one-5x4", 3, 35, 28, 96, 3, 7, 1, "bf16"), "route"),
    (BraConfig("one-4x8", 2, 16, 32, 64, 2, 4, 1, "bf16"), "route"),
    (BraConfig("one-3x11", 2, 9, 33, 64, 2, 3, 1, "bf16"), "route"),
    (BraConfig("one-6x8", 2, 24, 32, 64, 2, 4, 1, "bf16"), "route"),
    (BraConfig("one-7x7", 2, 49, 49, 64, 2, 7, 1, "bf16"), "route"),
    (BraConfig("one-9x7", 2, 27, 21, 64, 2, 3, 1, "bf16"), "route"),
    (BraConfig("one-8x8", 2, 56, 56, 64, 2, 7, 1, "bf16"), "route"),
    (BraConfig("one-64x1", 1, 128, 2, 32, 1, 2, 1, "bf16"), "route"),
    (BraConfig("one-13x5-two-kernels", 2, 26, 10, 64, 2, 2, 1, "bf16"), "route"),          # 65 tokens
    (BraConfig("one-4x4-two-kernels", 2, 16, 16, 64, 2, 4, 1, "bf16"), "route"),           # 16
    (BraConfig("one-cut-8x7", 2, 29, 27, 64, 2, 4, 1, "bf16"), "route"),
    (BraConfig("one-cut-rows-of-whole-regions", 1, 33, 40, 32, 1, 8, 1, "bf16"), "route"),
    (BraConfig("one-256-regions", 1, 80, 96, 32, 1, 16, 1, "bf16"), "route"),
    (BraConfig("one-144-regions-32-pairs", 16, 60, 48, 64, 2, 12, 1, "bf16"), "route"),    # (256 regions of one image: the direct kernels)
]


@pytest.mark.parametrize("cfg,kind", ONE_EDGES, ids=[c.name for c, _ in ONE_EDGES])
def test_gradients_of_topk_1_at_their_edges(bra, cfg, kind):
    run_edge(bra, cfg, "auto", kind)
    idx = np.zeros((cfg.B, cfg.heads, cfg.R, 1), np.int32)                                 # one list of every region, the rest empty
    idx[:, :, 1:cfg.R // 2] = cfg.R - 1
    run_backward_case(bra, cfg, seed=61, index=idx)
    run_backward_case(bra, cfg, seed=62, shared=True)


def test_bad_entries_of_topk_1_have_no_gradient(bra):
    import torch
    cfg = BraConfig("bad-one", 2, 29, 27, 64, 2, 4, 1, "bf16")
    x = synthetic.make_inputs(cfg, seed=103, with_do=True)
    idx = np.random.default_rng(104).integers(0, cfg.R, (cfg.B, cfg.heads, cfg.R, 1)).astype(np.int32)
    good = idx.copy()
    lost = (1, 5)
    for r, v in zip(lost, (-1, cfg.R)):
        idx[0, 0, r] = v
    t = to_dev(x, cfg)
    p = problem_of(bra, cfg, lce=False)
    ws = bra.workspace(p)
    dev = torch.from_numpy(idx).cuda()
    O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], dev, ws=ws)
    assert bra.bra_device_status(ws) == 9
    g = bra.bra_backward(p, t["Q"], t["K"], t["V"], dev, None, lse, t["dO"], ws=ws)
    assert bra.bra_device_status(ws) == 9
    dO = x["dO"].copy()
    for r in lost:
        dO[0][region_mask(cfg, r, r + 1), :cfg.d] = 0
    ref = orc.bra_backward(x["Q"], x["K"], x["V"], good, np.zeros_like(x["w"]), dO, cfg.heads, cfg.S)
    for name, a, r in zip(("dQ", "dK", "dV"), g, ref):
        assert np.abs(f64(a) - r).max() <= GRAD_MAX, name


@pytest.mark.parametrize("value", [float("inf"), float("nan")], ids=["inf", "nan"])
@pytest.mark.parametrize("hw", [(24, 28), (29, 27), (28, 24)])
def test_gradients_of_topk_1_keep_infinities_in_their_regions(bra, hw, value):
    run_isolation_case(bra, BraConfig("alone-one", 2, hw[0], hw[1], 64, 2, 4, 1, "bf16"), "auto", value)


@pytest.mark.parametrize("impl", ["auto", "mma"])
@pytest.mark.parametrize("hw", [(24, 28), (29, 27), (32, 32)], ids=["6x7-regions", "cut-map", "8x8-regions"])
def test_a_key_at_minus_infinity_leaves_its_neighbours_gradients_alone(bra, hw, impl):
    """A key that scores -inf with every query has P = 0: gradients of the region's other keys are those beside a key that scores far
    below all others.  (Rows that fill up a tile or a cut map are no queries: their score is 0 * inf.)"""
    import torch
    cfg = BraConfig("infinite-key", 2, hw[0], hw[1], 64, 2, 4, 1, "bf16")
    x = synthetic.make_inputs(cfg, seed=107, with_do=True)
    x["Q"][..., 3::32] = np.abs(x["Q"][..., 3::32]) + 0.5
    idx = np.zeros((cfg.B, cfg.heads, cfg.R, 1), np.int32)
    idx[:, :, cfg.R // 2:] = 5
    p = problem_of(bra, cfg, impl=IMPLS[impl], lce=False)
    ws = bra.workspace(p)
    dev = torch.from_numpy(idx).cuda()
    x["K"][:, 1, 1, 3::32] = -np.inf
    t = to_dev(x, cfg)
    O, lse = bra.bra_attend(p, t["Q"], t["K"], t["V"], dev, ws=ws)
    g = bra.bra_backward(p, t["Q"], t["K"], t["V"], dev, None, lse, t["dO"], ws=ws)
    assert bra.bra_device_status(ws) == 0
    x["K"][:, 1, 1, 3::32] = -2.0 ** 17                        # scores from 2^17 * 0.5 / sqrt(32) = 11585 below
    ref = orc.bra_backward(x["Q"], x["K"], x["V"], idx, np.zeros_like(x["w"]), x["dO"], cfg.heads, cfg.S)
    others = np.ones((cfg.H, cfg.W), bool)
    others[1, 1] = False
    for name, a, r in zip(("dK", "dV"), g[1:3], ref[1:3]):
        assert np.abs(f64(a) - r)[:, others].max() <= GRAD_MAX, name


# ------------------------------------------------------------------ inputs written right before the call; graphs
ORDER_CASES = [
    BraConfig("order-pool-rows", 16, 28, 28, 128, 4, 7, 4, "bf16"),
    BraConfig("order-pool-split", 16, 56, 56, 64, 2, 7, 1, "bf16"),
    BraConfig("order-pool-8", 8, 49, 49, 64, 2, 7, 2, "bf16"),
    BraConfig("order-pool-16", 2, 128, 128, 64, 2, 8, 4, "bf16"),
    BraConfig("order-padded", 4, 61, 53, 64, 2, 4, 3, "bf16"),
    BraConfig("order-dense", 16, 7, 7, 512, 16, 7, 49, "bf16"),
    BraConfig("order-fp32", 4, 28, 28, 64, 2, 7, 4, "f32"),
]


def order_step(bra, cfg, source, ws):
    """One kernel writes Q, K, V and dO, the calls follow it on the stream."""
    import torch
    p = problem_of(bra, cfg)
    X = torch.empty_like(source)
    w = torch.full((cfg.C, 5, 5), 0.01, device="cuda")
    index = torch.empty(cfg.B, cfg.heads, cfg.R, cfg.topk, dtype=torch.int32, device="cuda")

    def step():
        torch.mul(source, 1.0, out=X)
        O, _, lse = bra.bra_forward(p, X[0], X[1], X[2], w, index=index, ws=ws)
        g = bra.bra_backward(p, X[0], X[1], X[2], index, w, lse, X[3], ws=ws, want_bias_grad=True)
        return (O, index, lse) + tuple(g)

    return step, X


def order_sources(cfg, n):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    dt = torch.bfloat16 if cfg.dtype == "bf16" else torch.float32
    return [torch.randn(4, cfg.B, cfg.H, cfg.W, cfg.C, device="cuda", generator=gen).to(dt) for _ in range(n)]


@pytest.mark.parametrize("cfg", ORDER_CASES, ids=lambda c: c.name)
def test_calls_wait_for_the_kernel_that_writes_their_inputs(bra, cfg):
    """The first kernel of a call may be set up under the kernel before it in the stream: it must still see what that one wrote.
    The inputs are overwritten with NaN-free but other values between the steps, nothing synchronises in between."""
    import torch
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    sources = order_sources(cfg, 2)
    want = []
    for src in sources:
        step, X = order_step(bra, cfg, src, ws)
        X.copy_(src)
        torch.cuda.synchronize()
        want.append([t.clone() for t in step()])
        torch.cuda.synchronize()
    live = torch.empty_like(sources[0])
    step, X = order_step(bra, cfg, live, ws)
    got = []
    for it in range(6):
        live.copy_(sources[it % 2])
        X.fill_(3.0)
        got.append([t.clone() for t in step()])
    torch.cuda.synchronize()
    assert bra.bra_device_status(ws) == 0
    for it, outs in enumerate(got):
        for a, r in zip(outs, want[it % 2]):
            assert torch.equal(a, r), f"step {it}"


@pytest.mark.parametrize("cfg", ORDER_CASES, ids=lambda c: c.name)
def test_calls_in_a_cuda_graph(bra, cfg):
    """Forward and backward (its helper stream among them) captured behind the kernel that writes their inputs, replayed on
    other inputs: the results of the calls made directly."""
    import torch
    p = problem_of(bra, cfg)
    ws = bra.workspace(p)
    sources = order_sources(cfg, 2)
    want = []
    for src in sources:
        want.append([t.clone() for t in order_step(bra, cfg, src, ws)[0]()])
    live = sources[0].clone()
    step, _ = order_step(bra, cfg, live, ws)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        step()
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        outs = step()
    for it in range(4):
        live.copy_(sources[it % 2])
        graph.replay()
        torch.cuda.synchronize()
        assert bra.bra_device_status(ws) == 0
        for a, r in zip(outs, want[it % 2]):
            assert torch.equal(a, r), f"replay {it}"
    del graph
