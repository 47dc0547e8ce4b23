"""GPU parity of the BCQ product from the exported format (uq_bcq_gemv)
against the oracle's fp64 product (oracle.bcq_gemv).

Tolerance: the kernel accumulates in fp32 in its own fixed order (per-8-
column partial sums of x, per-lane terms z* S + sum_j alpha*_j (2 P_j - S),
a warp reduction, then the tiles).  Every rounding error is bounded by a
small multiple of the unit roundoff times the L1 mass of the expanded terms,
sum_i (sum_j |alpha*_j| + |z*|) |x_i| (computed in fp64 here); the tests
allow 1e-5 of that mass (about 170 unit roundoffs).
"""

import numpy as np
import pytest
import torch

import oracle as O
from paper_2506_03781_gb300 import api, synth
from tests import gpu_cases as C

pytestmark = pytest.mark.gpu
F32 = np.float32
F64 = np.float64
TOL = 1e-5


def mass(a_star, z_star, x, g):
    per_col = np.repeat(np.abs(np.asarray(a_star, F64)).sum(-1) + np.abs(np.asarray(z_star, F64)), g, axis=1)
    return np.abs(np.asarray(x, F64)) @ per_col.T             # [batch, out]


def random_export(out, n_in, q, g, seed):
    rng = np.random.default_rng(seed)
    planes = rng.integers(0, 2 ** 32, (q, out, n_in // 32), dtype=np.uint64).astype(np.uint32)
    a_star = (rng.standard_normal((out, n_in // g, q)) * 0.01).astype(F32)
    z_star = (rng.standard_normal((out, n_in // g)) * 0.003).astype(F32)
    return planes, a_star, z_star


def gpu_gemv(planes, a_star, z_star, x, g, xdtype="f32"):
    d = C.dev()
    pd = torch.from_numpy(planes.view(np.int32)).to(d)
    ad = torch.from_numpy(a_star).to(d)
    zd = torch.from_numpy(z_star).to(d)
    if xdtype == "bf16":
        raw, _ = synth.bf16_round(x)
        xd = api.weights_tensor(raw, d)
    else:
        xd = torch.from_numpy(np.ascontiguousarray(x, F32)).to(d)
    y = torch.full((x.shape[0], planes.shape[1]), float("nan"), device=d)
    # the workspace starts as NaN: every word the product reads must have been written by it
    ws = torch.full((api.uq_bcq_gemv_workspace_bytes(planes.shape[1], x.shape[1], x.shape[0]) // 4,), float("nan"),
                    device=d)
    api.uq_bcq_gemv(pd, ad, zd, xd, y, g, workspace=ws)
    api.uq_check_device()                         # no pipeline wait ran out, no layout refused
    return C.host(y)


def check(planes, a_star, z_star, x, g, xdtype="f32", label="", least=1e-30):
    if xdtype == "bf16":
        _, x = synth.bf16_round(x)               # the oracle sees the values the kernel reads
    y = gpu_gemv(planes, a_star, z_star, x, g, xdtype)
    ref = O.bcq_gemv(planes, a_star, z_star, x, g)
    err = np.abs(y.astype(F64) - ref)
    bound = TOL * mass(a_star, z_star, x, g) + least
    assert np.isfinite(y).all(), label
    assert (err <= bound).all(), f"{label}: worst {(err / bound).max():.3g} x tolerance"
    return y


# in: one ragged tile, several tiles, a non-multiple of 512.  In a multiple of 1024 with
# g <= 256 takes the wide-lane kernel (1024-column tiles, 4 to 32 groups per tile); other
# whole 512-column tiles with 4, 8 and 16 groups per tile the tensor-copy staging, the
# rest the per-lane copies (one token)
@pytest.mark.parametrize("out,n_in,g", [(40, 256, 32), (33, 512, 64), (17, 1536, 128), (64, 4096, 128),
                                        (9, 4096 + 32 * 3, 32), (5, 8192, 256), (3, 28672, 128), (300, 1024, 512),
                                        (24, 1024, 32), (13, 2560, 64), (11, 3072, 1024), (6, 4096, 2048)])
@pytest.mark.parametrize("q", [1, 2, 3, 4])
def test_gemv_matches_oracle(out, n_in, g, q):
    if n_in % g:
        pytest.skip("in must be a multiple of g")
    planes, a_star, z_star = random_export(out, n_in, q, g, seed=out + q)
    x = np.random.default_rng(q).standard_normal((1, n_in)).astype(F32)
    check(planes, a_star, z_star, x, g, label=f"{out}x{n_in} g{g} q{q}")


@pytest.mark.parametrize("batch", [2, 5])
@pytest.mark.parametrize("xdtype", ["f32", "bf16"])
def test_gemv_batches_and_bf16_activations(batch, xdtype):
    planes, a_star, z_star = random_export(48, 2048, 3, 128, seed=7)
    x = np.random.default_rng(batch).standard_normal((batch, 2048)).astype(F32)
    check(planes, a_star, z_star, x, 128, xdtype, label=f"batch {batch} {xdtype}")


@pytest.mark.parametrize("out,n_in,g,q", [(9000, 512, 64, 2), (9001, 2048, 64, 2), (2053, 3072, 32, 4),
                                          (1, 1024, 256, 1), (7, 1024, 128, 3)])
def test_gemv_many_rows(out, n_in, g, q):
    """Many more rows than one wave of row blocks, a ragged last batch of
    rows, and single-row and single-tile products, on both kernels."""
    planes, a_star, z_star = random_export(out, n_in, q, g, seed=9 + out)
    x = np.random.default_rng(0).standard_normal((2, n_in)).astype(F32)
    check(planes, a_star, z_star, x, g, label=f"{out} rows {n_in} g{g} q{q}")


# The tensor-core product (5 tokens and more, 2 to 4 where it is the faster one): row tiles of 128 with a
# remainder, one row, columns that are no whole 128-column pass (per-thread loads), slices that begin inside
# a pass's four groups, every group size class; 16, 32 and 64 matrix columns and several chunks of tokens (an
# fp32 token takes three columns)
@pytest.mark.parametrize("out,n_in,g,q", [(1, 32, 32, 3), (127, 96, 32, 1), (129, 192, 64, 2), (300, 320, 64, 4),
                                          (128, 128, 128, 3), (257, 640, 128, 2), (65, 11008, 128, 3),
                                          (40, 1280, 256, 4), (31, 3072, 1024, 1), (2500, 6080, 32, 2)])
@pytest.mark.parametrize("batch,xdtype", [(3, "bf16"), (5, "f32"), (6, "f32"), (17, "bf16"), (22, "f32"),
                                          (33, "bf16"), (64, "f32"), (64, "bf16")])
def test_gemv_tensor_core_product(out, n_in, g, q, batch, xdtype):
    planes, a_star, z_star = random_export(out, n_in, q, g, seed=out + batch)
    x = np.random.default_rng(batch + q).standard_normal((batch, n_in)).astype(F32)
    check(planes, a_star, z_star, x, g, xdtype, label=f"{out}x{n_in} g{g} q{q} batch {batch} {xdtype}")


# Two to four tokens on both sides of the lines by size, bit-width and group between the lookup tables and the
# tensor cores (the rows around a power of two of out * in, and of out = 2048 for larger groups)
@pytest.mark.parametrize("out,n_in,g,q,batch", [
    (2730, 1536, 32, 4, 3), (2731, 1536, 32, 3, 3), (682, 1536, 32, 2, 3), (683, 1536, 32, 2, 3), (682, 1536, 64, 3, 3),
    (683, 1536, 64, 3, 3), (2731, 1536, 64, 4, 3), (683, 1536, 128, 4, 3), (682, 1536, 128, 4, 3), (682, 1536, 32, 4, 4),
    (683, 1536, 64, 4, 4), (10922, 1536, 64, 2, 2), (10923, 1536, 64, 2, 2), (2047, 8704, 512, 3, 2),
    (2048, 8704, 512, 3, 2), (2048, 8704, 512, 4, 2), (2047, 8704, 512, 3, 3)])
def test_gemv_on_both_sides_of_a_path_line(out, n_in, g, q, batch):
    planes, a_star, z_star = random_export(out, n_in, q, g, seed=out + q)
    x = np.random.default_rng(batch).standard_normal((batch, n_in)).astype(F32)
    check(planes, a_star, z_star, x, g, "f32" if out % 2 else "bf16", label=f"{out}x{n_in} g{g} q{q} batch {batch}")


# Several row tiles per block with two and three warpgroups, planes through the ring of tensor copies: sizes the
# product was built for, tile counts that are no multiple of the warpgroups, a last tile of one row; and two
# groups of 256 loaded at a time, from slices that begin inside a four-pass window and at its start.  The rows
# checked are a few of every tile (outputs of other rows depend on other planes only).
@pytest.mark.parametrize("out,n_in,g,q,batch,xdtype", [
    (14336, 4096, 128, 3, 64, "bf16"), (8192, 28672, 128, 3, 4, "f32"), (128 * 152 * 5 + 1, 1024, 128, 2, 16, "bf16"),
    (128 * 152 * 4 - 100, 512, 64, 3, 30, "bf16"), (8192, 8192, 256, 3, 4, "bf16"), (6000, 8192, 256, 4, 22, "f32"),
    (700, 28672, 256, 2, 6, "f32"), (300, 11264, 256, 1, 33, "bf16")])
def test_gemv_tensor_core_product_of_many_tiles_and_slices(out, n_in, g, q, batch, xdtype):
    planes, a_star, z_star = random_export(out, n_in, q, g, seed=out + q)
    x = np.random.default_rng(q).standard_normal((batch, n_in)).astype(F32)
    if xdtype == "bf16":
        _, x = synth.bf16_round(x)
    y = gpu_gemv(planes, a_star, z_star, x, g, xdtype)
    assert np.isfinite(y).all()
    first = np.arange(0, out, 128)
    rows = np.unique(np.concatenate([first, np.minimum(first + 127, out - 1), np.random.default_rng(0).integers(0, out, 60)]))
    err = np.abs(y[:, rows] - O.bcq_gemv(np.ascontiguousarray(planes[:, rows]), a_star[rows], z_star[rows], x, g))
    assert (err <= TOL * mass(a_star[rows], z_star[rows], x, g)).all()


@pytest.mark.parametrize("xdtype", ["f32", "bf16"])
def test_gemv_extreme_activations_stay_in_their_token(xdtype):
    """Largest, smallest and tiny activations keep the bound; an infinity and
    a NaN make their own token's outputs non-finite and no other's."""
    out, n_in, g, q = 130, 1024, 64, 3
    planes, a_star, z_star = random_export(out, n_in, q, g, seed=3)
    x = np.random.default_rng(1).standard_normal((6, n_in)).astype(F32)
    x[1] *= F32(1e34)
    x[2] *= F32(1e-30)
    x[3, ::7] *= F32(1e12)
    check(planes, a_star, z_star, x, g, xdtype, label="extreme")
    x[4, 5], x[5, 77] = np.inf, np.nan
    if xdtype == "bf16":
        raw, _ = synth.bf16_round(np.where(np.isfinite(x), x, 0))
        raw[4, 5], raw[5, 77] = 0x7F80, 0x7FC0
        xd = api.weights_tensor(raw, C.dev())
    else:
        xd = torch.from_numpy(x).to(C.dev())
    y = torch.empty(6, out, device=C.dev())
    api.uq_bcq_gemv(torch.from_numpy(planes.view(np.int32)).to(C.dev()), torch.from_numpy(a_star).to(C.dev()),
                    torch.from_numpy(z_star).to(C.dev()), xd, y, g)
    assert torch.isfinite(y[:4]).all() and not torch.isfinite(y[4:]).any()


# 16, 32 and 64 matrix columns, blocks of one, two and four to a pass, and the lookup tables (one token)
@pytest.mark.parametrize("g,q", [(32, 2), (64, 3), (128, 3), (512, 4)])
@pytest.mark.parametrize("batch,xdtype", [(1, "f32"), (5, "f32"), (10, "f32"), (15, "bf16"), (15, "f32"), (40, "bf16")])
def test_gemv_holds_its_bound_over_the_whole_range_of_the_type(g, q, batch, xdtype):
    """Tokens down to the smallest numbers of the type (a bf16 piece or half of
    one of them would fall below it) and up to where a sum of 128 activations
    exceeds fp32 but the product does not, also with both in one token.  Each
    term may be rounded to a multiple of 2^-149 besides: n_in of them."""
    out, n_in = 140, 1024
    planes, a_star, z_star = random_export(out, n_in, q, g, seed=8)
    rng = np.random.default_rng(batch)
    x = rng.standard_normal((batch, n_in)).astype(F32)
    scales = [2.0 ** -112, 2.0 ** -120, 2.0 ** -126, 2.0 ** -133, 2.0 ** 122, 2.0 ** -64, 2.0 ** 108, 1.0]
    for b in range(batch):
        x[b] = (x[b].astype(F64) * scales[(b + batch) % len(scales)]).astype(F32)
    if batch > 1:
        x[1] = np.abs(x[1])                                       # one sign: sums that do not cancel
        x[0, :512] = rng.standard_normal(512).astype(F32) * F32(2.0 ** -124)       # other passes, other scales
        x[2, ::2] = rng.standard_normal(512).astype(F32) * F32(2.0 ** 109)         # ... and within a pass
    check(planes, a_star, z_star, x, g, xdtype, label=f"range g{g} q{q} batch {batch} {xdtype}",
          least=n_in * 2.0 ** -149)


def test_gemv_deterministic():
    planes, a_star, z_star = random_export(100, 8192, 3, 128, seed=11)
    x = np.random.default_rng(1).standard_normal((2, 8192)).astype(F32)
    a = gpu_gemv(planes, a_star, z_star, x, 128)
    b = gpu_gemv(planes, a_star, z_star, x, 128)
    assert np.array_equal(a, b)


def test_gemv_of_the_quantizer_export_reproduces_w_hat():
    """End to end on the GPU: forward (W^), export (bit-planes, alpha*, z*),
    then the product from the export alone against the oracle's product of
    the oracle's own export, and against x W^T (Theorem 1)."""
    q, g = 3, 128
    raw, W, P, codes, _ = C.make_inputs(64, 2048, q, g, seed=4)
    what, codes1 = C.gpu_fwd(raw, P, codes, q, g, api.MAP_LOCAL_PERIODIC, 0, 2)
    planes, a_s, z_s = C.gpu_export(raw, P, codes1, q, g, api.EXPORT_REUSE_CODES)
    r_planes, r_as, r_zs, _ = O.export_bcq(W, P["delta"], P["zu"], P["alpha"], P["zb"], codes1, g)
    x = np.random.default_rng(5).standard_normal((3, 2048)).astype(F32)
    y = gpu_gemv(planes, a_s, z_s, x, g)
    ref = O.bcq_gemv(r_planes, r_as, r_zs, x, g)
    assert (np.abs(y - ref) <= TOL * mass(r_as, r_zs, x, g)).all()
    # Theorem 1: the same numbers as the quantizer's own output times x
    thm = x.astype(F64) @ what.astype(F64).T
    assert (np.abs(y - thm) <= 2 * TOL * mass(r_as, r_zs, x, g)).all()


def test_gemv_full_size_headline_matrix():
    """14336 x 4096, q = 3, g = 128 (the benchmark's export), every row."""
    q, g, out, n_in = 3, 128, 14336, 4096
    planes, a_star, z_star = random_export(out, n_in, q, g, seed=21)
    x = np.random.default_rng(2).standard_normal((1, n_in)).astype(F32)
    check(planes, a_star, z_star, x, g, label="14336x4096")


def test_gemv_full_size_70b_down_projection_sampled():
    """8192 x 28672: the oracle recomputes a sample of rows (rows are
    independent: each output is one row of the product)."""
    q, g, out, n_in = 3, 128, 8192, 28672
    planes, a_star, z_star = random_export(out, n_in, q, g, seed=22)
    x = np.random.default_rng(3).standard_normal((1, n_in)).astype(F32)
    y = gpu_gemv(planes, a_star, z_star, x, g)
    rows = np.array(sorted(set([0, 1, 4095, 4096, out - 1]) | set(np.random.default_rng(0).choice(out, 40).tolist())))
    ref = O.bcq_gemv(np.ascontiguousarray(planes[:, rows]), a_star[rows], z_star[rows], x, g)
    assert (np.abs(y[:, rows] - ref) <= TOL * mass(a_star[rows], z_star[rows], x, g)).all()


def test_gemv_rejects_a_small_workspace():
    d = C.dev()
    planes, a_star, z_star = random_export(16, 1024, 2, 64, seed=1)
    need = api.uq_bcq_gemv_workspace_bytes(16, 1024, 1)
    assert need == 2 * 16 * 4
    ws = torch.empty(need // 4 - 1, device=d)
    y = torch.empty(1, 16, device=d)
    with pytest.raises(api.UQError) as e:
        api.uq_bcq_gemv(torch.from_numpy(planes.view(np.int32)).to(d), torch.from_numpy(a_star).to(d),
                        torch.from_numpy(z_star).to(d), torch.zeros(1, 1024, device=d), y, 64, workspace=ws)
    assert e.value.status == api.UQ_ERR_ARG


def test_gemv_tensor_core_product_in_a_cuda_graph():
    """Captured products of three kinds (one slice, several slices, per-thread loads)
    replay with the bits of the plain calls, on inputs changed in between."""
    d = C.dev()
    for out, n_in, g, batch in ((300, 512, 64, 8), (2000, 8192, 128, 5), (129, 192, 64, 6)):
        planes, a_star, z_star = random_export(out, n_in, 3, g, seed=out)
        pd, ad, zd = torch.from_numpy(planes.view(np.int32)).to(d), torch.from_numpy(a_star).to(d), torch.from_numpy(z_star).to(d)
        x, y = torch.zeros(batch, n_in, device=d), torch.empty(batch, out, device=d)
        ws = torch.empty(api.uq_bcq_gemv_workspace_bytes(out, n_in, batch) // 4, device=d)
        api.uq_bcq_gemv(pd, ad, zd, x, y, g, workspace=ws)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            api.uq_bcq_gemv(pd, ad, zd, x, y, g, workspace=ws)
        for seed in (1, 2):
            x.copy_(torch.from_numpy(np.random.default_rng(seed).standard_normal((batch, n_in)).astype(F32)))
            graph.replay()
            torch.cuda.synchronize()
            got = y.clone()
            y.fill_(float("nan"))
            api.uq_bcq_gemv(pd, ad, zd, x, y, g, workspace=ws)
            assert torch.equal(got, y)
        api.uq_check_device()
