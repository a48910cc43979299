"""lb_conservation_static over its node ranges: fields of one node, at the edges of a range, of every range, and of a
thread's strip of loads, with and without a mask, against numpy sums of the same FP64 values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
              (0, 1, -1), (0, -1, 1)])


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("dims", [(1, 1, 1), (1023, 1, 1), (32, 32, 1), (25, 41, 1), (2049, 1, 1), (257, 5, 7), (64, 32, 32), (96, 32, 32), (97, 33, 32)])
def test_sums_over_node_ranges(dims, masked):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_3915_gb300 import lbsc
    nx, ny, nz = dims
    rng = np.random.Generator(np.random.PCG64(nx + ny + nz))
    n = rng.uniform(0.01, 0.06, size=(2, 19, nz, ny, nx))
    solid = (rng.uniform(size=(nz, ny, nx)) < 0.3).astype(np.uint8) if masked else np.zeros((nz, ny, nx), np.uint8)
    dn, ds = torch.from_numpy(n).cuda(), torch.from_numpy(solid).cuda()
    out = torch.full((8,), float("nan"), dtype=torch.float64, device="cuda")

    def sums():
        lbsc.conservation_static(dn.data_ptr(), ds.data_ptr() if masked else None, nx, ny, nz, out.data_ptr())
        return out.cpu().numpy()

    got = sums()
    fluid = n[:, :, solid == 0]
    m = fluid.sum(2)
    ref = np.array([m[0].sum(), m[1].sum(), *(C.T @ m.sum(0)), 0.0, (solid == 0).sum(), 0.0])
    # FP64 sums of N positive values in another order: N 2^-53 at most
    assert np.abs(got - ref).max() <= n.size * 2.0 ** -53 * max(1.0, m.sum())
    assert got[5] == 0 and got[6] == ref[6]
    # values that are not finite are counted, on fluid nodes only
    dn[1, 4, nz - 1, ny - 1, nx - 1] = float("nan")
    dn[0, 0, 0, 0, 0] = float("inf")
    want = int(solid[-1, -1, -1] == 0) + int(solid[0, 0, 0] == 0)
    got = sums()
    assert got[5] == want and got[6] == ref[6]
    assert np.isfinite(got[:5]).all() == (want == 0)


def test_sums_of_values_far_apart():
    """Values over the whole range of exponents and both signs (the integer sums align them): as near to the exact sum
    (fractions) as FP64 addition in any order is held to."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from fractions import Fraction

    from paper_0910_3915_gb300 import lbsc
    nx, ny, nz = 61, 7, 3
    rng = np.random.Generator(np.random.PCG64(8))
    for scale in (lambda: rng.uniform(-300, 290), lambda: rng.uniform(-3, 3), lambda: -310.0, lambda: rng.uniform(-320, -290)):
        n = np.zeros((2, 19, nz, ny, nx))
        for k in range(19):
            e = scale()
            n[:, k] = rng.choice([-1.0, 1.0], size=(2, nz, ny, nx)) * 10.0 ** (e + rng.uniform(-12, 12, size=(2, nz, ny, nx)).clip(-325 - e, 300 - e))
        dn = torch.from_numpy(n).cuda()
        out = torch.zeros(8, dtype=torch.float64, device="cuda")
        lbsc.conservation_static(dn.data_ptr(), None, nx, ny, nz, out.data_ptr())
        got = out.cpu().numpy()
        flat = [[[Fraction(float(x)) for x in n[a, k].ravel()] for k in range(19)] for a in range(2)]
        tot = [[sum(v) for v in f] for f in flat]
        mag = [[sum(abs(x) for x in v) for v in f] for f in flat]
        want = [sum(tot[0]), sum(tot[1])] + [sum(int(C[k][d]) * tot[a][k] for a in range(2) for k in range(19)) for d in range(3)]
        size = sum(mag[0]) + sum(mag[1])
        for g, w in zip(got[:5], want):
            assert abs(Fraction(float(g)) - w) <= n.size * Fraction(2) ** -53 * size + Fraction(2) ** -1070
        assert got[5] == 0 and got[6] == nx * ny * nz


@pytest.mark.parametrize("masked", [False, True])
def test_a_large_field_without_finite_values_is_counted(masked):
    """The largest field there may be, every value NaN (a run that blew up): 38 values a fluid node, above 2^31 of them."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_3915_gb300 import lbsc
    nx, ny, nz = 512, 512, 256
    if torch.cuda.mem_get_info()[0] < 24e9:
        pytest.skip("the field takes 20.4 GB")
    n = torch.full((2, 19, nz, ny, nx), float("nan"), dtype=torch.float64, device="cuda")
    solid = torch.zeros((nz, ny, nx), dtype=torch.uint8, device="cuda")
    if masked:
        solid[0] = solid[-1] = 1
    out = torch.zeros(8, dtype=torch.float64, device="cuda")
    lbsc.conservation_static(n.data_ptr(), solid.data_ptr() if masked else None, nx, ny, nz, out.data_ptr())
    got = out.cpu().numpy()
    fluid = nx * ny * (nz - 2 * masked)
    assert got[5] == 38 * fluid and got[6] == fluid
    assert np.isnan(got[:5]).all()
    del n, solid
    torch.cuda.empty_cache()


def test_sums_captured_in_a_graph():
    """Under stream capture (the second kernel is launched dependently on the first): replayed twice on changed inputs, with
    a second call in the same capture, the sums are those of calls outside a capture, bit for bit."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0910_3915_gb300 import lbsc
    dims = [(97, 33, 32), (64, 9, 5)]
    n = [torch.rand((2, 19, nz, ny, nx), dtype=torch.float64, device="cuda") for nx, ny, nz in dims]
    out = [torch.zeros(8, dtype=torch.float64, device="cuda") for _ in dims]

    def sums():
        for a, (nx, ny, nz), o in zip(n, dims, out):
            lbsc.conservation_static(a.data_ptr(), None, nx, ny, nz, o.data_ptr())

    sums()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sums()
    for k in range(2):
        for a in n:
            a.mul_(0.5).add_(0.01 * k)
        sums()
        torch.cuda.synchronize()
        want = [o.cpu().numpy().copy() for o in out]
        for o in out:
            o.zero_()
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        for o, w in zip(out, want):
            assert np.array_equal(o.cpu().numpy(), w)
