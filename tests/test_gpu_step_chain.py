"""Steps launched back to back (each kernel may take its place while the one before drains) give
what steps with a wait between them give, bit for bit, on rows of every kind of length."""
import numpy as np
import pytest
import torch

from paper_1507_02518_gb300 import lb, workloads

pytestmark = pytest.mark.gpu
SHAPES = [(4, 3, 3), (30, 5, 4), (64, 6, 5), (66, 9, 7), (130, 3, 11), (33, 7, 6), (128, 128, 30)]


def begin(lat, shape, near):
    nx, ny, nz = shape
    z, y, x = np.meshgrid(*(np.arange(n) * 2 * np.pi / n for n in (nz, ny, nx)), indexing="ij")
    u = 0.04 * np.stack([np.sin(y) * np.cos(z), np.sin(z) * np.cos(x), np.sin(x) * np.cos(y)])
    if near:  # from equilibrium: the first steps send nodes through the FP64 pass
        lat.init_field(None, u)
    else:
        import oracle
        f = oracle.init_equilibrium(np.ones((nz, ny, nx)), u)
        lat.set_populations(f * (1 + 1e-3 * workloads.population_noise(nx, ny, nz, seed=3)))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("scheme", ["pull", "aa"])
@pytest.mark.parametrize("variant", ["d+t+q", "cd+ct+cq"])
@pytest.mark.parametrize("near", [False, True])
def test_back_to_back_steps(shape, storage, scheme, variant, near):
    steps = 7
    out = []
    for apart in (False, True):
        lat = lb.Lattice(*shape, nu=1e-3, storage=storage, scheme=scheme, variant=variant)
        begin(lat, shape, near)
        if apart:
            for _ in range(steps):
                lat.step(1)
                torch.cuda.synchronize()
        else:
            lat.step(steps)
        out.append(lat.get_populations())
    assert np.array_equal(out[0], out[1])


def test_two_streams_do_not_mix():
    """Two boxes stepped alternately on two streams."""
    ref = []
    lats = []
    for k in range(2):
        lat = lb.Lattice(64, nu=1e-3 * (k + 1), storage="f32", scheme="aa")
        begin(lat, (64, 64, 64), True)
        lat.step(40)
        ref.append(lat.get_populations())
        lats.append(lb.Lattice(64, nu=1e-3 * (k + 1), storage="f32", scheme="aa",
                               stream=torch.cuda.Stream()))
        begin(lats[k], (64, 64, 64), True)
    for _ in range(20):
        for lat in lats:
            lat.step(2)
    for k in range(2):
        assert np.array_equal(lats[k].get_populations(), ref[k])


def test_steps_in_a_captured_graph():
    lat = lb.Lattice(48, nu=1e-3, storage="f32", scheme="aa", stream=torch.cuda.Stream())
    begin(lat, (48, 48, 48), False)
    want = lb.Lattice(48, nu=1e-3, storage="f32", scheme="aa")
    begin(want, (48, 48, 48), False)
    want.step(12)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=lat.stream):
        lat.step(4)
    lb.lb_set_time(lat.ctx, 0)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(lat.get_populations(), want.get_populations())


@pytest.mark.parametrize("nx,variant", [(128, "d+t+q"), (130, "d+t+q"), (131, "d+t+q"), (256, "cd+ct+cq")])
@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("scheme", ["pull", "aa"])
def test_boxes_larger_than_l2(nx, variant, storage, scheme):
    """Populations over 129 MB take the kernels that prefetch a wave ahead; the same bits as the
    one-node kernel's (central moments, which have no such kernel here: as steps apart)."""
    ny, nz = 101, {"f32": 100, "f16": 200}[storage]
    P = nx * ny * nz
    assert 27 * P * {"f32": 4, "f16": 2}[storage] > 129 << 20
    u = 0.04 * torch.randn(3, nz, ny, nx, generator=torch.Generator("cuda").manual_seed(1),
                           dtype=torch.float64, device="cuda").clamp(-3, 3)
    out = []
    for kernel in ("auto", "direct"):
        lat = lb.Lattice(nx, ny, nz, nu=1e-3, storage=storage, scheme=scheme, variant=variant)
        if variant == "d+t+q":
            lat.set_kernel(kernel)
        lat.init_field(None, u)
        for n in ((3,) if kernel == "auto" else (1, 1, 1)):
            lat.step(n)
            torch.cuda.synchronize()
        f = torch.empty((27, nz, ny, nx), dtype=torch.float64, device="cuda")
        lb.lb_get_populations(lat.ctx, f.data_ptr(), True)
        out.append(f)
        del lat
    assert torch.equal(out[0], out[1])
