"""A host frame's maps go back strip by strip while later strips come in: the host loops' bits with
the map read by a later loop on the host, with the map written again by a later loop, with two
maps, and with the map bound to the frame's own memory; on the first run, the captured run
and the replayed one."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
H, WD = 2051, 2049  # over 16 MiB: copied in strips


@pytest.fixture(scope="module")
def gao():
    from paper_1806_01430_gb300 import _build
    _build.build()
    import paper_1806_01430_gb300 as g
    return g


def program(kind):
    """Buffers, loops, the maps compared, the genes to run."""
    L, o = W.Loop, W.OUTPUT
    bufs = [W.Buffer("X", H, WD, role=W.INPUT), W.Buffer("B", H, WD, role=o), W.Buffer("G", H, WD, role=o),
            W.Buffer("q", 1, WD, role=o)]
    blur, gx = L(W.STENCIL3, [0], [1], flags=0), L(W.STENCIL3, [1], [2], flags=2)
    if kind == "rewritten":
        return bufs, [blur, gx, L(W.RELU, [2], [1]), L(W.COLMAX, [1], [3])], (1, 2, 3), (0b1111, 0b0111)
    return bufs, [blur, gx, L(W.COLMAX, [1], [3])], (1, 2, 3), (0b111, 0b011, 0b001, 0b101)


@pytest.mark.parametrize("kind", ["maps", "rewritten"])
@pytest.mark.parametrize("fuse", [0, 1])
def test_maps_copied_back_by_strip(gao, kind, fuse):
    bufs, loops, maps, genes = program(kind)
    X = np.random.default_rng(5).standard_normal((H, WD)).astype(np.float32)
    p = gao.prog_create(bufs, loops, fuse_chains=fuse)
    gao.prog_set_input(p, 0, X)
    gao.prog_run(p, 0)
    want = {b: gao.prog_output(p, b).copy() for b in maps}
    for gene in genes:
        for _ in range(3):
            gao.prog_run(p, gene)
            for b in maps:
                assert np.array_equal(gao.prog_output(p, b).view(np.uint32), want[b].view(np.uint32)), (gene, b)
    gao.prog_destroy(p)


@pytest.mark.parametrize("shift", [0, 64 * WD])
def test_map_bound_over_the_frame(gao, shift):
    """The blurred map bound to the frame's memory, or to memory that overlaps it from `shift`
    values on."""
    torch = pytest.importorskip("torch")
    bufs, loops, _, _ = program("maps")
    n = H * WD
    X = np.random.default_rng(6).standard_normal(n).astype(np.float32)
    p = gao.prog_create(bufs, loops)
    gao.prog_set_input(p, 0, X.reshape(H, WD))
    gao.prog_run(p, 0)
    want = gao.prog_output(p, 1).copy()
    both = torch.empty(n + shift).pin_memory()
    gao.prog_bind_host(p, 0, both[shift:shift + n].view(H, WD))
    gao.prog_bind_host(p, 1, both[:n].view(H, WD))
    for _ in range(3):
        both[shift:shift + n] = torch.from_numpy(X)
        gao.prog_run(p, 0b111)
        assert np.array_equal(both[:n].numpy().view(np.uint32), want.ravel().view(np.uint32))
    gao.prog_destroy(p)
