"""Loading new links into a context that already solved: its link copies and solver graphs are
kept and refilled, so every result must be the one a new context gives, bit for bit."""
import numpy as np
import pytest

from paper_1810_04201_gb300 import gen

pytestmark = pytest.mark.gpu
DIMS, KAPPA = (4, 4, 6, 8), 0.12


def configure(lat, U, recon, inner, recon_in):
    lat.set_gauge(U, recon=recon)
    if recon_in != recon:
        lat.set_link_compression(inner, recon_in)


def results(lat, b, inner, eo):
    fx = lat.new_field()
    lat.cg(KAPPA, lat.pack(b), fx, tol=1e-10, inner=inner, precondition=eo)
    fo = lat.new_field(inner)
    lat.apply(KAPPA, lat.pack(b, inner), fo, inner)
    return lat.unpack(fx), lat.unpack(fo, inner)


@pytest.mark.parametrize("inner,eo", [(0, 0), (1, 0), (1, 1), (2, 1), (3, 0)])
def test_new_links_give_what_a_new_context_gives(inner, eo):
    from paper_1810_04201_gb300 import wd
    U1, U2 = gen.haar_links(DIMS, seed=1), gen.haar_links(DIMS, seed=2)
    U3 = U2.copy()
    U3[1, 5] *= 1.0 + 2.0 ** -8  # not unitary: the FP64 links change their layout
    b = gen.gaussian_source(DIMS, seed=3)
    steps = [(U1, 18, 18), (U2, 18, 18), (U3, 18, 18), (U1, 18, 12), (U2, 18, 12), (U1, 12, 12), (U2, 18, 18), (U1, 8, 8)]
    lat = wd.Lattice(DIMS)
    for U, recon, recon_in in steps:
        recon_in = recon if inner == 0 else recon_in
        configure(lat, U, recon, inner, recon_in)
        fresh = wd.Lattice(DIMS)
        configure(fresh, U, recon, inner, recon_in)
        for got, want in zip(results(lat, b, inner, eo), results(fresh, b, inner, eo)):
            assert np.array_equal(got, want)


def test_a_stale_copy_is_refused_where_a_missing_one_is():
    from paper_1810_04201_gb300 import wd
    lat = wd.Lattice(DIMS)
    src = gen.gaussian_source(DIMS, seed=3)
    for seed in (1, 2):
        lat.set_gauge(gen.haar_links(DIMS, seed=seed))
        f, o = lat.pack(src, 1), lat.new_field(1)
        with pytest.raises(wd.WDError) as e:
            lat.normal_apply_noalloc(KAPPA, f, o, 1)
        assert e.value.status == 8
        lat.apply(KAPPA, f, o, 1)
        lat.normal_apply_noalloc(KAPPA, f, o, 1)


@pytest.mark.parametrize("on_device", [False, True])
def test_new_links_wait_for_operators_on_an_earlier_stream(on_device):
    """Operators queued on the stream that a context used before must still see the old links."""
    import torch
    from paper_1810_04201_gb300 import wd
    dims = (8, 8, 8, 12)
    U1, U2 = gen.haar_links(dims, seed=1), gen.haar_links(dims, seed=2)
    if on_device:
        U2 = torch.from_numpy(U2).cuda()
    src = gen.gaussian_source(dims, seed=3)
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    for prec in (0, 1):
        with torch.cuda.stream(one):
            lat = wd.Lattice(dims)
            lat.set_gauge(U1)
            f, want, got = lat.pack(src, prec), lat.new_field(prec), lat.new_field(prec)
            lat.apply(KAPPA, f, want, prec)
            one.synchronize()
            torch.cuda._sleep(200_000_000)  # about a tenth of a second before the operator starts
            lat.apply(KAPPA, f, got, prec)
        with torch.cuda.stream(two):
            lat.set_stream()
            lat.set_gauge(U2)
            lat.apply(KAPPA, f, lat.new_field(prec), prec)
        torch.cuda.synchronize()
        assert torch.equal(got, want)


def test_links_are_not_converted_inside_a_stream_capture():
    """A copy of the links that a capture would have to make is refused, as it always was for one
    that had to be allocated: it would only be filled when the graph runs."""
    import torch
    from paper_1810_04201_gb300 import wd
    U1, U2 = gen.haar_links(DIMS, seed=1), gen.haar_links(DIMS, seed=2)
    src = gen.gaussian_source(DIMS, seed=3)
    with torch.cuda.stream(torch.cuda.Stream()):
        lat = wd.Lattice(DIMS)
        lat.set_gauge(U1)
        f, out = lat.pack(src, 1), lat.new_field(1)
        lat.apply(KAPPA, f, out, 1)
        lat.set_gauge(U2)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=torch.cuda.current_stream()):
            out.zero_()
            with pytest.raises(wd.WDError) as e:
                lat.apply(KAPPA, f, out, 1)
        assert e.value.status == 8
        lat.apply(KAPPA, f, out, 1)
        fresh = wd.Lattice(DIMS)
        fresh.set_gauge(U2)
        want = fresh.new_field(1)
        fresh.apply(KAPPA, f, want, 1)
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        graph = torch.cuda.CUDAGraph()  # with the copy in place the operator is captured
        with torch.cuda.graph(graph, stream=torch.cuda.current_stream()):
            lat.apply(KAPPA, f, out, 1)
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)


def test_link_copies_that_the_new_configuration_does_not_use_are_given_back():
    """A configuration that works in another precision holds what a new context would: the copies
    kept for refilling go before others are allocated."""
    import torch
    from paper_1810_04201_gb300 import wd
    dims = (16, 16, 16, 16)  # a DF32 copy of the links is 38 MB
    U = torch.from_numpy(gen.haar_links((4, 4, 4, 4), seed=1)).cuda().repeat(1, 256, 1, 1).contiguous()

    def held(precs):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        lat = wd.Lattice(dims)
        for prec in precs:
            lat.set_gauge(U)
            lat.apply(KAPPA, src[prec], dst[prec], prec)
        torch.cuda.synchronize()
        n = free - torch.cuda.mem_get_info()[0]
        lat.close()
        return n

    one = wd.Lattice(dims)
    src, dst = [one.new_field(p) for p in range(4)], [one.new_field(p) for p in range(4)]
    held([1])
    assert held([3, 1]) <= held([1]) + (4 << 20)
    assert held([3, 2, 1, 2]) <= held([1]) + (4 << 20)
