"""Hops, which are launched as programmatic dependents of the kernel before them, where
that kernel is the caller's own: on the same stream, and on another one joined by an
event, eagerly and in a captured graph."""

import pytest

import gen
from gpu_util import to_device, to_planar

DIMS = (8, 8, 8, 8)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "ff64"])
@pytest.mark.parametrize("other", [False, True])
def test_source_written_just_before_the_hop(prec, other):
    import torch

    import paper_2303_08609_gb300 as weo

    wide = prec in ("f64", "ff64")
    psi = to_device(to_planar(gen.gaussian_spinor(DIMS, seed=1402)[0]), "f64" if wide else "f32")
    with weo.WilsonEO(DIMS, 0.13, to_device(gen.gauge_field(DIMS, "haar", seed=1401)), prec="f64" if wide else prec) as op:
        apply = op.apply_ff64 if prec == "ff64" else op.apply
        want = [apply((k + 1) * psi) for k in range(4)]
        x, y, z, factor = torch.empty_like(psi), torch.empty_like(psi), torch.empty_like(psi), torch.ones((), device="cuda")
        side = torch.cuda.Stream()

        def step():
            here = torch.cuda.current_stream()
            if other:
                side.wait_stream(here)
                with torch.cuda.stream(side):
                    torch.mul(psi, factor, out=x)
                here.wait_stream(side)
            else:
                torch.mul(psi, factor, out=x)
            apply(x, out=y)
            if other:  # and a hop beside another stream's kernel
                side.wait_stream(here)
                with torch.cuda.stream(side):
                    torch.neg(y, out=z)
                here.wait_stream(side)
            else:
                torch.neg(y, out=z)

        step()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step()
        for run in (step, graph.replay):
            for k in range(4):
                factor.fill_(k + 1.0)
                run()
                torch.cuda.synchronize()
                assert torch.equal(y, want[k]) and torch.equal(z, -want[k])
