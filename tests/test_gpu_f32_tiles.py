"""The fp32 GEMMs at the edges of their tiles (64 and 128 wide), k slices (16 deep) and
cluster splits along K (the projection's K is V, the update's T), with and without rows
that allow 16-byte accesses, against the fp64 oracle.

Bound: sums of up to 2600 fp32 products in a fixed order; the rounding of a random-sign sum
of n terms grows like sqrt(n) 2^-24 (3e-6 at 2600), and the fp32 parity tolerance 1e-5
covers the chain of three such products."""
import pytest
import torch

from helpers import f64, rel_frob
import synth
from synth import Workload
from test_gpu_parity import F32_TOL, check, gpu_step, oracle_step

pytestmark = pytest.mark.gpu

SHAPES = [
    (128, 64, 128, 64),       # whole tiles, one 64-column logits partial
    (129, 65, 257, 1001),     # one past a tile everywhere, unaligned rows
    (63, 260, 66, 2600),      # below one 64-tile of tokens, deep K in the projection
    (1100, 36, 70, 130),      # deep K in the update, a partial last vector
    (17, 1028, 12, 515),
]


@pytest.fixture(params=[64, 128])
def tile(fpo, request):
    """Either tile width, whichever the sizes would choose (64: they are small)."""
    fpo.set_simt_tile(request.param)
    yield request.param
    fpo.set_simt_tile(0)


@pytest.mark.parametrize("shape", SHAPES, ids=["T%dd%df%dV%d" % s for s in SHAPES])
def test_fp32_step_at_tile_edges(fpo, shape, tile):
    T, d, d_ff, V = shape
    wl = Workload("tiles32", T=T, d=d, d_ff=d_ff, V=V, layers=2, dtype="f32", targets="zipf",
                  lr=1e-2)
    inp = synth.make_all(wl)
    ref = oracle_step(wl, inp)
    runs = [gpu_step(fpo, wl, inp, algo=a, t_chunk=c) for a, c in ((2, 0), (1, 0), (2, 40))]
    check(runs[0], ref, inp, wl.lr, F32_TOL)
    fpo.set_simt_tile(192 - tile)
    runs.append(gpu_step(fpo, wl, inp, algo=2))
    # the order of a sum depends neither on the algorithm or the chunking nor on the tiles
    for r in runs[1:]:
        for a, b in zip([runs[0]["g"], runs[0]["lse"]] + runs[0]["G"] + runs[0]["W"],
                        [r["g"], r["lse"]] + r["G"] + r["W"]):
            assert torch.equal(a, b)


def test_fp32_gate_up_at_tile_edges(fpo, tile):
    T, d, d_ff = 130, 1030, 67
    gen = torch.Generator(device="cuda").manual_seed(5)
    r = lambda *s: torch.randn(*s, device="cuda", generator=gen)  # noqa: E731
    g, W3, a, b = r(T, d), 0.02 * r(d, d_ff), r(T, d_ff), r(T, d_ff)
    dA, dB = torch.empty_like(a), torch.empty_like(b)
    assert fpo.get_device_status(fpo.gate_up_signals(g, W3, a, b, dA, dB)) == fpo.OK
    e = g.double() @ W3.double()
    sg = torch.sigmoid(a.double())
    assert rel_frob(f64(dA), f64(e * b * sg * (1 + a * (1 - sg)))) < F32_TOL
    assert rel_frob(f64(dB), f64(e * a * sg)) < F32_TOL
    fpo.set_simt_tile(192 - tile)
    oA, oB = torch.empty_like(a), torch.empty_like(b)
    fpo.gate_up_signals(g, W3, a, b, oA, oB)
    assert torch.equal(dA, oA) and torch.equal(dB, oB)


def test_fp32_sizes_that_choose_128_tiles(fpo):
    """Without an override: a logits pass and a grouped update of more tiles of 64 than the
    SMs hold at once, odd everywhere, whose chunks of 40 tokens choose the tiles of 64."""
    wl = Workload("tiles32", T=777, d=131, d_ff=1027, V=5003, layers=6, dtype="f32",
                  targets="zipf", lr=1e-2)
    inp = synth.make_all(wl)
    runs = [gpu_step(fpo, wl, inp, t_chunk=0), gpu_step(fpo, wl, inp, t_chunk=40, grouped=False)]
    check(runs[0], oracle_step(wl, inp), inp, wl.lr, F32_TOL)
    assert torch.equal(runs[0]["g"], runs[1]["g"]) and torch.equal(runs[0]["lse"], runs[1]["lse"])
    assert all(torch.equal(a, b) for a, b in zip(runs[0]["W"], runs[1]["W"]))
