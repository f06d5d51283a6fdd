"""A U(1) matvec prepares the operands of its own precision only: a split-TF32 call launches nothing
for the FP64 engine, an FP64 call nothing for the split-TF32 one, and a context that uses both
gives each the values it has alone."""
import pytest
import torch

from paper_1610_02244_gb300 import synth
from test_gpu_u1 import dev, problem, u1_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tnt():
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt as t
    return t


def test_operands_of_one_precision_only(tnt):
    qa, qb = synth.gaussian_sector_labels(192, 9, 2.0, 15), synth.gaussian_sector_labels(200, 9, 2.0, 17)
    Le, W1, W2, Re, th = u1_inputs(5, qa, qb, 4)
    p = problem(Le, W1, W2, Re, qa, qb)
    ctx = tnt.Context(0)
    x = ctx.u1_pack(p, dev(th))

    def run(precision, engine):
        ctx.set_fp64_gemm(engine)
        n = ctx.launch_count()
        y, _ = ctx.heff_apply_u1([p], x, precision=precision)
        return y, ctx.launch_count() - n

    run(1, 1)  # (the tiles of this block structure are chosen once)
    mixed = {engine: run(1, engine) for engine in (1, 0)}
    fp64 = {engine: run(0, engine) for engine in (1, 0)}
    assert torch.equal(mixed[0][0], mixed[1][0])
    assert mixed[1][1] == mixed[0][1]
    # two packs and five kernels of split TF32, two packs, W, gather and either products in FP64
    assert mixed[1][1] == 7 and fp64[0][1] == 6
    assert fp64[1][1] > fp64[0][1]  # slices: this structure is above the line
    assert torch.equal(run(0, 1)[0], fp64[1][0]) and torch.equal(run(1, 1)[0], mixed[1][0])
