"""The relative error of a tensor that does not start on a 16-byte boundary (mode-0 size a multiple of
four, where the aligned kernels would load 16 bytes at a time) against the oracle, 1e-5 of the error."""
import numpy as np
import pytest

import tt_oracle as O
from paper_2309_08093_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_08093_gb300 import build as _build  # noqa: E402

_build.build()
from paper_2309_08093_gb300 import lib  # noqa: E402


@pytest.mark.parametrize("dtype,offset", [("f32", 1), ("f32", 2), ("f64", 1), ("bf16", 1), ("bf16", 4), ("fp8", 1), ("fp8", 8)])
def test_rel_error_off_the_16_byte_grid(dtype, offset):
    dims, ranks = (32, 12, 9), (1, 4, 3, 1)
    true = synth.random_tt(dims, ranks, 3)
    a = synth.add_noise(synth.contract_cores(true), 0.05, np.random.default_rng(4))
    flat, scales, exact = synth.quantize(a, dtype)
    A = lib.device_tensor(np.concatenate([np.zeros(offset, flat.dtype), flat]), dtype)[offset:]
    sc = torch.from_numpy(scales).cuda() if scales is not None else None
    ctx = lib.Context(dims, ranks, 64, 1e-3, 5, dtype)
    got = ctx.tt_rel_error(A, lib.device_cores(true), sc)
    ref = O.rel_error(exact, [np.asarray(g, np.float32).astype(np.float64) for g in true])
    assert abs(got - ref) <= 1e-5 * ref
    ctx.close()
