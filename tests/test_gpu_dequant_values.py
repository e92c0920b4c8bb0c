"""The dequantising epilogue at the ends of its range: codes that saturate on either side (-127, not -128), the activation on
negative, NaN and infinite results, scales of zero; every result type and order, against the oracle where it is finite."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_device, to_host_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [False, True])
@pytest.mark.parametrize("relu", [False, True])
@pytest.mark.parametrize("cd", ["i8", "bf16", "f16", "f32"])
@pytest.mark.parametrize("M,N,K", [(64, 96, 64), (288, 480, 512)])
def test_ends_of_the_range(M, N, K, cd, relu, cols):
    from paper_2104_08378_b200 import binding as sp
    rng = np.random.default_rng(M + N)
    a, bt = (rng.integers(-128, 128, s, dtype=np.int8) for s in ((M, K), (N, K)))
    vals, meta, _ = sp.compress(to_device(a, "i8"))
    acc = oracle.prune(a, "i8").astype(np.int32) @ bt.astype(np.int32).T
    scale = (rng.normal(size=M) * 1e-3).astype(np.float32)
    bias = rng.normal(size=M).astype(np.float32)
    scale[1::16], scale[2::16], scale[3::16], bias[4::16] = 0.0, 1.0, np.inf, np.nan
    out = sp.gemm_i8_dequant(vals, meta, to_device(bt, "i8"), torch.from_numpy(scale).cuda(), bias=torch.from_numpy(bias).cuda(),
                             relu=relu, out_scale=0.02, cd=cd, cd_col_major=cols)
    got = to_host_f64(out.t() if cols else out)
    with np.errstate(invalid="ignore"):
        value = scale[:, None].astype(np.float64) * acc + bias[:, None]
    fine = np.isfinite(value)
    ref, code = oracle.dequant(acc, np.where(np.isfinite(scale), scale, 1).astype(np.float32), np.nan_to_num(bias), relu=relu, out_scale=0.02)
    if cd == "i8":
        assert np.array_equal(got[fine], code[fine]) and got.min() >= (0 if relu else -127)
        assert (got[np.isnan(value)] == 0).all()
        assert (got[value == np.inf] == 127).all() and (got[value == -np.inf] == (0 if relu else -127)).all()
        return
    # one rounding to the type, one in FP32 before it (and half of FP16's smallest step)
    eps = {"bf16": 2.0 ** -8, "f16": 2.0 ** -11, "f32": 2.0 ** -23}[cd] + 2.0 ** -23
    in_range = fine & (np.abs(ref) < 6e4)
    assert (np.abs(got - ref)[in_range] <= eps * (np.abs(ref) + np.abs(bias[:, None]))[in_range] + 2.0 ** -24).all()
    assert (got[np.isnan(value)] == 0).all() if relu else np.isnan(got[np.isnan(value)]).all()
    assert (got[value == -np.inf] == (0 if relu else -np.inf)).all() and (got[value == np.inf] == np.inf).all()
