"""Single kernels and dispatch branches at the sizes and values where they can go wrong (edges of tiles, remainders,
the ends of their ranges), against the fp64 oracle.  Gates as in test_gpu_parity.py."""
import numpy as np
import pytest
import torch

from oracle import rehyat_oracle as orc
from paper_2601_04342_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2601_04342_b200 import build
    build.build()


def _forward(wl, x, layout="bhnd", **kw):
    from paper_2601_04342_b200 import binding
    op = binding.for_workload(wl, **kw)
    q, k, v = (x[n].cuda() for n in ("q", "k", "v"))
    if layout == "bnhd":
        q, k, v = (t.transpose(1, 2).contiguous() for t in (q, k, v))
    pq, pk = ({n: t.cuda() for n, t in x[m].items()} for m in ("phi_q", "phi_k"))
    y = op.forward(q, k, v, pq, pk, wl.T, wl.H, wl.W, wl.Tc, wl.To, layout=layout)
    assert op.status() == 0
    op.close()
    return (y.transpose(1, 2) if layout == "bnhd" else y).double().cpu().numpy()


def _oracle(wl, x, **kw):
    f = synth.to_f64(x)
    return orc.hybrid_direct(f["q"], f["k"], f["v"], f["phi_q"], f["phi_k"], wl.T, wl.HW, wl.Tc, wl.To, P=wl.P, **kw)


def _gate(y, ref, dtype):
    err = np.abs(y - ref)
    if dtype == "fp32":
        assert err.max() <= 1e-4, f"max-abs {err.max():.3e}"
        return
    assert err.max() <= 2e-2, f"max-abs {err.max():.3e}"
    worst = (err / (3e-3 + 2.0 ** -7 * np.abs(ref))).max()
    assert worst <= 1.0, f"internal gate exceeded x{worst:.2f}, max-abs {err.max():.3e}"
    assert np.sqrt((err ** 2).mean() / (ref ** 2).mean()) <= 1e-2


@pytest.mark.parametrize("act_hidden,act_out,P,Dp", [("gelu", "softplus", 1, 256), ("softplus", "elu1", 4, 96),
                                                     ("elu1", "relu", 3, 192), ("gelu", "relu", 2, 96)])
def test_activations_over_their_whole_range(act_hidden, act_out, P, Dp):
    """The activations of the tensor-core phi kernels with arguments from deep in the tails to well above zero
    (first layer of standard deviation 4 here, 0.2 in the other tests), parts that end inside 16 columns."""
    wl = synth.Workload("acts", 1, 2, 128, 5, 10, 20, 2, 1, "bf16", True, P=P, seed=synth.BASE_SEED + 401, phi_dim=Dp)
    x = synth.make_inputs(wl, v_frame_offsets=True)
    for m in ("phi_q", "phi_k"):
        x[m]["W1"] = (x[m]["W1"].float() * 18).to(torch.bfloat16)
    y = _forward(wl, x, act_hidden=act_hidden, act_out=act_out)
    _gate(y, _oracle(wl, x, act_hidden=act_hidden, act_out=act_out), "bf16")


# (dtype, d, heads, T, H, W, Tc, To, D_h, D', P, layers): the CUDA-core kernels.  Chunks that end inside tiles of 32, 64
# and 128 rows and keys, window shares of a key group that are empty, phi widths that end inside blocks of 8 to 32
# columns and slabs of 16 or 32, one and both shapes of the window kernel (336 tiles of 128 rows take the wide one).
@pytest.mark.parametrize("dtype,d,nh,T,H,W,Tc,To,Dh,Dp,P,layers", [
    ("fp32", 64, 2, 5, 1, 3, 1, 1, 8, 8, 1, 2), ("fp32", 128, 3, 4, 3, 11, 1, 2, 24, 40, 2, 3),
    ("fp32", 64, 24, 7, 10, 13, 1, 1, 128, 128, 2, 2), ("fp32", 128, 24, 7, 3, 43, 1, 0, 136, 200, 2, 2),
    ("fp32", 128, 2, 3, 8, 16, 1, 1, 256, 256, 4, 4), ("bf16", 64, 24, 7, 10, 13, 1, 1, 72, 104, 1, 2),
    ("bf16", 128, 2, 6, 5, 13, 2, 1, 40, 136, 2, 3), ("bf16", 64, 2, 4, 9, 17, 2, 1, 256, 8, 1, 2)])
def test_cuda_core_kernels(dtype, d, nh, T, H, W, Tc, To, Dh, Dp, P, layers):
    wl = synth.Workload("simt", 1, nh, d, T, H, W, Tc, To, dtype, dtype == "bf16", P=P, seed=synth.BASE_SEED + 402, phi_hidden=Dh,
                        phi_dim=Dp, phi_layers=layers)
    x = synth.make_inputs(wl, v_frame_offsets=True)
    _gate(_forward(wl, x, impl="simt"), _oracle(wl, x), dtype)


# fp32 windows on the tensor cores: one to seven key tiles of 64 with remainders, several items of a CTA one after the
# other with odd and even numbers of tiles, moving row maxima, both conventions for c.
@pytest.mark.parametrize("d,nh,T,HW,Tc,To,c_mode", [(64, 3, 4, 129, 1, 0, "rowmax"), (128, 2, 5, 65, 1, 1, "zero"), (64, 160, 3, 65, 1, 1, "rowmax"),
                                                    (128, 100, 6, 100, 3, 1, "rowmax"), (64, 61, 9, 43, 3, 2, "zero"), (64, 2, 3, 43, 1, 1, "rowmax"), (128, 7, 3, 150, 1, 2, "rowmax")])
def test_fp32_window_on_the_tensor_cores(d, nh, T, HW, Tc, To, c_mode):
    wl = synth.Workload("f32tc", 1, nh, d, T, 1, HW, Tc, To, "fp32", False, seed=synth.BASE_SEED + 404)
    x = synth.make_inputs(wl, v_frame_offsets=True)
    x["q"] = x["q"] * (2 if c_mode == "rowmax" else 0.5)
    _gate(_forward(wl, x, impl="auto", c_mode=c_mode), _oracle(wl, x, c_mode=c_mode), "fp32")


@pytest.mark.parametrize("where,value", [("k", -3.4e38), ("k", float("-inf")), ("v", float("inf")), ("q", float("nan")), ("v", 1e30),
                                         ("q", 2.0 ** 41)])
def test_fp32_values_that_cannot_be_split(where, value):
    """Values beyond what the split into bf16 parts carries are computed by the CUDA-core kernels, as if they were alone (the
    state sums of the two calls are split differently over CTAs: fp32 sums in another order)."""
    wl = synth.Workload("f32big", 1, 3, 128, 4, 10, 20, 1, 1, "fp32", False, seed=synth.BASE_SEED + 405)
    x = synth.make_inputs(wl)
    x[where][0, 1, 333, 5] = value
    np.testing.assert_allclose(_forward(wl, x, impl="auto"), _forward(wl, x, impl="simt"), rtol=1e-5, atol=1e-6)


# fp32 phi on the tensor cores: widths that end inside quarters of 64 and halves of 128 columns, chunks that end inside
# tiles of 128 tokens, several tiles of a CTA, all degrees and activations (more than one round of tiles of 32 on the SMs).
# The features are non-negative: with both signs the denominator of Eq. 5 may vanish and no tolerance holds.
@pytest.mark.parametrize("d,nh,T,HW,Tc,To,Dh,Dp,P,act_hidden,act_out", [
    (64, 60, 6, 150, 1, 0, 8, 8, 1, "relu", "relu"), (128, 60, 6, 150, 1, 0, 72, 136, 2, "gelu", "softplus"),
    (128, 40, 7, 129, 3, 1, 256, 256, 4, "relu", "relu"), (64, 40, 7, 100, 3, 2, 200, 192, 3, "elu1", "elu1"),
    (64, 4, 9, 400, 4, 1, 128, 128, 2, "relu", "relu"), (128, 6, 9, 410, 4, 1, 64, 64, 2, "identity", "softplus")])
def test_fp32_phi_on_the_tensor_cores(d, nh, T, HW, Tc, To, Dh, Dp, P, act_hidden, act_out):
    wl = synth.Workload("f32phi", 1, nh, d, T, 1, HW, Tc, To, "fp32", False, P=P, seed=synth.BASE_SEED + 406, phi_hidden=Dh, phi_dim=Dp)
    x = synth.make_inputs(wl, v_frame_offsets=True, phi_scale=2.0)
    y = _forward(wl, x, act_hidden=act_hidden, act_out=act_out)
    _gate(y, _oracle(wl, x, act_hidden=act_hidden, act_out=act_out), "fp32")
