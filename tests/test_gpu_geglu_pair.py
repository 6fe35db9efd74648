"""The packed GeGLU of the tcgen05 epilogue against the recipe, fp32 bit for bit, on every gate that it
takes (2^-60 to 2^60 of both signs, 2.0e9 values: its rounding of some quotients rests on the GPU's reciprocal), and
the gates around 2^-24, whose divisors are such ones, through the FFN block."""
import ctypes
import os
import struct
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def _bits(x):
    return struct.unpack("<I", struct.pack("<f", x))[0]


def test_every_gate(tmp_path):
    from paper_2608_28003_gb300 import build
    so = str(tmp_path / "geglu_sweep.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", os.path.join(HERE, "geglu_sweep.cu"), "-o", so],
                   check=True)
    sweep = ctypes.CDLL(so).geglu_sweep
    sweep.argtypes = [ctypes.c_uint32, ctypes.c_ulonglong, ctypes.c_float, ctypes.c_void_p]
    torch.zeros(1, device="cuda")
    span = _bits(2.0 ** 60) - _bits(2.0 ** -60)
    for sign in (0, 0x80000000):
        counts = torch.zeros(3, dtype=torch.int64, device="cuda")
        assert sweep(sign | _bits(2.0 ** -60), span, 1.0, counts.data_ptr()) == 0
        taken, wrong, at = counts.tolist()
        assert taken == span and wrong == 0, (taken, wrong, hex(at))


def test_gates_at_the_top_of_a_binade():
    from paper_2608_28003_gb300 import build
    build.build()
    from paper_2608_28003_gb300 import binding as B
    from oracle import geglu as OG
    H, F, M = 64, 64, 40
    # one nonzero input channel: the bf16 gates and ups are its products, exactly
    gates = np.float32(2.0) ** -24 * (1 + np.arange(F, dtype=np.float32) / 128)
    gates[F // 2:] *= -1
    wg = torch.zeros(F, H, dtype=torch.bfloat16)
    wg[:, 0] = torch.from_numpy(gates).to(torch.bfloat16)
    wu = torch.zeros(F, H, dtype=torch.bfloat16)
    wu[:, 0] = 1.0
    x = torch.zeros(M, H, dtype=torch.bfloat16)
    x[:, 0] = 1.0
    f = B.FfnWeights(H, F, gate_up_bf16=B.interleave_gate_up(wg.cuda(), wu.cuda()),
                     down_bf16=torch.zeros(H, F, dtype=torch.bfloat16, device="cuda"))
    _, h = B.ffn_block(f, B.W8A8_PREC_BF16, x.cuda(), want_h=True)
    want = torch.from_numpy(OG.geglu_f32(wg[:, 0].float().numpy(), np.ones(F, np.float32))).to(torch.bfloat16)
    assert torch.equal(h.cpu().view(torch.int16), want.view(torch.int16).expand(M, F))
