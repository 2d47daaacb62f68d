"""What the kernels read before the kernel in front has ended is read again when it has: an engine's kernel that
releases its dependents at once may write a call's inputs until it ends."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import parity_util as pu
from paper_2503_17922_b200 import binding, build
from paper_2503_17922_b200 import workloads as wl

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def early_write(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("early") / "libearly.so")
    subprocess.check_call([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC", "-shared", "-o", so,
                           os.path.join(HERE, "early_writer.cu")])
    lib = ctypes.CDLL(so)

    def write(dst, src, stream):
        assert lib.early_write(ctypes.c_void_p(dst.data_ptr()), ctypes.c_void_p(src.data_ptr()), dst.numel(), 40,
                               ctypes.c_void_p(stream.cuda_stream)) == 0
    return write


@pytest.mark.parametrize("entry", ["select", "gather", "inplace"])
@pytest.mark.parametrize("l_obs", [16, 64], ids=["64rows", "256rows"])
def test_lengths_that_the_kernel_in_front_writes_last(early_write, entry, l_obs):
    """The device copy of cu_seqlens holds another split until just before the call: the call goes by what is there when the
    kernel in front has ended."""
    w = wl.scaled(wl.llama8b_single_group(), name="early", dtype="bf16", batch=3, n_layers=2, gamma=2, n_q_heads=8, n_kv_heads=2,
                  head_dim=128, max_seqlen=2500, l_obs=l_obs, window=8, top_p=4, budget_frac=0.2, n_planted=0, config_id=9, ragged=True)
    grp = wl.make_group(w, 0)
    ref = pu.run_gpu_group(w, grp)
    prob = ref["prob"]
    now = prob.cu_dev.clone()
    other = now.clone()
    other[1:-1] -= 301
    q = binding.to_device(grp["q_obs"])
    stream = torch.cuda.Stream()
    for _ in range(5):
        ks, vs = ([binding.to_device(x) for x in grp[name]] for name in ("k_layers", "v_layers"))
        out, work = prob.alloc_outputs(w.gamma, fill_byte=pu.FILL_BYTE), prob.alloc_workspace()
        idx = torch.from_numpy(ref["window_idx"]).cuda()
        before = [binding.to_host_bits(t) for t in ks + vs]
        prob.cu_dev.copy_(other)
        torch.cuda.synchronize()
        early_write(prob.cu_dev, now, stream)
        if entry == "select":
            binding.wkv_select_leader_windows(prob, q, ks[0], out["window_scores"], out["window_idx"], out["kept_len"], work, stream=stream)
        elif entry == "gather":
            binding.wkv_gather_kv(prob, ks, vs, idx, out["k_out"], out["v_out"], keep_capacity=out["keep_capacity"], stream=stream)
        else:
            binding.wkv_compact_kv_inplace(prob, ks, vs, idx, stream=stream)
        torch.cuda.synchronize()
        if entry == "select":
            assert binding.device_status(work) == 0
            for name in ("window_scores", "window_idx", "kept_len"):
                np.testing.assert_array_equal(out[name].cpu().numpy(), ref[name])
        for name, got in (("k_out", ks), ("v_out", vs)):
            for l in range(w.gamma):
                if entry == "gather":
                    np.testing.assert_array_equal(binding.to_host_bits(out[name][l]), ref[name][l])
                elif entry == "inplace":
                    rows, old = binding.to_host_bits(got[l]), before[l + (w.gamma if name == "v_out" else 0)]
                    for b in range(w.batch):
                        lo, hi = int(grp["cu_seqlens"][b]), int(grp["cu_seqlens"][b + 1])
                        for h in range(w.n_kv_heads):
                            kept = int(ref["kept_len"][b, h])
                            np.testing.assert_array_equal(rows[lo:lo + kept, h], ref[name][l][b, h, :kept])
                            np.testing.assert_array_equal(rows[lo + kept:hi, h], old[lo + kept:hi, h])
