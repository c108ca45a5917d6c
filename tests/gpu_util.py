"""Helpers shared by the GPU parity tests: move generated inputs to the device, call through the C ABI."""
import numpy as np
import torch

import paper_2609_27396_b200 as dp


def dev_bf16(bits: np.ndarray) -> torch.Tensor:
    return torch.from_numpy(np.ascontiguousarray(bits).view(np.int16)).cuda().view(torch.bfloat16)


def host_bits(t: torch.Tensor) -> np.ndarray:
    return t.detach().cpu().contiguous().view(torch.int16).numpy().view(np.uint16)


def run_attention(inp, *, out_dtype=torch.float32, want_lse=True, with_blk=True, **kw):
    sh = inp.shape
    args = [dev_bf16(x) for x in (inp.q, inp.k_ctx, inp.v_ctx)]
    ks, vs = dev_bf16(inp.k_spine), dev_bf16(inp.v_spine)
    kb, vb = (dev_bf16(inp.k_blk), dev_bf16(inp.v_blk)) if with_blk else (None, None)
    res = dp.draft_all_boundaries(args[0], args[1], args[2], [int(x) for x in inp.ctx_offsets], ks, vs, kb, vb,
                                  prefix_base=sh.prefix_base, out_dtype=out_dtype, want_lse=want_lse, **kw)
    torch.cuda.synchronize()
    return res


def run_verify(v, mode):
    kw = {}
    if mode == 1:
        kw = dict(draft_probs=torch.from_numpy(v.draft_probs).cuda(), uniforms=torch.from_numpy(v.uniforms).cuda())
    res = dp.verify_select(torch.from_numpy(v.target).cuda(), torch.from_numpy(v.draft_tokens).cuda(),
                           dev_bf16(v.reps) if v.reps is not None else None, mode=mode, **kw)
    torch.cuda.synchronize()
    return res


def check_verify(res, ref):
    for k in ("accept_len", "bonus", "gather_idx", "out_tokens"):
        assert np.array_equal(res[k].cpu().numpy(), ref[k]), k
    if ref["selected"] is not None:
        assert np.array_equal(host_bits(res["selected"]), ref["selected"])
    assert int(res["status"].item()) == ref["status"]


def compile_native(tmp_path, text, without=None):
    """A library of this CUDA source, with the library's own flags and headers, loaded.  without: linked with the library's other objects but this one."""
    import ctypes
    import os
    import subprocess
    from paper_2609_27396_b200 import build
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

    def run(*cmd):
        r = subprocess.run([nvcc, *cmd], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr

    def compile_one(src, obj):
        run(*build.NVCC_FLAGS, "-I", build.CSRC, "-c", "-o", str(obj), str(src))

    src, lib = tmp_path / "native.cu", tmp_path / "native.so"
    src.write_text(text)
    objects = [tmp_path / "native.o"]
    compile_one(src, objects[0])
    for s in build.sources() if without else []:
        name = os.path.basename(s)[:-3]
        if name != without:
            obj = os.path.join(build.OBJ, name + ".o")
            if not os.path.exists(obj):
                obj = tmp_path / (name + ".o")
                compile_one(s, obj)
            objects.append(obj)
    run("-shared", *build.NVCC_FLAGS[:2], "-o", str(lib), *map(str, objects))
    return ctypes.CDLL(str(lib))
