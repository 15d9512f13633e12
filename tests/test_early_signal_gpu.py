"""Calls behind a caller's kernel that signals its dependents before it writes.

A kernel may execute griddepcontrol.launch_dependents at once and write its results
later: a programmatic dependent then starts meanwhile, and sees those results only
after its own griddepcontrol.wait.  Here such a kernel copies every input of a call
into place (after some 20 us), and the call gives the same bits as on inputs that were
there long before.  The inputs alternate between two problems of one shape, so that a
value read too early is one of the other problem.
"""
import ctypes
import subprocess

import pytest
import torch

from paper_2606_03075_gb300 import synth

import _parity as P

pytestmark = pytest.mark.gpu

_SOURCE = r"""
#include <cuda_runtime.h>
#include <stdint.h>
__global__ void early_copy_kernel(uint4* dst, const uint4* src, long long n, int clocks) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long c0 = clock64();
    for (int i = 0; i < 1000000 && clock64() - c0 < clocks; ++i) {}
    for (long long i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        dst[i] = src[i];
}
extern "C" int early_copy(void* dst, const void* src, long long bytes, void* stream) {
    early_copy_kernel<<<4, 256, 0, (cudaStream_t)stream>>>((uint4*)dst, (const uint4*)src, bytes / 16,
                                                           40000);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def api():
    assert torch.cuda.is_available(), "the GPU tests need a CUDA device"
    from paper_2606_03075_gb300 import build
    build.build()
    from paper_2606_03075_gb300 import api as _api
    return _api


@pytest.fixture(scope="module")
def early_copy(tmp_path_factory):
    from paper_2606_03075_gb300 import build
    d = tmp_path_factory.mktemp("early")
    (d / "early.cu").write_text(_SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-o",
                    str(d / "early.so"), str(d / "early.cu")], check=True)
    fn = ctypes.CDLL(str(d / "early.so")).early_copy
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p]

    def copy(dst, src):
        assert fn(dst.data_ptr(), src.data_ptr(), dst.numel(),
                  torch.cuda.current_stream().cuda_stream) == 0
    return copy


def _shape(name, L, H_q, H_kv, d, vision, text, window="all_text"):
    """Two problems of one shape whose vision keys stand at other positions."""
    return [synth.custom(f"{name}{head}", L, H_q, H_kv, d,
                         [("text", head), ("vision", vision), ("text", text - head)], window=window)
            for head in (9, 31)]


SHAPES = {
    "packed": _shape("packed", 2, 8, 8, 64, 300, 60),
    "pairs": _shape("pairs", 2, 12, 2, 128, 500, 90),
    "many_heads": _shape("many_heads", 16, 32, 32, 64, 200, 40),
}


def _inputs(api, wl, kind, seed, opts):
    """Everything the call reads, by name."""
    inp = synth.generate_prefill(wl, seed=seed)
    dev = P.device_inputs(inp)
    desc = api.desc_for_workload(wl, **opts)
    dev["q_all"] = torch.from_numpy(inp["q_all"]).cuda().view(torch.bfloat16)
    if kind == "evict_with_stats":
        dev["stats"] = torch.empty((wl.L, wl.H_q, wl.n_win, 3), device="cuda")
        api.tgvkv_prefill(desc, dev["q_all"], dev["k"], dev["v"], dev["modality"], dev["text_pos"],
                          torch.empty_like(dev["q_all"]), dev["q"], dev["stats"],
                          api.new_workspace(desc))
    if kind == "select_compact":
        out = api.alloc_outputs(desc, 0.2)
        api.tgvkv_evict(desc, dev["q"], dev["k"], dev["v"], dev["modality"], dev["text_pos"],
                        dev["w"], 0.2, out, api.new_workspace(desc))
        dev["scores"], dev["budgets"] = out.scores, out.budgets
    if kind == "decode":
        dev["q_dec"] = dev["q_all"][:, :, -1].contiguous()
        n = wl.L * wl.H_kv
        step = torch.arange(n + 1, device="cuda") * (wl.N - 1 - seed)
        dev["offsets"] = step + seed
    names = {"evict": "q k v modality text_pos w", "evict_with_stats": "q k v modality text_pos w stats",
             "select_compact": "scores budgets k v modality", "decode": "q_dec k v offsets",
             "prefill": "q_all k v modality text_pos"}[kind].split()
    return {n: dev[n] for n in names}


def _call(api, desc, kind, t, ws):
    if kind == "decode":
        o = torch.zeros((desc.L, desc.H_q, desc.d), device="cuda")
        return lambda: api.tgvkv_decode(desc, t["q_dec"], t["k"].view(-1, desc.d),
                                        t["v"].view(-1, desc.d), t["offsets"], o, ws), [o]
    if kind == "prefill":
        o = torch.zeros_like(t["q_all"])
        qt = torch.zeros((desc.L, desc.H_q, desc.n_win, desc.d), dtype=torch.bfloat16, device="cuda")
        st = torch.zeros((desc.L, desc.H_q, desc.n_win, 3), device="cuda")
        return lambda: api.tgvkv_prefill(desc, t["q_all"], t["k"], t["v"], t["modality"], t["text_pos"],
                                         o, qt, st, ws), [o, qt, st]
    out = api.alloc_outputs(desc, 0.2)
    res = [out.scores, out.tvb_stat, out.budgets, out.offsets, out.idx, out.k_out, out.v_out]
    if kind == "select_compact":
        return lambda: api.tgvkv_select_compact(desc, t["scores"], None, t["budgets"], t["modality"],
                                                t["k"], t["v"], out.offsets, out.idx, out.k_out,
                                                out.v_out, ws), res[3:]
    if kind == "evict_with_stats":
        return lambda: api.tgvkv_evict_with_stats(desc, t["q"], t["k"], t["v"], t["modality"],
                                                  t["text_pos"], t["w"], 0.2, t["stats"], out, ws), res
    return lambda: api.tgvkv_evict(desc, t["q"], t["k"], t["v"], t["modality"], t["text_pos"], t["w"],
                                   0.2, out, ws), res


@pytest.mark.parametrize("shape,kind,opts", [
    ("packed", "evict", {}), ("pairs", "evict", {}), ("many_heads", "evict", {}),
    ("pairs", "evict", dict(weights="eq7", basis="all", keep_first=4)),
    ("packed", "evict_with_stats", {}), ("pairs", "evict_with_stats", {}),
    ("packed", "select_compact", {}), ("many_heads", "select_compact", {}),
    ("packed", "select_compact", dict(keep_first=2)),
    ("packed", "decode", {}), ("many_heads", "decode", {}), ("pairs", "prefill", {}),
])
def test_inputs_written_after_an_early_signal(api, early_copy, shape, kind, opts):
    both = SHAPES[shape]
    desc = api.desc_for_workload(both[0], **opts)
    ws = api.new_workspace(desc)
    sets = [_inputs(api, wl, kind, s, opts) for s, wl in enumerate(both)]
    # the inputs side by side in one buffer, 256 bytes apart
    place, end = {}, 0
    for n, x in sets[0].items():
        place[n] = end
        end += (x.numel() * x.element_size() + 255) // 256 * 256
    staged = []
    for s in sets:
        flat = torch.zeros(end, dtype=torch.uint8, device="cuda")
        for n, x in s.items():
            flat[place[n]:place[n] + x.numel() * x.element_size()] = x.contiguous().view(-1).view(torch.uint8)
        staged.append(flat)
    live = torch.empty(end, dtype=torch.uint8, device="cuda")
    t = {n: live[place[n]:place[n] + x.numel() * x.element_size()].view(x.dtype).view(x.shape)
         for n, x in sets[0].items()}
    call, outs = _call(api, desc, kind, t, ws)
    ref = []
    for flat in staged:
        live.copy_(flat)
        for x in outs:
            x.zero_()
        torch.cuda.synchronize()
        call()
        torch.cuda.synchronize()
        ref.append([x.clone() for x in outs])
    assert not all(torch.equal(a, b) for a, b in zip(*ref))
    for i in range(8):
        for x in outs:      # (what a call does not write stays zero)
            x.zero_()
        early_copy(live, staged[i % 2])
        call()
        got = [x.clone() for x in outs]
        assert api.tgvkv_status(ws) == 0
        for a, b in zip(got, ref[i % 2]):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
