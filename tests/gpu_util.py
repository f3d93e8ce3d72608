"""Helpers shared by the GPU parity tests: feed one seeded input to both the CUDA
path (through the C ABI) and the CPU oracle, and compare; and read which kernels a call launches."""
import ctypes
import re

import numpy as np
import torch

import oracle
import paper_2607_02501_gb300 as emb
from workloads import activation_bits_np, weight_np


def to_dev_bf16(bits: np.ndarray) -> torch.Tensor:
    """bf16 device tensor holding exactly the given bit patterns."""
    t = torch.from_numpy(np.ascontiguousarray(bits).view(np.int16))
    return t.cuda().view(torch.bfloat16)


def bits_of(x: torch.Tensor) -> np.ndarray:
    return x.contiguous().view(torch.int16).cpu().numpy().view(np.uint16)


def gpu_quantize(fmt: int, W_host: np.ndarray) -> torch.Tensor:
    Wd = torch.from_numpy(np.ascontiguousarray(W_host, dtype=np.float32)).cuda()
    return emb.quantize(fmt, Wd)


def check_close(Y: np.ndarray, Yref: np.ndarray, B: np.ndarray, what: str = "") -> float:
    """|Y - Yref| <= B elementwise (B = 1e-3 sum|w x| + 1e-6); returns the largest
    error / sum|w x| ratio seen (for reporting)."""
    Y = np.asarray(Y, dtype=np.float64)
    err = np.abs(Y - Yref)
    assert np.isfinite(Y).all(), f"{what}: non-finite output"
    bad = err > B
    if bad.any():
        idx = np.argwhere(bad)[:5]
        raise AssertionError(f"{what}: {int(bad.sum())} of {bad.size} outside tolerance, "
                             f"first {idx.tolist()} err={err[bad][:5]} bound={B[bad][:5]}")
    mag = (B - 1e-6) / 1e-3
    with np.errstate(divide="ignore", invalid="ignore"):
        r = np.where(mag > 0, err / mag, 0.0)
    return float(r.max()) if r.size else 0.0


def run_case(fmt: int, M: int, N: int, K: int, seed: int):
    """Quantise + matmul on the GPU and in the oracle from the same seeded inputs."""
    W = weight_np(N, K, seed)
    Xb = activation_bits_np(M, K, seed + 1)
    img = gpu_quantize(fmt, W)
    X = to_dev_bf16(Xb)
    Y = emb.qmatmul(fmt, img, X, N)
    torch.cuda.synchronize()
    ref_img = oracle.quantize(fmt, W)
    Yref, B = oracle.qmatmul(fmt, ref_img, Xb, N, K)
    return Y.cpu().numpy(), Yref, B, img, ref_img


class _KernelNode(ctypes.Structure):
    """CUDA_KERNEL_NODE_PARAMS (second version) of the driver API."""
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def launches(call):
    """(kernel, template arguments, grid) of every kernel that `call()` enqueues on the current
    stream, in order of capture: the call is captured into a graph that never runs."""
    cu = ctypes.CDLL("libcuda.so.1")

    def ok(status):
        assert status == 0, f"driver call failed: {status}"

    stream, graph, count = torch.cuda.Stream(), ctypes.c_void_p(), ctypes.c_size_t(0)
    with torch.cuda.stream(stream):
        handle = ctypes.c_void_p(stream.cuda_stream)
        ok(cu.cuStreamBeginCapture_v2(handle, 1))  # thread-local mode
        try:
            call()
        finally:
            ok(cu.cuStreamEndCapture(handle, ctypes.byref(graph)))
    out = []
    try:
        ok(cu.cuGraphGetNodes(graph, None, ctypes.byref(count)))
        nodes = (ctypes.c_void_p * count.value)()
        ok(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(count)))
        for node in nodes:
            p, name = _KernelNode(), ctypes.c_char_p()
            ok(cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)))
            if p.func:
                ok(cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(p.func)))
            else:
                ok(cu.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(p.kern)))
            m = re.search(r"\d([a-z_]+_kernel)(?:I((?:L[a-z]\d+E)+)E)?", name.value.decode())
            args = re.findall(r"L[a-z](\d+)E", m.group(2) or "")
            out.append((m.group(1), tuple(int(a) for a in args), tuple(p.grid)))
    finally:
        ok(cu.cuGraphDestroy(graph))
    return out


def route(fmt: int, M: int, N: int, K: int, epilogue: int = 0):
    """The one launch of a layer of this size: (kernel, template arguments, grid)."""
    img, X = emb.empty_qweight(fmt, N, K), torch.empty(M, K, dtype=torch.bfloat16, device="cuda")
    Y = torch.empty(M, N, device="cuda")
    got = launches(lambda: emb.emb_qlayer_seq([(fmt, img, N, K, X, Y, epilogue)], M))
    assert len(got) == 1
    return got[0]


def layout_rows(fmt: int, img: torch.Tensor, N: int, K: int, rows) -> np.ndarray:
    """The packed image restricted to the given rows (codes rows, Q6_0 high-bit rows,
    scale rows), laid out as the image of that row subset (what the oracle produces for
    W[rows])."""
    rows = torch.as_tensor(np.asarray(rows), device=img.device, dtype=torch.long)
    n = rows.numel()
    rb = K if fmt == emb.EMB_Q8_0 else K // 2
    hb = K // 4 if fmt == emb.EMB_Q6_0 else 0
    r256 = lambda v: (v + 255) // 256 * 256
    codes = img[:N * rb].view(N, rb)[rows]
    hoff, sub_hoff = r256(N * rb), r256(n * rb)
    off = r256(hoff + N * hb) if hb else r256(N * rb)
    sub_off = r256(sub_hoff + n * hb) if hb else r256(n * rb)
    ldS = (K // 32 + 7) // 8 * 8
    scales = img[off:off + N * ldS * 2].view(N, ldS * 2)[rows]
    out = torch.zeros(sub_off + n * ldS * 2, dtype=torch.uint8, device=img.device)
    out[:n * rb] = codes.reshape(-1)
    if hb:
        out[sub_hoff:sub_hoff + n * hb] = img[hoff:hoff + N * hb].view(N, hb)[rows].reshape(-1)
    out[sub_off:] = scales.reshape(-1)
    return out.cpu().numpy()


def sample_rows(N: int, count: int, seed: int) -> np.ndarray:
    rng = np.random.default_rng(seed)
    rows = set([0, N - 1]) | set(rng.choice(N, size=min(count, N), replace=False).tolist())
    return np.array(sorted(rows), dtype=np.int64)
