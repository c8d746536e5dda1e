"""What a call reads and writes is ordered behind the kernel in front of it on the stream, whatever that kernel is.

The calls are launched as programmatic dependents.  A kernel of the caller's may let such dependents start long before it has done
its work; a call behind it then has to wait, however long that takes, and find what the kernel wrote in the end.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from oracle import rmsmp_oracle as O
from paper_2111_00153_b200 import binding as R
from paper_2111_00153_b200 import build
from paper_2111_00153_b200 import synth

pytestmark = pytest.mark.gpu

SOURCE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native", "early_trigger.cu")


@pytest.fixture(scope="module")
def early_trigger(tmp_path_factory):
    """call(in_dst, in_src, out_dst, out_src, ns): the kernel in front, on the current stream; tensors of bytes."""
    import torch
    lib = str(tmp_path_factory.mktemp("native") / "early_trigger.so")
    subprocess.check_call([build._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-shared", "-Xcompiler", "-fPIC", SOURCE, "-o", lib])
    launch = ctypes.CDLL(lib).early_trigger_copy_launch
    launch.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong] * 2 + [ctypes.c_longlong, ctypes.c_void_p]

    def call(in_dst, in_src, out_dst, out_src, ns):
        assert in_dst.nbytes == in_src.nbytes and out_dst.nbytes == out_src.nbytes
        assert launch(in_dst.data_ptr(), in_src.data_ptr(), in_dst.nbytes, out_dst.data_ptr(), out_src.data_ptr(), out_dst.nbytes, ns,
                      torch.cuda.current_stream().cuda_stream) == 0
    return call


# name: M, Cin, k, stride, B, H, call.  A linear layer has H = 1 and B tokens.  One of every kernel that a call may go to.
ROUTES = {
    "plain_small": (256, 512, 1, 1, 64, 1, "gemm"),                     # the reduction shared by a cluster, codes expanded by its warps
    "plain_resident": (128, 512, 1, 1, 40000, 1, "gemm"),               # weights expanded once and resident
    "plain_ring": (256, 1024, 1, 1, 20000, 1, "gemm"),                  # weights expanded for every tile
    "plain_gathered": (64, 20, 3, 1, 4, 28, "conv"),                    # activations gathered by threads
    "workspace_small": (512, 512, 3, 1, 1, 7, "workspace"),             # the reduction shared by a cluster
    "workspace_half_grid": (64, 64, 3, 1, 4, 56, "workspace"),          # the grid leaves half of the SMs free
    "workspace_resident": (192, 32, 1, 1, 16, 56, "workspace"),
    "workspace_column_shift": (64, 64, 3, 1, 64, 56, "workspace"),
    "workspace_wide_shift": (128, 128, 3, 1, 128, 28, "workspace"),
    "workspace_ring": (384, 512, 1, 1, 20000, 1, "workspace"),
    "workspace_sums": (512, 2048, 1, 1, 20000, 1, "workspace_acc"),     # two row blocks a tile
    "workspace_pair": (256, 2048, 1, 1, 20000, 1, "workspace"),
    "workspace_pair_shift": (256, 256, 3, 1, 64, 14, "workspace"),
    "requant_small": (512, 512, 3, 1, 1, 7, "requant"),
    "requant_resident": (192, 32, 1, 1, 64, 56, "requant"),
    "requant_ring": (256, 768, 1, 1, 20000, 1, "requant"),
    "depthwise": (96, 1, 3, 1, 4, 28, "depthwise"),
}


class Layer:
    """A layer's buffers in one block of bytes: packed weights, expanded weights, activation codes."""

    def __init__(self, name, seed):
        import torch
        self.M, self.Cin, self.k, self.stride, self.B, self.H, self.call = ROUTES[name]
        g = synth.rng(150, seed)
        depthwise = self.call == "depthwise"
        W = synth.weights_kaiming(g, self.M, self.Cin, self.k, self.k)
        scheme, bits = O.assign_rows(synth.weights_kaiming(synth.rng(150, 99), self.M, self.Cin, self.k, self.k), (50, 30, 20))
        if seed % 2:
            scheme, bits = scheme[::-1].copy(), bits[::-1].copy()       # other rows of the same kinds
        self.layer = R.rmsmp_layer_init(self.M, self.Cin, self.k, self.k, scheme, bits)
        up = lambda n: (n + 255) // 256 * 256
        n_packed, n_ws = up(self.layer.packed_bytes), up(R.rmsmp_workspace_bytes(self.layer))
        channels = self.M if depthwise else self.Cin
        codes = g.integers(0, 16, size=(self.B, self.H, self.H, channels)).astype(np.int8)
        self.at = (0, n_packed, n_packed + n_ws)
        self.code_bytes = codes.size
        self.block = torch.zeros(n_packed + n_ws + up(codes.size), dtype=torch.uint8, device="cuda")
        packed, ws, c = self.parts(self.block)
        R.rmsmp_quantize_pack(torch.from_numpy(W).cuda(), R.W_CONV_OIHW, self.layer, scheme, bits, synth.alpha_rows(W), R.POT_NEAREST, packed)
        if not depthwise:
            R.rmsmp_expand_weights(self.layer, packed, ws)
        c.copy_(torch.from_numpy(codes.reshape(-1)).cuda())
        self.N = self.B * ((self.H + 2 * (self.k // 2) - self.k) // self.stride + 1) ** 2
        self.out_type = torch.int8 if self.call == "requant" else torch.float32
        torch.cuda.synchronize()

    def parts(self, block):
        import torch
        a, b, c = self.at
        return block[a:a + self.layer.packed_bytes], block[b:c].view(torch.int8), block[c:c + self.code_bytes].view(torch.int8)

    def out(self):
        import torch
        return torch.full((self.N, self.M), 99, dtype=self.out_type, device="cuda")

    def run(self, block, y, acc=None):
        packed, ws, codes = self.parts(block)
        L, B, H, s, pad = self.layer, self.B, self.H, self.stride, self.k // 2
        if self.call == "gemm":
            R.rmsmp_gemm(L, packed, codes, self.N, self.Cin, 0.25, y, self.M, R.OUT_NM)
        elif self.call == "conv":
            R.rmsmp_conv_implicit(L, packed, codes, B, H, H, s, pad, 0.25, y)
        elif self.call == "workspace_acc":
            R.rmsmp_gemm_workspace(L, packed, ws, codes, self.N, self.Cin, 0.25, y, self.M, R.OUT_NM, acc)
        elif self.call == "workspace":
            R.rmsmp_conv_implicit_workspace(L, packed, ws, codes, B, H, H, s, pad, 0.25, y)
        elif self.call == "requant":
            R.rmsmp_conv_implicit_workspace_requant(L, packed, ws, codes, B, H, H, s, pad, 0.25, 3.0, R.ACT_U4, y)
        else:
            R.rmsmp_conv_depthwise(L, packed, codes, B, H, H, s, pad, 0.25, y)


def _behind_a_late_kernel(early_trigger, name, ns, part):
    """Runs a route's call behind a kernel that, ns nanoseconds after its dependents may start, copies another layer's bytes (`part` of
    the block on) to where the call reads, and takes a copy of the call's output buffer as it was."""
    import torch
    old, new = Layer(name, 1), Layer(name, 2 if part == 0 else 3)      # (an odd seed: rows of the same kinds)
    acc = torch.zeros((old.N, old.M), dtype=torch.int32, device="cuda") if old.call == "workspace_acc" else None
    at = old.at[part]
    block = old.block.clone()
    y0 = old.out()
    old.run(block, y0, acc)                                            # (also loads the kernels)
    expect_block = old.block.clone()
    expect_block[at:] = new.block[at:]
    expect = old.out()
    old.run(expect_block, expect, acc)
    torch.cuda.synchronize()
    assert not torch.equal(expect, y0)
    y = old.out()
    before, was = torch.zeros_like(y), y.clone()
    torch.cuda.synchronize()
    early_trigger(block[at:], new.block[at:], before, y, ns)
    old.run(block, y, acc)
    torch.cuda.synchronize()
    assert R.rmsmp_last_device_status(old.parts(block)[0]) == R.OK
    assert torch.equal(y, expect)
    assert torch.equal(before, was)


@pytest.mark.parametrize("name", ROUTES)
def test_a_call_waits_for_a_long_kernel_in_front(early_trigger, name):
    """Longer than the kernels' bounded waits, which begin when the kernel in front is over."""
    _behind_a_late_kernel(early_trigger, name, 1_500_000_000, part=2)


@pytest.mark.parametrize("name", ROUTES)
def test_a_call_reads_weights_that_the_kernel_in_front_writes_late(early_trigger, name):
    """Packed codes with their metadata and the expanded copy are as the kernel in front leaves them, not as it finds them."""
    _behind_a_late_kernel(early_trigger, name, 20_000_000, part=0)


def test_weights_packed_and_expanded_again_between_calls():
    """Two layers in turn, packed into the same buffer, expanded into the same workspace and into the library's scratch, with nothing
    between the calls: each uses its own weights."""
    import torch
    M, K, N = 512, 1024, 200
    g = synth.rng(151)
    scheme, bits = O.assign_rows(synth.weights_normal(g, (M, K)), (50, 30, 20))
    layer = R.rmsmp_layer_init(M, K, 1, 1, scheme, bits)
    packed = torch.zeros(layer.packed_bytes, dtype=torch.uint8, device="cuda")
    ws = torch.zeros(R.rmsmp_workspace_bytes(layer), dtype=torch.int8, device="cuda")
    codes = torch.from_numpy(synth.act_codes_uniform(g, (N, K))).cuda()
    Ws = [synth.weights_normal(g, (M, K)) for _ in range(2)]
    alphas = [synth.alpha_rows(W) for W in Ws]
    refs = [O.layer_linear(W, scheme, bits, a, codes.cpu().numpy(), np.float32(0.25))[-1].reshape(N, M) for W, a in zip(Ws, alphas)]
    dW = [torch.from_numpy(W).cuda() for W in Ws]
    outs = torch.full((24, 4, N, M), float("nan"), dtype=torch.float32, device="cuda")
    n16 = torch.full((24, 16, M), float("nan"), dtype=torch.float32, device="cuda")
    arrs = [R.make_gemm_items([(layer, packed, codes, 16, K, 0.25, n16[i], M, None, 1)]) for i in range(24)]
    tables = [torch.empty(R.rmsmp_grouped_plan_bytes(arrs[0]), dtype=torch.uint8, device="cuda") for _ in range(24)]
    plans = [R.rmsmp_gemm_grouped_prepare(a, R.OUT_NM, t) for a, t in zip(arrs, tables)]
    torch.cuda.synchronize()
    for i in range(24):
        R.rmsmp_quantize_pack(dW[i % 2], R.W_LINEAR, layer, scheme, bits, alphas[i % 2], R.POT_NEAREST, packed)
        if i % 4 < 2:
            R.rmsmp_gemm_grouped_launch(plans[i])                       # directly behind the packing
            R.rmsmp_gemm(layer, packed, codes, N, K, 0.25, outs[i, 0], M, R.OUT_NM)
        else:
            R.rmsmp_gemm(layer, packed, codes, N, K, 0.25, outs[i, 0], M, R.OUT_NM)
            R.rmsmp_gemm_grouped_launch(plans[i])
        R.rmsmp_expand_weights(layer, packed, ws)
        R.rmsmp_gemm_workspace(layer, packed, ws, codes, N, K, 0.25, outs[i, 1], M)
        R.rmsmp_gemm_builtin_scratch(layer, packed, codes, N, K, 0.25, outs[i, 2], M)
        R.rmsmp_gemm_builtin_scratch(layer, packed, codes, N, K, 0.25, outs[i, 3], M)
    torch.cuda.synchronize()
    assert R.rmsmp_last_device_status(packed) == R.OK
    got, got16 = outs.cpu().numpy(), n16.cpu().numpy()
    for i in range(24):
        for k in range(4):
            assert np.array_equal(got[i, k].view(np.uint32), refs[i % 2].view(np.uint32)), (i, k)
        assert np.array_equal(got16[i].view(np.uint32), refs[i % 2][:16].view(np.uint32)), i
