"""Kernel branches at the sizes where they can go wrong (tile edges, ragged
columns, smallest and largest of a branch's range), against the CPU oracle."""
import pytest

from paper_2401_16757_gb300 import capi
import synth
from helpers import Runner, check_close, oracle_outputs
from oracle import plan as OP

pytestmark = pytest.mark.gpu


def _linear(src, k, n, act="none", res=None, res_post=False, bias=True):
    return dict(op="linear", src=[src], k=k, n=n, act=act, res=res, res_post=res_post, bias=bias)


def _check(layers, inp, dtype, budget=None):
    """The resident engine against the oracle, and a swapped one (where the
    model has layers enough to swap) bit-equal to it."""
    m = dict(name="yolov3", model_id=43, dtype=dtype, input=inp, layers=layers, outputs=[len(layers) - 1])
    w, x, d = synth.gen.model_weights(m), synth.gen.model_input(m), capi.Desc(m)
    host = capi.HostWeights(w)
    rs = Runner(m, w, capi.Plan.resident(d), host)
    got = rs.run(x)
    check_close(m, rs.decode(got), oracle_outputs(m, w, x))
    biggest = max(sum(OP.align(b) for b in OP.layer_tensor_bytes(m, i)) for i in range(len(layers)))
    sw = Runner(m, w, capi.Plan.partition(d, 2 * biggest + 512, capi.options(swap_variant=capi.SWAP_ZEROCOPY)), host)
    assert all(a.tobytes() == b.tobytes() for a, b in zip(sw.run(x), got)), "swapped and resident differ"
    return rs


def _routes(rs):
    """Per unit on the tensor cores: which kernel, its N tile, the splits of K and, persistent, the 128-row parts of a
    tile.  A test of a kernel's edges asserts them, so that a change of the choice does not empty it."""
    return [("pair" if t["pair"] else "persist" if t["persistent"] else "tile", t["n_tile"], t["splits"], t["sub_tiles"])
            for t in rs.engine.unit_tiling()]


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("act,res_post", [("relu", False), ("leaky", True), ("swiglu", False)])
@pytest.mark.parametrize("rows,k,n,route", [
    (200, 256, 40, ("tile", 64, 1, 1)),       # one 32-column piece and a quarter
    (200, 256, 255, ("tile", 64, 1, 1)),      # odd width: 2-byte moves
    (1000, 200, 1000, ("tile", 64, 1, 1)),    # ragged k-block, ragged last columns
    (897, 64, 1501, ("tile", 128, 1, 1)),     # one k-block
    (40, 2048, 130, ("tile", 64, 7, 1)),      # K split over a cluster, rows shared out, odd multiple of 2
    (129, 4096, 264, ("tile", 64, 8, 1)),     # the same, second M tile of one row
    (12, 2048, 520, ("tile", 64, 8, 1)),      # few rows: columns shared out
    (16, 2048, 333, ("tile", 64, 8, 1)),
    (1101, 264, 1975, ("persist", 128, 1, 1)),
    (2377, 2552, 1935, ("persist", 256, 1, 1)),
    (20001, 72, 33, ("persist", 64, 1, 1)),
    (97700, 456, 47, ("persist", 64, 1, 2)),
])
def test_tile_epilogue(dtype, act, res_post, rows, k, n, route):
    rs = _check([_linear(-1, k, n), _linear(-1, k, n, act, res=0, res_post=res_post)], (rows, 1, 1, k), dtype)
    assert _routes(rs) == [route] * 2


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("rows,k,n,n_tile,splits", [
    (5, 8, 8, 64, 1),          # one ragged k-block, one piece of 8 columns
    (16, 72, 1001, 64, 1),     # odd width
    (15, 1336, 77, 64, 7),     # column shares of 16: the last splits own none
    (9, 1992, 130, 64, 8),
    (8, 3264, 3778, 128, 4),
    (13, 64, 9793, 128, 1),    # one k-block
    (7, 1032, 19551, 256, 1),
    (16, 4872, 10561, 256, 3),  # shares of 88 columns, the last of 80
])
def test_few_row_gemm(dtype, rows, k, n, n_tile, splits):
    rs = _check([_linear(-1, k, n, "relu")], (rows, 1, 1, k), dtype)
    t = rs.engine.unit_tiling()[0]
    assert (t["n_tile"], t["splits"], t["persistent"]) == (n_tile, splits, 0)


@pytest.mark.parametrize("layer,route", [
    ((20000, 256, 256), ("persist", 128, 1, 1)),        # wide and short: 7.8 us, 11.4 on pairs with N tiles of 64
    ((628, 144, 6272), ("persist", 256, 1, 1)),         # 6.0, 11.0
    ((200, 4096, 4096), ("tile", 64, 1, 1)),            # 9.8, 12.0
    ((100, 1016, 64), ("tile", 64, 8, 1)),              # ragged rows: 4.0 split, 5.3 not
    ((100, 1024, 64), ("tile", 64, 1, 1)),              # 3.8, 3.9 split
    ((3, 96, 96, 9), ("tile", 64, 7, 1)),               # gathered: 4.9 split, 9.4 not
    ((3, 256, 12, 182), ("pair", 64, 1, 2)),            # few features: 16.7, 32.8 on single SMs
    ((3, 256, 512, 26, 4), ("tile", 128, 1, 1)),        # one wave of taps: 9.4, 10.2 persistent
    ((3, 64, 71, 217, 16), ("pair", 96, 1, 2)),         # many waves of them: 160, 210 on single SMs
])
def test_choice_of_kernel(layer, route):
    """Layers whose second-best choice costs much more (us measured on the GB300)."""
    if len(layer) == 3:
        rows, k, n = layer
        lay, inp = _linear(-1, k, n), (rows, 1, 1, k)
    else:
        k, cin, cout, hw, batch = layer + (1,) * (5 - len(layer))
        lay = dict(op="conv", src=[-1], cin=cin, cout=cout, kh=k, kw=k, stride=1, pad=k // 2, act="none", res=None, res_post=False)
        inp = (batch, hw, hw, cin)
    m = dict(name="yolov3", model_id=53, dtype="f16", input=inp, layers=[lay], outputs=[0])
    rs = Runner(m, synth.gen.model_weights(m), capi.Plan.resident(capi.Desc(m)))
    assert _routes(rs) == [route]


@pytest.mark.parametrize("k,cin,cout,hw,batch,route", [
    (1, 456, 40, 222, 2, ("persist", 64, 1, 2)),  # A by 2-D TMA
    (3, 64, 48, 161, 6, ("persist", 64, 1, 2)),   # by 4-D TMA
    (3, 64, 40, 91, 3, ("persist", 64, 1, 1)),
    (1, 64, 48, 160, 2, ("persist", 64, 1, 1)),
    (5, 128, 17, 93, 4, ("pair", 64, 1, 2)),      # few features
])
def test_sub_tiles_with_a_residual(k, cin, cout, hw, batch, route):
    """Two 128-row sub-tiles per tile, the residual of the next sub-tile
    requested during the one before; one, and a pair of SMs, beside it."""
    conv = dict(op="conv", src=[-1], cin=cin, cout=cout, kh=k, kw=k, stride=1, pad=k // 2, act="none", res=None,
                res_post=False)
    rs = _check([conv, dict(conv, act="leaky", res=0, res_post=True)], (batch, hw, hw, cin), "f16")
    assert _routes(rs) == [route] * 2


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("act,res_post", [("none", False), ("swiglu", False)])
@pytest.mark.parametrize("rows,k,n,n_tile", [
    (1000, 520, 4000, 224),   # ragged last rows, k-block and columns
    (1793, 520, 1501, 192),   # odd width; an odd number of 128-row blocks, one row in the last, the other CTA's empty
    (5001, 1032, 1001, 160),
    (4097, 1032, 500, 128),
    (2049, 1032, 3104, 224),  # two rounds of tiles
    (897, 1032, 9001, 256),
])
def test_paired_gemm(dtype, act, res_post, rows, k, n, n_tile):
    rs = _check([_linear(-1, k, n), _linear(-1, k, n, act, res=0, res_post=res_post)], (rows, 1, 1, k), dtype)
    assert _routes(rs) == [("pair", n_tile, 1, 2)] * 2


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("k,stride,cout,hw,batch,sub_tiles", [
    (3, 1, 64, 161, 2, 2),   # an odd number of taps, ragged patches
    (3, 2, 40, 301, 2, 1),
    (4, 2, 128, 320, 3, 1),  # an even number, N tiles of 128
    (5, 1, 64, 104, 32, 2),
])
def test_two_taps_per_k_block(dtype, k, stride, cout, hw, batch, sub_tiles):
    """Convolutions of 32 channels on the persistent kernel, A by 4-D TMA."""
    conv = dict(op="conv", src=[-1], cin=32, cout=cout, kh=k, kw=k, stride=stride, pad=k // 2, act="leaky", res=None,
                res_post=False)
    rs = _check([conv, dict(conv, res=0, res_post=True)], (batch, hw, hw, 32), dtype)
    assert _routes(rs) == [("persist", 128 if cout > 64 else 64, 1, sub_tiles)] * 2
    assert all(t["tap_tma"] for t in rs.engine.unit_tiling())


@pytest.mark.parametrize("stride,cin,cout,hw,batch,route", [
    (1, 64, 256, 52, 3, ("persist", 256, 1, 1)),  # 4-D TMA on single SMs
    (2, 128, 160, 101, 8, ("pair", 160, 1, 2)),
    (1, 128, 416, 57, 4, ("pair", 224, 1, 2)),
    (2, 256, 320, 75, 5, ("pair", 160, 1, 2)),   # an odd number of patches
    (2, 128, 160, 75, 5, ("tile", 128, 1, 1)),   # 4-D TMA per tile
    (1, 64, 96, 57, 4, ("tile", 128, 1, 1)),
])
def test_paired_conv(stride, cin, cout, hw, batch, route):
    """Convolutions by 4-D TMA on pairs of SMs: patches past the last one, strides, ragged patch edges."""
    conv = dict(op="conv", src=[-1], cin=cin, cout=cout, kh=3, kw=3, stride=stride, pad=1, act="leaky", res=None,
                res_post=False)
    rs = _check([conv, dict(conv, res=0, res_post=True)], (batch, hw, hw, cin), "f16")
    assert _routes(rs) == [route] * 2 and all(t["tap_tma"] for t in rs.engine.unit_tiling())


@pytest.mark.parametrize("dtype,rows,k,n", [
    ("f32", 17, 64, 33),        # one chunk, 16-byte copies
    ("f32", 33, 1001, 129),     # rows of odd length: 4-byte copies, ragged last chunk
    ("f32", 100, 1000, 1000),
    ("f32", 65, 7, 31),         # K below one 4-wide step of every k group
    ("f32", 512, 260, 1029),    # 64 x 64 tiles, all edges ragged
    ("f32", 700, 1023, 768),
    ("f16", 20, 1001, 70),      # 16-bit rows that neither TMA nor 16-byte loads take
    ("bf16", 600, 333, 1100),
])
def test_tiled_linear(dtype, rows, k, n):
    rs = _check([_linear(-1, k, n, "relu"), _linear(-1, k, n, "leaky", res=0, res_post=True)], (rows, 1, 1, k), dtype)
    assert set(rs.engine.unit_kernels()) == {"tiled_linear"}


def test_tiled_linear_pieces_sum_as_the_whole_layer():
    """A fp32 layer split into column pieces by a small budget: same bits as the whole layer."""
    m = dict(name="yolov3", model_id=44, dtype="f32", input=(130, 1, 1, 900), outputs=[1],
             layers=[_linear(-1, 900, 3000, "relu"), _linear(0, 3000, 40)])
    w, x, d = synth.gen.model_weights(m), synth.gen.model_input(m), capi.Desc(m)
    host = capi.HostWeights(w)
    sw = Runner(m, w, capi.Plan.partition(d, 4_000_000, capi.options(swap_variant=capi.SWAP_ZEROCOPY)), host)
    rs = Runner(m, w, capi.Plan.resident(d), host)
    assert len(sw.plan.units()) > 2
    got = rs.run(x)
    assert all(a.tobytes() == b.tobytes() for a, b in zip(sw.run(x), got))
    check_close(m, rs.decode(got), oracle_outputs(m, w, x))


@pytest.mark.parametrize("rows", [70, 16])
def test_swiglu_extreme_gates(rows):
    """Gates far out on both sides (e^-gate overflows to infinity, vanishes, stays normal) and zeros, through the
    tensor-core epilogues: the float64 definition, to the rounding of the stored type."""
    import numpy as np
    import torch
    k = 1024
    m = dict(name="yolov3", model_id=45, dtype="bf16", input=(rows, 1, 1, k), outputs=[0, 1],
             layers=[_linear(-1, k, k, bias=False), _linear(-1, k, k, "swiglu", res=0, bias=False)])
    eye = torch.eye(k, dtype=torch.bfloat16).view(torch.uint16).numpy()
    gates = torch.tensor([0.0, -0.0, 1e-30, -1e-30, 1.0, -1.0, 20.0, -20.0, 80.0, -80.0, -87.0, -88.5, -89.0, -100.0, 100.0,
                          -300.0, 3e4, -3e4], dtype=torch.bfloat16)
    x = gates.repeat(rows * k // gates.numel() + 1)[:rows * k].view(rows, k)
    r = Runner(m, [[eye], [eye]], capi.Plan.resident(capi.Desc(m)))
    gate, out = (torch.from_numpy(t.copy()).view(torch.bfloat16).double().reshape(rows, k) for t in r.run(x.view(torch.uint16).numpy()))
    g = x.double()
    assert torch.equal(gate, g)
    ref = g * torch.sigmoid(g) * g
    # one rounding to bf16 and two fp32 roundings (2^-8 + 2^-22); below 1e-33 fp32's own range ends
    assert torch.all((out - ref).abs() <= ref.abs() * 2.0 ** -8 * 1.01 + 1e-33)


_QUOTIENT_SWEEP = r"""
#include <cstdio>
#include "tc_epi.cuh"
using namespace swapnet;
template <typename T> __device__ float value(unsigned i) {
  const unsigned short b = (unsigned short)i;
  return to_f<T>(*reinterpret_cast<const T*>(&b));
}
template <> __device__ float value<float>(unsigned i) { return ((int)i - (1 << 25)) * (110.0f / (1 << 25)); }
template <typename T> __global__ void sweep(unsigned* differ) {
  const float r = value<T>(blockIdx.x * 256u + threadIdx.x), d = 1.0f + expf(-r);
  const float a = r / d, b = gate_quotient(r, d);
  if (__float_as_uint(a) != __float_as_uint(b) && !(isnan(a) && isnan(b))) atomicAdd(differ, 1u);
}
int main() {
  unsigned *n, h;
  if (cudaMalloc(&n, 4) != cudaSuccess || cudaMemset(n, 0, 4) != cudaSuccess) return 2;
  sweep<__half><<<256, 256>>>(n);
  sweep<__nv_bfloat16><<<256, 256>>>(n);
  sweep<float><<<1 << 18, 256>>>(n);
  if (cudaMemcpy(&h, n, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  std::printf("%u\n", h);
  return 0;
}
"""


def test_gate_quotient_is_the_division(tmp_path):
    """The SwiGLU epilogue's quotient, bit for bit against the division: every fp16 and bf16 gate, and 2^26 fp32 gates
    over the range of expf."""
    import subprocess
    from paper_2401_16757_gb300 import build
    src, exe = tmp_path / "sweep.cu", tmp_path / "sweep"
    src.write_text(_QUOTIENT_SWEEP)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["0"]


def _attention(dtype, tokens, heads, pos, max_seq):
    """One attention layer behind its projections on a random cache: the engine's stored query, key and value rows
    and outputs, the cache before and after, and the float64 result on the stored (rotated) queries and cache."""
    import numpy as np
    import torch
    td, d = (torch.float16 if dtype == "f16" else torch.bfloat16), heads * 128
    m = dict(name="llm", model_id=46, dtype=dtype, input=(tokens, 1, 1, d), outputs=[0, 1, 2, 3],
             layers=[_linear(-1, d, d, bias=False), _linear(-1, d, d, bias=False), _linear(-1, d, d, bias=False),
                     dict(op="attention", src=[0, 1, 2], heads=heads, max_seq=max_seq, theta=10000.0)])
    g = torch.Generator().manual_seed(7)
    host = lambda t: t.view(torch.uint16).numpy() if dtype == "bf16" else t.numpy()
    w = [[host((torch.randn((d, d), generator=g) * d ** -0.5 * s).to(td))] for s in (2.0, 2.0, 1.0)]
    cache = torch.randn((2, max_seq, d), generator=g).to(td)
    r = Runner(m, w, capi.Plan.resident(capi.Desc(m)))
    state = torch.zeros(r.info["state_bytes"], dtype=torch.uint8, device="cuda")
    state[:4].view(torch.int32).fill_(pos)
    state[256:].view(td).view(2, max_seq, d).copy_(cache)
    r.engine.bind_state(state.data_ptr(), r.info["state_bytes"])
    x = torch.randn((tokens, d), generator=g).to(td)
    q, k, v, out = (torch.from_numpy(t.copy().view(np.int16)).view(td).double().reshape(tokens, d) for t in r.run(host(x)))
    after = state[256:].view(td).view(2, max_seq, d).cpu()
    n = pos + tokens
    kk, vv = (after[j, :n].double().view(n, heads, 128).permute(1, 0, 2) for j in (0, 1))
    s = q.view(tokens, heads, 128).permute(1, 0, 2) @ kk.transpose(1, 2) / 128 ** 0.5
    s = s.masked_fill(torch.arange(n)[None, :] > torch.arange(pos, n)[:, None], -torch.inf)
    ref = (torch.softmax(s, -1) @ vv).permute(1, 0, 2).reshape(tokens, d)
    return k, v, out, cache, after, ref


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("tokens,heads,pos,max_seq", [
    (1, 8, 0, 40), (1, 8, 299, 300),                    # one query: the split-key kernel, first and last position
    (3, 4, 62, 200), (5, 2, 510, 4096), (127, 1, 130, 1030),  # the run's own keys across chunks and load passes
    (15, 8, 200, 400), (16, 8, 200, 400),               # either side of 128 (query, head) pairs
    (63, 8, 20, 128), (64, 8, 64, 128),                 # a cache of one key tile
    (47, 8, 81, 128), (48, 8, 20, 128),                 # the same, either side of 384 pairs
    (128, 2, 200, 400), (40, 4, 1000, 1100), (300, 3, 250, 2000),  # key tiles shared by a cluster: rows that see
    (64, 2, 100, 4000), (513, 8, 300, 900),             # nothing of a CTA's, uneven shares, caches barely filled
    (128, 1, 0, 129), (129, 1, 127, 256), (130, 2, 126, 1000),  # query and key tiles full, one over
])
def test_attention_against_float64(dtype, tokens, heads, pos, max_seq):
    """The attention kernels on the engine's own stored (rotated) queries and cache, against float64; and the
    appended cache rows, the positions around them untouched."""
    import torch
    k, v, out, cache, after, ref = _attention(dtype, tokens, heads, pos, max_seq)
    d = heads * 128
    n = pos + tokens
    assert torch.equal(after[:, :pos], cache[:, :pos]) and torch.equal(after[:, n:], cache[:, n:])
    assert torch.equal(after[1, pos:n].double(), v)
    i = torch.arange(64, dtype=torch.float64)
    ang = torch.arange(pos, n, dtype=torch.float64)[:, None, None] * 10000.0 ** (-2.0 * i / 128)
    a, b = k.view(tokens, heads, 64, 2).unbind(-1)
    rot = torch.stack((a * ang.cos() - b * ang.sin(), a * ang.sin() + b * ang.cos()), -1).reshape(tokens, d)
    # angles are fp32: their error is up to |angle| 2^-23, a few 1e-5 here, below the rounding of the stored type
    assert torch.linalg.norm(after[0, pos:n].double() - rot) <= 2e-3 * torch.linalg.norm(rot) * (1 if dtype == "f16" else 2)
    # one rounding to the stored type (relative 2^-12 and 2^-9 rms) and fp32 sums
    assert torch.linalg.norm(out - ref) <= (4e-4 if dtype == "f16" else 2.5e-3) * torch.linalg.norm(ref)


@pytest.mark.parametrize("tokens,heads,pos,max_seq", [
    (3, 32, 300, 400),                                      # the split-key kernel
    (63, 8, 900, 1000), (17, 16, 200, 300), (63, 16, 60, 128),  # short runs on the tensor cores; keys shared or not
])
def test_attention_of_short_runs_keeps_fp32_probabilities(tokens, heads, pos, max_seq):
    """Runs of fewer than 64 queries: bf16 outputs other than the rounded float64 result are as rare as fp32 sums make
    them.  A relative error of 2^-20 crosses the middle between two bf16 values (2^-8 to 2^-7 apart) for up to
    2 x 2^-20 / 2^-8 = 2^-11 of the outputs, bounded here at twice that; with 16 bits of the probabilities it is 2e-3."""
    import torch
    out, ref = _attention("bf16", tokens, heads, pos, max_seq)[2::3]
    assert float((out != ref.to(torch.bfloat16).double()).double().mean()) <= 2.0 ** -10


def test_side_branch_whose_input_is_overwritten_before_its_consumer():
    """A long convolution that may run beside three short ones, the last of which is given the space of its input:
    the bits of one stream, many times over."""
    conv = lambda src, k, res=None: dict(op="conv", src=[src], cin=64, cout=64, kh=k, kw=k, stride=1, pad=k // 2, act="relu",
                                         res=res, res_post=False)
    layers = [conv(-1, 1), conv(0, 1), conv(0, 11), conv(1, 1), conv(3, 1), conv(4, 1, res=2)]
    m = dict(name="yolov3", model_id=52, dtype="f16", input=(2, 40, 40, 64), layers=layers, outputs=[5])
    offs = OP.workspace(m)[1]
    assert offs[4] == offs[0]
    w, x, d = synth.gen.model_weights(m), synth.gen.model_input(m), capi.Desc(m)
    host = capi.HostWeights(w)
    one, both = (Runner(m, w, capi.Plan.resident(d, capi.options(branches=b)), host) for b in (0, 1))
    ref = one.run(x)
    check_close(m, one.decode(ref), oracle_outputs(m, w, x))
    for _ in range(20):
        assert both.run(x)[0].tobytes() == ref[0].tobytes()


@pytest.mark.parametrize("tokens,heads", [(1, 8), (3, 2), (64, 8), (130, 32)])
@pytest.mark.parametrize("pos", ["full", -1, -100, 2 ** 31 - 1, -2 ** 31])
def test_positions_outside_the_cache_are_refused(tokens, heads, pos):
    """A cache position that leaves no room for the run, or none at all (negative, or so large that adding the run
    overflows): reported by the next sync, nothing written around the cache, and the engine usable afterwards."""
    import torch
    d, max_seq, guard = heads * 128, 160, 1 << 20
    if pos == "full":
        pos = max_seq - tokens + 1
    m = dict(name="llm", model_id=51, dtype="bf16", input=(tokens, 1, 1, d), outputs=[3],
             layers=[_linear(-1, d, d, bias=False), _linear(-1, d, d, bias=False), _linear(-1, d, d, bias=False),
                     dict(op="attention", src=[0, 1, 2], heads=heads, max_seq=max_seq, theta=10000.0)])
    w, x = synth.gen.model_weights(m), synth.gen.model_input(m)
    r = Runner(m, w, capi.Plan.resident(capi.Desc(m)))
    size = r.info["state_bytes"]
    memory = torch.full((2 * guard + size,), 0x3c, dtype=torch.uint8, device="cuda")
    state = memory[guard:guard + size]
    r.engine.bind_state(state.data_ptr(), size)
    state[:4].view(torch.int32).fill_(0)
    good = r.run(x)
    state.fill_(0x3c)
    state[:4].view(torch.int32).fill_(pos)
    with pytest.raises(capi.SwapnetError) as ei:
        r.run(x)
    assert ei.value.code == capi.ERR_INVALID_ARG
    torch.cuda.synchronize()
    room = max(0, max_seq - pos) if pos > 0 else 0  # rows of the run that still had a place
    rows = memory.clone()
    rows[guard:guard + 4] = 0x3c
    cache = rows[guard + 256:guard + size].view(2, max_seq, d * 2)
    if room:
        cache[:, pos:] = 0x3c
    assert torch.all(rows == 0x3c)
    state.zero_()
    assert all(a.tobytes() == b.tobytes() for a, b in zip(r.run(x), good))


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("rows,k,n,count,route", [
    # at most 16 rows, loaded in 16-row boxes like a layer alone: every N tile, ragged columns
    (16, 72, 1001, 3, ("tile", 64, 1, 1)), (13, 64, 9793, 2, ("tile", 128, 1, 1)), (5, 1992, 11001, 3, ("tile", 256, 1, 1)),
    (40, 200, 130, 2, ("tile", 64, 1, 1)), (200, 256, 255, 3, ("tile", 64, 1, 1)),   # ragged columns
    (600, 320, 1000, 3, ("tile", 128, 1, 1)), (513, 64, 2056, 3, ("tile", 128, 1, 1)),
    # pairs of SMs: ragged last tile of every layer, one row in the last row tile
    (513, 520, 3001, 3, ("pair", 192, 1, 2)), (1025, 264, 1001, 3, ("pair", 224, 1, 2)), (897, 520, 1501, 2, ("pair", 192, 1, 2)),
    (2600, 128, 96, 4, ("tile", 64, 1, 1)),     # more siblings than one launch takes
])
def test_sibling_linears_share_a_launch(dtype, rows, k, n, count, route):
    """Tensor-core linear layers that read the same input in one launch: the bits of one launch each, and the oracle."""
    layers = [_linear(-1, k, k, "relu")] + [_linear(0, k, n, "leaky", bias=i != 1) for i in range(count)]
    m = dict(name="yolov3", model_id=47, dtype=dtype, input=(rows, 1, 1, k), layers=layers,
             outputs=list(range(1, count + 1)))
    w, x, d = synth.gen.model_weights(m), synth.gen.model_input(m), capi.Desc(m)
    host = capi.HostWeights(w)
    runs = [Runner(m, w, capi.Plan.resident(d, capi.options(merge=g)), host) for g in (1, 0)]
    got, sep = (r.run(x) for r in runs)
    launches = [r.engine.stats()["kernel_launches"] for r in runs]
    tiling, alone = (r.engine.unit_tiling()[1:] for r in runs)
    assert _routes(runs[0])[1] == route
    assert all(t == tiling[0] and t["shared"] for t in tiling[:3]) and not any(t["shared"] for t in tiling[3:] + alone)
    assert launches[1] - launches[0] == (count - 1 if count <= 3 else count - 2)
    assert all(a.tobytes() == b.tobytes() for a, b in zip(got, sep))
    check_close(m, runs[0].decode(got), oracle_outputs(m, w, x))


@pytest.mark.parametrize("dtype,rows", [("f16", 2), ("bf16", 200), ("bf16", 1), ("f32", 1)])
@pytest.mark.parametrize("residual", [False, True])
def test_siblings_whose_buffers_overlap_run_one_by_one(dtype, rows, residual):
    """A sibling that would write, in a shared launch, where another one's unread output or its residual lies: the
    workspace gives both layers one buffer, so they run one after the other."""
    if residual:
        layers = [_linear(-1, 256, 256), _linear(0, 256, 256), _linear(-1, 256, 256, "relu", res=1),
                  _linear(-1, 256, 256), _linear(2, 256, 256, res=3)]
        early, late = 1, 3
    else:
        layers = [_linear(-1, 256, 256), _linear(-1, 256, 256), _linear(1, 256, 256)]
        early, late = 0, 1
    m = dict(name="yolov3", model_id=49, dtype=dtype, input=(rows, 1, 1, 256), layers=layers, outputs=[len(layers) - 1])
    offs = OP.workspace(m)[1]
    assert offs[early] == offs[late]
    w, x, d = synth.gen.model_weights(m), synth.gen.model_input(m), capi.Desc(m)
    host = capi.HostWeights(w)
    runs = [Runner(m, w, capi.Plan.resident(d, capi.options(merge=g)), host) for g in (1, 0)]
    got, sep = (r.run(x) for r in runs)
    assert [r.engine.stats()["kernel_launches"] for r in runs] == [len(layers)] * 2
    assert all(a.tobytes() == b.tobytes() for a, b in zip(got, sep))
    check_close(m, runs[0].decode(got), oracle_outputs(m, w, x))


@pytest.mark.parametrize("rows", [2, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("k,n", [(4, 1), (128, 9), (1020, 40), (1024, 64), (1028, 7), (3000, 130),
                                 (100, 5003), (200, 4999), (512, 5001),  # one, two, four warps to a row
                                 (1032, 5001)])                          # two rows: 16 features per CTA
def test_few_row_fp32_linear(rows, k, n):
    """The few-row kernel at the edges of its k chunks (1024), features per CTA and rows; with a residual."""
    rs = _check([_linear(-1, k, n, "leaky"), _linear(-1, k, n, "relu", res=0)], (rows, 1, 1, k), "f32")
    assert set(rs.engine.unit_kernels()) == {"skinny_linear"}


@pytest.mark.parametrize("rows", [2, 3, 5, 8, 16])
@pytest.mark.parametrize("wide", [9, 5003])  # (5003: teams of warps)
def test_few_row_fp32_siblings_share_a_launch(rows, wide):
    """fp32 siblings of ragged widths in one launch, one with a residual, and a gate with its SwiGLU layer in another:
    the bits of one launch each, and the oracle."""
    layers = [_linear(-1, 1300, 260), _linear(0, 260, 13), _linear(0, 260, 260, "relu", res=0), _linear(0, 260, wide, bias=False),
              _linear(2, 260, 4 * wide), _linear(2, 260, 4 * wide, "swiglu", res=4)]
    m = dict(name="yolov3", model_id=50, dtype="f32", input=(rows, 1, 1, 1300), layers=layers, outputs=[1, 2, 3, 5])
    w, x, d = synth.gen.model_weights(m), synth.gen.model_input(m), capi.Desc(m)
    host = capi.HostWeights(w)
    a, b = (Runner(m, w, capi.Plan.resident(d, capi.options(merge=g)), host) for g in (1, 0))
    got = a.run(x)
    assert all(p.tobytes() == q.tobytes() for p, q in zip(got, b.run(x)))
    assert a.engine.stats()["kernel_launches"] == 3 and b.engine.stats()["kernel_launches"] == 6
    check_close(m, a.decode(got), oracle_outputs(m, w, x))


@pytest.mark.parametrize("dtype,rows", [("f16", 1), ("bf16", 1), ("f16", 2), ("bf16", 3), ("f16", 4), ("f32", 1)])
@pytest.mark.parametrize("k,n", [(8, 1), (2048, 9), (2056, 40), (4104, 300), (11008, 21), (1024, 5000),
                                 (96, 1301), (200, 1304), (504, 2501), (1016, 2600)])  # one, two, four warps to a row
def test_gemv(dtype, rows, k, n):
    """The GEMV at the edges of its passes (2048 or 1024 k), weight-row groups (8) and one group per CTA; a residual,
    and a gate with its SwiGLU layer in one launch."""
    rs = _check([_linear(-1, k, n), _linear(-1, k, n, "swiglu", res=0, bias=False), _linear(1, n, 24, "relu")] if n % 8 == 0
                else [_linear(-1, k, n), _linear(-1, k, n, "leaky", res=0, res_post=True)], (rows, 1, 1, k), dtype)
    assert set(rs.engine.unit_kernels()) == {"skinny_linear"}


@pytest.mark.parametrize("k,n", [(520, 700), (520, 1301), (264, 4003)])
def test_gemv_segments_of_ragged_widths(k, n):
    """Three siblings of widths that are no multiple of a group in one launch: the bits of one launch each."""
    layers = [_linear(-1, k, 13), _linear(-1, k, n, "relu"), _linear(-1, k, 8)]
    m = dict(name="yolov3", model_id=48, dtype="bf16", input=(1, 1, 1, k), layers=layers, outputs=[0, 1, 2])
    w, x, d = synth.gen.model_weights(m), synth.gen.model_input(m), capi.Desc(m)
    host = capi.HostWeights(w)
    a, b = (Runner(m, w, capi.Plan.resident(d, capi.options(merge=g)), host) for g in (1, 0))
    got = a.run(x)
    assert all(p.tobytes() == q.tobytes() for p, q in zip(got, b.run(x)))
    assert a.engine.stats()["kernel_launches"] == 1 and b.engine.stats()["kernel_launches"] == 3
    check_close(m, a.decode(got), oracle_outputs(m, w, x))
