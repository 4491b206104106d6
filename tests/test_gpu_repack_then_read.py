"""A handle packed again in place, with the calls that read it ahead of their wait for earlier kernels right behind it: the
few-outputs kernel (3x3 and 1x1), the stem, a tensor-path layer, to-dense with a ragged tail.  Round after round with other
weights, in a stream and in a graph, through rtoss_pack and through the whole-model pass: every result is the one of a handle
packed freshly, with the device idle in between."""
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2303_02191_b200 import binding as rt
    import gpu_util as gu

# ks, Cin, Cout, H, W, stride, layout: few outputs, stem, tensor path
LAYERS = [(3, 19, 11, 9, 8, 1, 0), (1, 23, 9, 9, 8, 1, 0), (3, 3, 32, 32, 32, 2, 1), (3, 64, 72, 20, 20, 1, 1)]
ROUNDS = 12


def _run(c, L, packed, x, y, dense):
    ks, Cin, Cout, H, W, S, layout = L
    fn = c.rtoss_conv3x3_pattern if ks == 3 else c.rtoss_conv1x1_pattern
    fn(packed, x, y, 1, H, W, S, layout, rt.ACT_NONE, path=rt.PATH_AUTO if layout else rt.PATH_FMA)
    c._check(rt.lib.rtoss_packed_to_dense(c.h, packed.h, dense.data_ptr(), torch.cuda.current_stream().cuda_stream))


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("batch", [False, True])
def test_reads_what_was_just_packed(batch, graph):
    c, masks = gu.ctx(), rt.rtoss_pattern_preset(4, rt.PRESET_CENTRE8)
    g = torch.Generator(device="cuda").manual_seed(4)
    rnd = lambda shape: torch.empty(shape, device="cuda").normal_(generator=g)
    jobs = []
    for L in LAYERS:
        ks, Cin, Cout, H, W, S, layout = L
        ws = [rnd((Cout, Cin, ks, ks)) for _ in range(ROUNDS)]
        x = rnd((1, H, W, Cin) if layout else (1, Cin, H, W)).to(torch.bfloat16)
        Ho, Wo = (H - 1) // S + 1, (W - 1) // S + 1
        n = Cout * Cin if ks == 3 else Cout * Cin // 9
        j = dict(L=L, ws=ws, x=x, w=ws[0].clone(), pid=torch.empty(n, dtype=torch.uint8, device="cuda"), y=[], dense=[], want=[])
        for w in ws:
            y, d = torch.empty((1, Ho, Wo, Cout) if layout else (1, Cout, Ho, Wo), dtype=torch.bfloat16, device="cuda"), torch.empty(w.numel(), dtype=torch.bfloat16, device="cuda")
            p = c.rtoss_pack(w, ks, masks, 4, c.rtoss_select_patterns(w, ks, masks, 4), rt.BF16)
            torch.cuda.synchronize()
            _run(c, L, p, x, y, d)
            torch.cuda.synchronize()
            p.close()
            j["want"].append((y, d))
            j["y"].append(torch.zeros_like(y))
            j["dense"].append(torch.zeros_like(d))
        j["packed"] = c.rtoss_pack(j["w"], ks, masks, 4, c.rtoss_select_patterns(j["w"], ks, masks, 4), rt.BF16)
        jobs.append(j)
    b = c.rtoss_batch_create([dict(w=j["w"], ksize=j["L"][0], masks=masks, k=4, packed=j["packed"]) for j in jobs])

    def rounds():
        for r in range(ROUNDS):
            for j in jobs:
                j["w"].copy_(j["ws"][r])
            if batch:
                b.rtoss_batch_select_pack()
            for j in jobs:
                if not batch:
                    ks = j["L"][0]
                    c.rtoss_select_patterns(j["w"], ks, masks, 4, pid=j["pid"])
                    c.rtoss_pack(j["w"], ks, masks, 4, j["pid"], rt.BF16, into=j["packed"])
                _run(c, j["L"], j["packed"], j["x"], j["y"][r], j["dense"][r])

    rounds()
    if graph:
        torch.cuda.synchronize()
        cg = torch.cuda.CUDAGraph()
        with torch.cuda.graph(cg):
            rounds()
        for j in jobs:
            for t in j["y"] + j["dense"]:
                t.zero_()
        for _ in range(3):
            cg.replay()
    torch.cuda.synchronize()
    assert c.rtoss_device_status() == 0
    for j in jobs:
        for r in range(ROUNDS):
            assert torch.equal(j["y"][r], j["want"][r][0]) and torch.equal(j["dense"][r], j["want"][r][1]), (j["L"], r)
    b.close()
    for j in jobs:
        j["packed"].close()
