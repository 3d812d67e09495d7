"""kkm_distances_noalloc over its tile forms: 64- and 128-row query tiles, rows
read four columns at a time and one at a time, widths on either side of the
16-column step, a last pass of one row, an empty center and more centers than
a block has groups. Against FP64 torch at the FP32 bound; norms that leave the
range of the FP32 pair sums are covered by scaled rows."""
import pytest

from paper_2410_05902_gb300 import kkm as kb

from gpu_helpers import DIST_TOL, torch_cuda

pytestmark = pytest.mark.gpu


def _reference(torch, kind, param, Q, Y, w, off, cn):
    Q, Y, w = Q.double(), Y.double(), w.double()
    out = []
    for j in range(len(off) - 1):
        Yj, wj = Y[off[j]:off[j + 1]], w[off[j]:off[j + 1]]
        if kind == "linear":
            K, self_k = Q @ Yj.T, (Q * Q).sum(1)
        else:
            d2 = torch.cat([(q[:, None, :] - Yj[None, :, :]).square().sum(2) for q in Q.split(64)])
            K = torch.exp(-(d2 if kind == "gaussian" else d2.sqrt()) / param)
            self_k = torch.ones(len(Q), dtype=torch.float64, device=Q.device)
        out.append(self_k - 2.0 * (K @ wj) + cn[j])
    return torch.stack(out, 1)


@pytest.mark.parametrize("kind", ["gaussian", "laplacian", "linear"])
@pytest.mark.parametrize("m,d,k,rows,pad,shift", [
    (1, 1, 1, 1, 0, 0), (64, 64, 50, 200, 0, 0), (65, 16, 60, 130, 4, 0), (65, 17, 40, 130, 3, 0),
    (1025, 64, 40, 70, 0, 0), (1024, 130, 33, 65, 2, 0), (300, 63, 40, 100, 1, 4), (300, 61, 300, 3, 3, 0),
    (200, 33, 40, 100, 3, 2)])
def test_noalloc_tile_forms(kind, m, d, k, rows, pad, shift):
    torch = torch_cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(m + d)

    def held(n):
        big = torch.zeros((n, d + pad + shift), device="cuda")
        view = big[:, shift:shift + d]
        view.copy_(torch.randn((n, d), generator=g, device="cuda"))
        return view
    sizes = [0 if j == 1 else rows + j % 3 for j in range(k)]
    off = [0]
    for s in sizes:
        off.append(off[-1] + s)
    Q, Y = held(m), held(off[-1])
    w = torch.rand(off[-1], generator=g, device="cuda") / rows
    cn = torch.rand(k, generator=g, device="cuda").double()
    param = {"gaussian": 4.0 * d, "laplacian": 2.0 * d ** 0.5, "linear": 1.0}[kind]
    dist = torch.empty((m, k), device="cuda")
    assign = torch.empty(m, dtype=torch.int32, device="cuda")
    kern = kb.kkm_kernel(kb.KERNELS[kind], param, 0.0, 2)
    kb.kkm_distances_noalloc(Q.data_ptr(), m, Q.stride(0), d, Y.data_ptr(), off[-1], Y.stride(0), w.data_ptr(),
                             torch.tensor(off, dtype=torch.int32, device="cuda").data_ptr(), cn.data_ptr(), k, kern,
                             dist.data_ptr(), assign.data_ptr(), torch.cuda.current_stream().cuda_stream)
    ref = _reference(torch, kind, param, Q, Y, w, off, cn)
    scale = float(ref.abs().max())
    assert float((dist.double() - ref).abs().max()) <= DIST_TOL["fp32"] * scale
    picked = ref.gather(1, assign.long()[:, None])[:, 0]
    assert float((picked - ref.min(1).values).max()) <= 2 * DIST_TOL["fp32"] * scale


@pytest.mark.parametrize("scale", [0.0, 1e-18, 1e-14, 1.0, 1e17, 1e18])
def test_noalloc_norms_over_the_range(scale):
    """(x, x) through the linear kernel's K(q, q): an empty center's distance is the row's norm."""
    torch = torch_cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    m, d = 70, 37
    Q = scale * torch.randn((m, d), generator=g, device="cuda")
    off = torch.zeros(2, dtype=torch.int32, device="cuda")
    cn = torch.zeros(1, dtype=torch.float64, device="cuda")
    dist = torch.empty((m, 1), device="cuda")
    kb.kkm_distances_noalloc(Q.data_ptr(), m, d, d, 0, 0, 0, 0, off.data_ptr(), cn.data_ptr(), 1,
                             kb.kkm_kernel(kb.KERNELS["linear"], 1.0, 0.0, 2), dist.data_ptr(), None,
                             torch.cuda.current_stream().cuda_stream)
    ref = (Q.double() ** 2).sum(1)
    # one FP32 rounding of the norm, of the result, and half the smallest subnormal
    tol = 2.0 ** -23 * ref + 2.0 ** -149
    assert bool(((dist[:, 0].double() - ref).abs() <= tol).all())
