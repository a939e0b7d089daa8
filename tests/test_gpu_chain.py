"""Runs of identity blocks as one launch per pass, at sizes where their tiles, images per CTA and pieces have edges: every layer
of the forward and of the backward pass against the oracle's layer functions on the library's own inputs to it (bars: one
bfloat16 ulp of the largest element is 4e-3), and an inference pass against float64."""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

import fdg_synth as S
from oracle import layers as L
from tests.layerwise import check_backward_layerwise, take, units_of

pytestmark = pytest.mark.gpu
EPS = 1e-5

# (batch, image side, blocks per stage, K, splits): single images and groups; partly filled tiles (28 = 7 groups, 28 of 32 rows);
# several column blocks (40) and tiles per image; more images than CTAs (149, 161) and the most that a CTA holds; one-pixel maps;
# runs of one block, of several pieces in the backward pass
CASES = [(1, 12, 2, 1, ()), (5, 28, 3, 1, ()), (3, 40, 2, 2, (3,)), (149, 16, 2, 1, ()), (161, 32, 2, 4, (1, 2, 4)), (7, 4, 3, 1, ()),
         (9, 20, 5, 1, ()), (2, 8, 13, 1, ()),
         # two modules whose runs do not fit the device together (76 + 76 CTAs of one image): one of them goes layer by layer
         (76, 40, 2, 2, (1,))]


def _context(case, lr=0.0, **kw):
    from paper_1906_09108_b200 import binding as B
    batch, hw, n, K, splits = case
    arch = dict(family="resnet6n2", n_per_stage=n, widths=(16, 32, 64), stem_width=16, in_h=hw, in_w=hw, in_c=3, num_classes=10, batch=batch)
    g = B.FDG(B.make_arch(**arch), K=K, split_after_block=splits, beta=0.5, precision=B.FDG_BF16_TC, lr=lr, weight_decay=0.0, **kw)
    params = {}
    for k in range(1, K + 1):
        params[k] = S.init_params(0, k, g.param_layout(k), jitter=True)
        g.set_params(k, params[k])
    return g, params, arch


def _runs(g, K):
    """[(blocks of a run, runs)] of every module, and the blocks with a projection: what a context's layouts say."""
    runs, proj = [], 0
    for k in range(1, K + 1):
        last = None
        for name, ent in units_of(g.param_layout(k)):
            if not name.startswith("block"):
                last = None
            elif len(ent) > 6:
                proj, last = proj + 1, None
            elif last is None:
                runs.append(1)
                last = True
            else:
                runs[-1] += 1
    return runs, proj


@pytest.mark.parametrize("case", CASES[:-1])
def test_every_run_is_one_launch_forward_and_one_a_piece_backward(case):
    """Convolution launches of one iteration in flight: stem, three a projection block, one a run; backward one for each
    piece of a run (the last of up to 4 blocks, the others of up to 12)."""
    g, _, arch = _context(case)
    b, hw, K = arch["batch"], arch["in_h"], case[3]
    runs, proj = _runs(g, K)
    for t in range(1, 2 * K + 4):
        if t == 2 * K + 3:
            g.sync()
            g.profile_enable()
        g.step(torch.from_numpy(S.images(0, t, b, hw, hw, 3)).cuda(), torch.from_numpy(S.labels(0, t, b, 10)).cuda())
    g.sync()
    rows = {r["name"]: r["launches"] for r in g.profile_read()}
    assert rows["conv_fprop"] == 1 + 3 * proj + len(runs)
    assert rows["conv_dgrad"] == 3 * proj + sum(1 if n <= 4 else 1 + -(-(n - 4) // 12) for n in runs)
    g.close()


def _relmax(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-30))


@pytest.mark.parametrize("case", CASES)
def test_backward(case):
    g, params, arch = _context(case)
    checked, _ = check_backward_layerwise(g, params, arch, case[3])
    assert checked == 3 * case[2]
    assert g.check_guards() == -1
    g.close()


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("case", CASES)
def test_forward(case, graphs):
    g, params, arch = _context(case, graphs=graphs)
    b, hw, K = arch["batch"], arch["in_h"], case[3]
    for t in range(1, 2 * K + 4):
        g.step(torch.from_numpy(S.images(0, t, b, hw, hw, 3)).cuda(), torch.from_numpy(S.labels(0, t, b, 10)).cuda())
    g.sync()
    checked = 0
    for k in range(1, K + 1):
        units = units_of(g.param_layout(k))
        for u in range(1, len(units)):
            name, ent = units[u]
            if not name.startswith("block") or len(ent) > 6:
                continue
            co = ent[0][1][0]
            w1, w2 = L.round_bf16(take(params[k], ent[0])), L.round_bf16(take(params[k], ent[3]))
            bn1, bn2 = [take(params[k], e) for e in ent[1:3]], [take(params[k], e) for e in ent[4:6]]
            _, x = g.saved_tensor(k, u - 1, 3)
            side = int(round((x.size / (b * co)) ** 0.5))
            got = [x] + [g.saved_tensor(k, u, w)[1] for w in range(4)]
            x, c1, a1, c2, y = (v.reshape(b, side, side, co).astype(np.float64) for v in got)
            assert _relmax(c1, L.round_bf16(L.conv2d_forward(x, w1, 1, 1))) <= 1e-2, (k, name)
            assert _relmax(a1, L.round_bf16(L.relu_forward(L.batchnorm_forward(c1, *bn1, EPS)[0]))) <= 1e-2, (k, name)
            assert _relmax(c2, L.round_bf16(L.conv2d_forward(a1, w2, 1, 1))) <= 1e-2, (k, name)
            assert _relmax(y, L.round_bf16(L.relu_forward(L.batchnorm_forward(c2, *bn2, EPS)[0] + x))) <= 1e-2, (k, name)
            checked += 1
    assert checked > 0 and g.check_guards() == -1
    g.close()


@pytest.mark.parametrize("case", [(5, 28, 3, 1, ()), (149, 16, 2, 1, ()), (161, 32, 2, 4, (1, 2, 4)), (9, 20, 5, 1, ()), (2, 8, 13, 1, ())])
def test_running_statistics_of_every_layer_of_a_run(case):
    """One iteration moves the running mean and (unbiased) variance of each batch norm by a tenth towards those of the
    convolution output that the iteration saved."""
    g, _, arch = _context(case)
    b, hw, K = arch["batch"], arch["in_h"], case[3]
    for t in range(1, 2 * K + 4):
        if t == 2 * K + 3:
            before = [np.asarray(g.get_running(k), dtype=np.float64) for k in range(1, K + 1)]
        g.step(torch.from_numpy(S.images(0, t, b, hw, hw, 3)).cuda(), torch.from_numpy(S.labels(0, t, b, 10)).cuda())
    g.sync()
    checked = 0
    for k in range(1, K + 1):
        after, at = np.asarray(g.get_running(k), dtype=np.float64), 0
        for u, (name, ent) in enumerate(units_of(g.param_layout(k))):
            if name == "head":
                continue
            co = ent[0][1][0]
            for which in ((0,) if name == "stem" else (0, 2)):
                if name != "stem" and len(ent) <= 6:
                    c = g.saved_tensor(k, u, which)[1].reshape(-1, co).astype(np.float64)
                    sq = (c ** 2).mean(0)
                    for stat, got, old in ((c.mean(0), after[at:at + co], before[k - 1][at:at + co]),
                                           (c.var(0) * len(c) / (len(c) - 1), after[at + co:at + 2 * co], before[k - 1][at + co:at + 2 * co])):
                        # fp32 sums of a few hundred values a thread, fp32 results
                        assert (np.abs(got - (0.9 * old + 0.1 * stat)) <= 1e-5 * (np.abs(old) + np.sqrt(sq) + sq)).all(), (k, name, which)
                    checked += 1
                at += 2 * co
            at += 2 * co if len(ent) > 6 else 0
        assert at == after.size
    assert checked == 2 * (3 * case[2] - 2)
    g.close()


def _eval_reference(g, params, K, x):
    """float64 with the tensors rounded to bfloat16 that the inference pass keeps between two layers."""
    def q(v):
        return v.to(torch.bfloat16).double()

    def conv(v, w, stride, pad):
        return q(F.conv2d(v, q(torch.from_numpy(w)).permute(0, 3, 1, 2), stride=stride, padding=pad))

    def bn(v, ga, be, mean, var):
        inv = 1.0 / torch.sqrt(var + EPS)
        return (v - mean.view(1, -1, 1, 1)) * (torch.from_numpy(ga) * inv).view(1, -1, 1, 1) + torch.from_numpy(be).view(1, -1, 1, 1)

    x = q(x.double().cpu()).permute(0, 3, 1, 2)
    for k in range(1, K + 1):
        running, at = torch.from_numpy(np.asarray(g.get_running(k), dtype=np.float64)), 0

        def stats(c):
            nonlocal at
            at += 2 * c
            return running[at - 2 * c:at - c], running[at - c:at]
        for name, ent in units_of(g.param_layout(k)):
            p = [take(params[k], e) for e in ent]
            if name == "stem":
                x = q(F.relu(bn(conv(x, p[0], 1, 1), p[1], p[2], *stats(p[0].shape[0]))))
            elif name == "head":
                return x.mean(dim=(2, 3)) @ torch.from_numpy(p[0].reshape(p[0].shape[0], -1)).T + torch.from_numpy(p[1].reshape(-1))
            else:
                proj, co = len(p) > 6, p[0].shape[0]
                s1, s2 = stats(co), stats(co)
                a = q(F.relu(bn(conv(x, p[0], 2 if proj else 1, 1), p[1], p[2], *s1)))
                sc = bn(conv(x, p[6], 2, 0), p[7], p[8], *stats(co)) if proj else x
                x = q(F.relu(bn(conv(a, p[3], 1, 1), p[4], p[5], *s2) + sc))


@pytest.mark.parametrize("case", CASES)
def test_inference(case):
    g, params, arch = _context(case)
    b, hw, K = arch["batch"], arch["in_h"], case[3]
    for t in range(1, 2 * K + 4):
        g.step(torch.from_numpy(S.images(0, t, b, hw, hw, 3)).cuda(), torch.from_numpy(S.labels(0, t, b, 10)).cuda())
    g.sync()
    x = torch.from_numpy(S.images(0, 99, b, hw, hw, 3)).cuda()
    logits = torch.empty((b, 10), device="cuda")
    g.eval(x, torch.zeros(b, dtype=torch.int32, device="cuda"), logits_dev=logits)
    torch.cuda.synchronize()
    want = _eval_reference(g, params, K, x).numpy()
    got = logits.double().cpu().numpy()
    # half a bfloat16 unit (2^-9) for each tensor rounded differently, 6 n + 2 of them in a row at worst, adding up like noise
    assert np.linalg.norm(got - want) <= 2.0 ** -9 * (6 * case[2] + 2) ** 0.5 * np.linalg.norm(want)
    g.close()


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("case", [(9, 20, 5, 1, ()), (76, 16, 3, 2, (4,)), (8, 12, 2, 3, (1, 3))])
def test_inference_and_a_loaded_state_leave_a_run_s_training_as_it_is(case, graphs):
    """Training keeps its scratch, the words of the exchanges among it, where an inference pass works: with passes in between and
    a saved state loaded, parameters, momentum and running statistics are those of a run without, bit for bit."""
    batch, hw, K = case[0], case[1], case[3]
    feeds = [(torch.from_numpy(S.images(0, t, batch, hw, hw, 3)).cuda(), torch.from_numpy(S.labels(0, t, batch, 10)).cuda()) for t in range(1, 31)]
    res = []
    for between in (False, True):
        g, _, _ = _context(case, lr=0.05, graphs=graphs)
        blob = None
        for t, (x, y) in enumerate(feeds):
            g.step(x, y)
            if between and t in (3, 14, 15, 24):
                g.eval(x, y)
            if between and t == 20:
                blob = g.save_state()
            if between and t == 22:                       # two iterations again, from the state of before
                g.eval(x, y)
                g.load_state(blob)
                for again in feeds[21:23]:
                    g.step(*again)
        g.sync()
        assert g.check_guards() == -1
        res.append([np.asarray(get(k)) for get in (g.get_params, g.get_momentum, g.get_running) for k in range(1, K + 1)])
        g.close()
    for u, v in zip(*res):
        assert np.isfinite(u).all() and np.array_equal(u, v)
