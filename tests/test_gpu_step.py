"""GPU parity of the learner step and of whole rounds (Algorithm 1, Sec. 3.1):
the CUDA path, called through the C ABI, against the oracle on the same seeded
inputs.  Errors are normwise per parameter tensor, max|gpu - oracle| / max|oracle|.

Per step (one step from a shared state, and every step of a teacher-forced round):
the parameters after the step within 1e-5 (fp32 path) or 1e-2 (bf16-operand path,
against an oracle that rounds the same operands to bf16), asserted outright.

The update w_new - w_old of a bf16 step is also checked (2e-2, max and Frobenius
norms).  A ReLU decision on a pre-activation within rounding distance of zero can go
either way under two valid fp32 accumulation orders, which swaps one sample's term
in one row of the update; so an update row beyond the bound is accepted only where
such a flip is provable (the oracle's pre-activation in that row is below the
worst-case difference of two fp32 summation orders plus two bf16 rounding decisions
of the inputs), and every accepted row is counted and reported (none at the 16-learner workload, at most one row in a
thousand at the full-size workloads).

Whole rounds end to end (no teacher forcing): such flips compound over the round's
steps, so the bound there is max(tolerance, SPREAD x the error between two valid
oracles: bf16 operands with exact products, and with fp32 accumulation)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1903_05133_gb300 import configs
from paper_1903_05133_gb300.hier_avg import HierAvg
from paper_1903_05133_gb300.inputs import initial_layers, learner_data, perturbed_layers

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "bf16": 1e-2}
UPDATE_TOL = {"fp32": 1e-5, "bf16": 2e-2}
SPREAD = 3.0


@pytest.fixture(scope="module", autouse=True)
def _cuda(lib):
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def rel_err(got: np.ndarray, want: np.ndarray) -> float:
    scale = np.max(np.abs(want))
    return float(np.max(np.abs(got.astype(np.float64) - want.astype(np.float64))) / max(scale, 1e-30))


def frob_err(got: np.ndarray, want: np.ndarray) -> float:
    d = np.linalg.norm((got.astype(np.float64) - want.astype(np.float64)).ravel())
    return float(d / max(np.linalg.norm(want.astype(np.float64).ravel()), 1e-30))


def setup(w: configs.Workload, layers=None, N=None, data_device="cpu", perturb=None):
    X, y = learner_data(w, device=data_device, N=N)
    if layers is None:
        layers = initial_layers(w, device=data_device)
    ha = HierAvg(w.P, w.S, w.K1, w.K2, w.lr, w.B, w.dims, w.precision)
    params = ha.pack(layers)
    if perturb is not None:
        # distinct learner states with nonzero biases, drawn on the GPU
        g = torch.Generator(device="cuda")
        g.manual_seed(1234)
        for Wl, bl in ha.unpack(params):
            Wl.add_(torch.randn(Wl.shape, generator=g, device="cuda"), alpha=perturb[0])
            bl.add_(torch.randn(bl.shape, generator=g, device="cuda"), alpha=perturb[1])
    ha.bind(params, X.cuda(), y.cuda())
    return ha, X, y


def oracle_params(ha: HierAvg, params_gpu: torch.Tensor, learners=None):
    """The per-layer arrays [W_1, b_1, ...] of a GPU parameter matrix (host copy)."""
    learners = list(range(ha.P)) if learners is None else learners
    out = []
    for W, b in ha.unpack(params_gpu):
        out += [W[learners].cpu().numpy(), b[learners].cpu().numpy()]
    return out


def make_oracle(w, ha, X, y, params, learners=None, mode=None):
    learners = list(range(w.P)) if learners is None else learners
    Xn = X[learners].float().cpu().numpy()
    yn = y[learners].cpu().numpy().astype(np.int64)
    if mode is None:
        mode = "fp32" if w.precision == "fp32" else "bf16"
    prob = oracle.MLPProblem(Xn, yn, w.B, len(w.dims) - 1, mode)
    o = oracle.HierAvgOracle(len(learners), w.S if len(learners) % w.S == 0 else 1, w.K1, w.K2,
                             w.lr, prob, params, mode)
    return o


# A ReLU decision on a pre-activation within rounding distance of zero can go either
# way in two correct implementations; it swaps one sample's term in one row of that
# layer's update.  Two fp32 sums of the same K products in different orders differ by
# at most 2 K u sum_k |h_k w_k| (u = 2^-24); and the bf16 inputs h_k of the two can
# differ where an earlier layer's value sat on a rounding boundary, each such decision
# moving z by at most 2^-8 |h_k w_k|.  So a flip is possible only where the exact
# pre-activation is below 2 K u sum |h w| + 2 * 2^-8 max |h w| (the order bound plus two
# input decisions).  An update row beyond its bound is accepted only if some sample's
# pre-activation in that row is (the "flip ratio" |z| / that bound is at most 1), and
# every accepted row is counted.
U32 = 2.0 ** -24
U_BF16 = 2.0 ** -8


def _flip_rows(o, k, L, bad, before):
    """Rows flagged `bad` ([learners, out]) of tensor k that a provable ReLU flip
    explains, as (count, flip ratios), or (0, ratios) if any row is not explained."""
    layer = k // 2
    if layer >= L - 1 or before is None or not getattr(o.problem, "last_preacts", None):
        return 0, []
    X = o.problem.X
    rows = oracle.batch_rows_from(o.cursor - o.B, o.B, X.shape[1])
    n, ratios = 0, []
    for jj in range(bad.shape[0]):
        flagged = np.nonzero(bad[jj])[0]
        if len(flagged) == 0:
            continue
        pre = o.problem.last_preacts[jj]
        z = pre[layer]                                        # [B, out], the oracle's Z_l
        if layer == 0:
            H = oracle.bf16_round(X[jj, rows].astype(np.float32)).astype(np.float64)
        else:
            H = oracle.bf16_round(np.maximum(pre[layer - 1], 0).astype(np.float32)).astype(np.float64)
        W = oracle.bf16_round(before[2 * layer][jj].astype(np.float32)).astype(np.float64)
        K = W.shape[1]
        for r in flagged:
            prod = np.abs(H) * np.abs(W[r])                    # [B, K]
            bound = 2.0 * K * U32 * prod.sum(axis=1) + 2.0 * U_BF16 * prod.max(axis=1) + 1e-300
            ratio = float(np.min(np.abs(z[:, r]) / bound))
            ratios.append(ratio)
            if ratio > 1.0:
                return 0, ratios
            n += 1
    return n, ratios


def _check(name, k, g, want, lim, fn, o, L, report, stats, before=None):
    e = fn(g, want)
    if report is not None:
        report.append((k, name, e, lim))
    if e <= lim:
        return e
    if before is not None and fn is rel_err:
        scale = np.max(np.abs(want))
        rows = np.max(np.abs(g - want).reshape(g.shape[0], g.shape[1], -1), axis=2) / scale
        n, ratios = _flip_rows(o, k, L, rows > lim, before)
        if n:
            if stats is not None:
                stats["exempt_rows"] = stats.get("exempt_rows", 0) + n
                stats.setdefault("exempt", []).append((k, name, round(e, 5), lim, n,
                                                       [round(x, 4) for x in ratios]))
            return e
        raise AssertionError(f"tensor {k}: {name} err {e:.3e} > {lim:.3e}; flip ratios {ratios}")
    raise AssertionError(f"tensor {k}: {name} err {e:.3e} > {lim:.3e}")


def compare(ha, o, learners=None, tol=None, before=None, o_ref=None, report=None,
            end_to_end=False, stats=None):
    """Check the GPU parameters against oracle `o` (and, with `before`, the update
    itself).  Per step the parameter bound is `tol` outright.  End to end
    (`end_to_end`, with a second oracle `o_ref`), the bound widens to SPREAD times
    the oracle-vs-oracle error.  Update rows beyond their bound must be explained by
    near-zero ReLU inputs; `stats` counts them."""
    tol = TOL[ha.precision] if tol is None else tol
    utol = UPDATE_TOL[ha.precision]
    learners = list(range(ha.P)) if learners is None else learners
    got = oracle_params(ha, ha.params, learners)
    worst = 0.0
    if stats is not None:
        stats.setdefault("exempt_rows", 0)
    for k, (g, want) in enumerate(zip(got, o.params)):
        g, want = g.astype(np.float64), want.astype(np.float64)
        ref = o_ref.params[k].astype(np.float64) if o_ref is not None else None
        lim = tol
        if end_to_end and ref is not None:
            lim = max(tol, SPREAD * rel_err(ref, want))
        worst = max(worst, _check("param", k, g, want, lim, rel_err, o, ha.L, report, stats))
        if before is None:
            continue
        b0 = before[k]
        if np.max(np.abs(want - b0)) == 0:
            continue
        for name, fn in (("update-max", rel_err), ("update-frob", frob_err)):
            _check(name, k, g - b0, want - b0, utol, fn, o, ha.L, report, stats, before=before)
    return worst


SMALL_BF16 = configs.Workload("tiny_mlp_bf16", P=4, S=2, K1=2, K2=2, rounds=1,
                              dims=(256, 192, 10), precision="bf16", N=96, B=48, lr=0.05,
                              sigma_mu=0.1, init="he")
RAGGED_BF16 = configs.Workload("ragged_mlp_bf16", P=6, S=3, K1=1, K2=2, rounds=1,
                               dims=(264, 136, 200, 13), precision="bf16", N=50, B=20, lr=0.05,
                               sigma_mu=0.1, init="he")
SOFTMAX_BF16 = configs.Workload("softmax_bf16", P=4, S=2, K1=2, K2=2, rounds=1, dims=(256, 10),
                                precision="bf16", N=64, B=16, lr=0.05, sigma_mu=0.1, init="he")
WIDE_SOFTMAX_BF16 = configs.Workload("softmax_bf16_c40", P=4, S=2, K1=1, K2=2, rounds=1,
                                     dims=(256, 40), precision="bf16", N=48, B=16, lr=0.05,
                                     sigma_mu=0.1, init="he")
MANY_CLASSES_BF16 = configs.Workload("mlp_bf16_c300", P=4, S=4, K1=1, K2=2, rounds=1,
                                     dims=(128, 64, 300), precision="bf16", N=64, B=32, lr=0.05,
                                     sigma_mu=0.1, init="he")
HEAD_C13 = configs.Workload("mlp_bf16_c13", P=4, S=2, K1=1, K2=2, rounds=1, dims=(192, 128, 13),
                            precision="bf16", N=48, B=24, lr=0.05, sigma_mu=0.1, init="he")
# Head slices of 128 features (20 learners: clusters of 8 CTAs per learner would not fit
# in one wave, so 4 per learner), a ragged 320-wide layer (last slice 64 wide) and a batch
# that is not a multiple of 16.
HEAD_F128 = configs.Workload("mlp_bf16_head_f128", P=20, S=4, K1=3, K2=2, rounds=1,
                             dims=(256, 320, 10), precision="bf16", N=120, B=24, lr=0.05,
                             sigma_mu=0.1, init="he")
# Dynamic work items with both whole tiles and tail tiles split into pieces (3136
# inputs = 49 chunks: pieces of 48 and 1 chunk), 32 learners in clusters of 4: the
# pieces of a tile are summed in piece order by whichever CTA completes the tile.
FUSE_PIECES = configs.Workload("mlp_bf16_pieces", P=32, S=4, K1=3, K2=2, rounds=1,
                               dims=(3136, 1024, 10), precision="bf16", N=160, B=32, lr=0.05,
                               sigma_mu=0.1, init="he")
# The backward's pieces: the second layer's dX sums over 3136 outputs (49 chunks), so
# its tiles are split and their dX partials added in piece order.
BWD_PIECES = configs.Workload("mlp_bf16_bwd_pieces", P=32, S=4, K1=2, K2=2, rounds=1,
                              dims=(256, 256, 3136, 10), precision="bf16", N=128, B=32, lr=0.05,
                              sigma_mu=0.1, init="he")


SMALL_FP32 = configs.Workload("tiny_mlp_fp32", P=4, S=2, K1=2, K2=2, rounds=1,
                              dims=(100, 37, 10), precision="fp32", N=40, B=7, lr=0.05,
                              sigma_mu=0.1, init="he")


# Last-layer paths: the head kernels (<= 16 classes; SMALL_BF16, SOFTMAX_BF16 which reads X
# directly, the 16-learner MLP), whole steps in one launch (nets as small as HEAD_C13 and
# RAGGED_BF16), tensor-core forward with the CE in its epilogue (WIDE_SOFTMAX_BF16),
# and the standalone CE kernel (MANY_CLASSES_BF16: 300 classes over 3 tiles).
STEP_CASES = [configs.SOFTMAX_P4, SMALL_FP32, SMALL_BF16, SOFTMAX_BF16, HEAD_C13,
              WIDE_SOFTMAX_BF16, RAGGED_BF16, MANY_CLASSES_BF16, configs.MLP512_P16, FUSE_PIECES,
              BWD_PIECES]


@pytest.mark.parametrize("w", STEP_CASES, ids=lambda w: w.name)
def test_one_step_from_distinct_learners(w):
    # Learners start from different parameters, so every learner's step is checked.
    layers = perturbed_layers(w, 0.01, seed=1)
    ha, X, y = setup(w, layers)
    start = oracle_params(ha, ha.params)
    o = make_oracle(w, ha, X, y, start)
    ha.step()
    ha.check()
    o.step()
    stats = {}
    compare(ha, o, before=[a.astype(np.float64) for a in start], stats=stats)
    print(w.name, "exempt update rows:", stats["exempt_rows"], stats.get("exempt", []))
    if w is configs.MLP512_P16:
        assert stats["exempt_rows"] == 0
    gl = ha.losses().numpy()
    assert np.allclose(gl, o.problem.last_loss, rtol=1e-3, atol=1e-4)


@pytest.mark.parametrize("w", [configs.SOFTMAX_P4, SMALL_FP32, SMALL_BF16, SOFTMAX_BF16,
                               HEAD_C13, WIDE_SOFTMAX_BF16, RAGGED_BF16, MANY_CLASSES_BF16,
                               HEAD_F128, FUSE_PIECES, BWD_PIECES,
                               SMALL_BF16.replace(name="tiny_mlp_bf16_kavg", S=1)],
                         ids=lambda w: w.name)
def test_full_run_against_oracle(w):
    ha, X, y = setup(w)
    o = make_oracle(w, ha, X, y, oracle_params(ha, ha.params))
    o_ref = (make_oracle(w, ha, X, y, oracle_params(ha, ha.params), mode="bf16_acc32")
             if w.precision == "bf16" else None)
    for _ in range(w.rounds):
        ha.round()
        o.round()
        if o_ref is not None:
            o_ref.round()
    ha.check()
    report = []
    compare(ha, o, o_ref=o_ref, end_to_end=True, report=report)
    print(w.name, "end to end (err, bound):", [(k, f"{e:.2e}", f"{lim:.2e}") for k, _, e, lim in report])
    # every learner holds the same parameters after the global average
    p = ha.params.cpu().numpy().view(np.uint32)
    assert np.all(p == p[0])
    assert ha.get_step() == w.rounds * w.K1 * w.K2


# The step that closes a local block inside round() updates W_1 for groups of Q = 4
# learners of a cluster (2 where S is not a multiple of 4 or the batch exceeds 32) and
# stores only their sum in the first levels of the averaging tree; the local average
# finishes the tree from the S / Q group sums.  Cases: Q = 4 with S = 8 (two group sums
# per cluster); Q = 2 with S = 6 (three per cluster: the generic tree) and a ragged
# 200-input layer; Q = 4 with S = 12 and K1 = 1 (every step both reads the cluster
# means and writes group sums); Q = 2 because the batch is 64.
# (GROUP_S6 and GROUP_SP are small enough for whole steps in one launch, which store no group
# sums; test_group_sums_past_small_nets has them, and the others, on wider nets.)
GROUP_S8 = configs.Workload("mlp_bf16_group4_S8", P=16, S=8, K1=2, K2=3, rounds=1,
                            dims=(256, 192, 10), precision="bf16", N=128, B=32, lr=0.05,
                            sigma_mu=0.1, init="he")
GROUP_S6 = configs.Workload("mlp_bf16_group2_S6", P=12, S=6, K1=2, K2=2, rounds=1,
                            dims=(200, 136, 13), precision="bf16", N=144, B=48, lr=0.05,
                            sigma_mu=0.1, init="he")
GROUP_S12_K1 = configs.Workload("mlp_bf16_group4_S12_K1_1", P=24, S=12, K1=1, K2=3, rounds=1,
                                dims=(128, 64, 10), precision="bf16", N=64, B=16, lr=0.05,
                                sigma_mu=0.1, init="he")
GROUP_B64 = configs.Workload("mlp_bf16_group2_B64", P=8, S=4, K1=2, K2=2, rounds=1,
                             dims=(256, 128, 10), precision="bf16", N=256, B=64, lr=0.05,
                             sigma_mu=0.1, init="he")
# The first step after a compact local average forwards groups of G learners of a
# cluster with one product per weight tile (N = G * Bn <= 128).  Cases: G = 2 with a
# 48-sample batch (N = 96), a ragged 1200-wide layer, whole and tail group tiles, the
# tail split into pieces; G = 8 with a 16-sample batch, a 300-class logits layer (mode
# 1); and the 300-class net with K1 = 1, where every step but the first reads the means.
GFWD_B48 = configs.Workload("mlp_bf16_gfwd2_B48", P=32, S=2, K1=2, K2=2, rounds=1,
                            dims=(3136, 1200, 10), precision="bf16", N=192, B=48, lr=0.05,
                            sigma_mu=0.1, init="he")
GFWD_B16 = configs.Workload("mlp_bf16_gfwd8_B16", P=32, S=8, K1=2, K2=2, rounds=1,
                            dims=(1024, 1152, 300), precision="bf16", N=64, B=16, lr=0.05,
                            sigma_mu=0.1, init="he")


# S = 1 (K-AVG: the local average is the identity, every average in place); one cluster
# of all 8 learners (S = P, quad sums and groups of 4); and 150 rows per learner with a
# 32-row batch, so that batches straddle the end of the data set (the gather path, also
# in the grouped forward, and steps whose successor's batch is not contiguous).
KAVG_BF16 = SMALL_BF16.replace(name="tiny_mlp_bf16_kavg", S=1)
GROUP_SP = configs.Workload("mlp_bf16_group4_S8_P8", P=8, S=8, K1=2, K2=2, rounds=1,
                            dims=(256, 192, 10), precision="bf16", N=128, B=32, lr=0.05,
                            sigma_mu=0.1, init="he")
PIECES_WRAP = FUSE_PIECES.replace(name="mlp_bf16_pieces_wrap", N=150)


# round() writes each intermediate local average as one mean row per cluster, read by
# the next step, and fuses the last local average into the global one; the literal
# sequence writes every row each time.  Cases: clusters of 2 (group sums of 2: one per
# cluster); clusters of 3 over a ragged three-layer net (the generic, non-power-of-two
# averaging path, with K1 = 1: a compact average after every step but the last; no
# groups); 5 clusters of 4 (a global tree over a non-power-of-two count of clusters),
# head slices of 128 features; the group update and group forward cases above.
@pytest.mark.parametrize("w", [SMALL_BF16, RAGGED_BF16.replace(K2=3), HEAD_F128, GROUP_S8,
                               GROUP_S6, GROUP_S12_K1, GROUP_B64, GFWD_B48, GFWD_B16,
                               MANY_CLASSES_BF16.replace(K2=3), KAVG_BF16, GROUP_SP,
                               PIECES_WRAP],
                         ids=lambda w: w.name)
def test_literal_sequence_equals_round(w):
    # step/local_average/global_average in Algorithm 1's order give the same bits
    # as round()
    ha1, X, y = setup(w, perturb=(0.01, 0.01))
    ha2, _, _ = setup(w, perturb=(0.01, 0.01))
    ha1.round()
    for b in range(w.K2):
        for k in range(w.K1):
            ha2.step()
        ha2.local_average()
    ha2.global_average()
    torch.cuda.synchronize()
    assert torch.equal(ha1.params.view(torch.int32), ha2.params.view(torch.int32))


# Inside round(), a step whose successor starts no local block and reads a contiguous
# batch also computes that successor's first-layer output (update+forward kernel, same
# schedule and arithmetic as the forward).  Cases: ragged 192-wide layer in cluster
# split-K mode; the 16-learner MLP (cluster split-K, cq = 2); 128 tiles in stream-K mode
# with K1 = 3, so the middle step both consumes and produces a fused H_1.
FUSE_STREAMK = configs.Workload("mlp_bf16_streamk", P=16, S=4, K1=3, K2=2, rounds=1,
                                dims=(512, 1024, 10), precision="bf16", N=200, B=32, lr=0.05,
                                sigma_mu=0.1, init="he")
# Three layers: the first layer's update computes the next H_1, the last layer keeps its
# own kernel (it does not follow the first).
FUSE_THREE = configs.Workload("mlp3_bf16_fused", P=4, S=2, K1=3, K2=2, rounds=1,
                              dims=(256, 320, 192, 10), precision="bf16", N=160, B=32, lr=0.05,
                              sigma_mu=0.1, init="he")


def _fused_steps(w):
    return sum(1 for t in range(w.K1 * w.K2)
               if t % w.K1 != w.K1 - 1 and ((t + 1) * w.B) % w.N + w.B <= w.N)


@pytest.mark.parametrize("w", [SMALL_BF16, configs.MLP512_P16.replace(N=512), FUSE_STREAMK,
                               FUSE_THREE, FUSE_PIECES, BWD_PIECES], ids=lambda w: w.name)
def test_fused_next_forward_equals_steps(w):
    ha1, X, y = setup(w, perturb=(0.01, 0.01))
    ha2, _, _ = setup(w, perturb=(0.01, 0.01))
    ha1.profile(["update_forward", "forward"])
    n0 = ha1.launches()
    ha1.round()
    n_round = ha1.launches() - n0
    n_fused = ha1.profile_read("update_forward").launches
    n_fwd = ha1.profile_read("forward").launches
    ha1.profile(False)
    steps, L = w.K1 * w.K2, len(w.dims) - 1
    assert n_fused == _fused_steps(w) > 0
    # forward launches: every layer before the head kernel, less the fused first layers
    assert n_fwd == steps * (L - 1) - n_fused
    n1 = ha2.launches()
    for b in range(w.K2):
        for k in range(w.K1):
            ha2.step()
        ha2.local_average()
    ha2.global_average()
    # the literal sequence launches every kernel; round() saves the fused forwards and
    # fuses the last local average into the global one.  With S even, each of the K2
    # block ends stores group sums of W_1, and with quads (S a multiple of 4, B <= 32)
    # of every later tensor-core layer's W too (a backward without update, then the
    # grouped update); its average takes one launch per column range (each grouped W
    # region and the range after it).
    head = w.dims[-1] <= 16
    quads = w.S % 4 == 0 and w.B <= 32
    n_grouped = (len(w.dims) - 1 - (1 if head else 0)) if quads else 1
    extra = (n_grouped - 1) + (2 * n_grouped - 1) if w.S % 2 == 0 else 0
    saved = n_fused + 1 - w.K2 * extra
    assert ha2.launches() - n1 == n_round + saved
    ha1.check()
    ha2.check()
    assert torch.equal(ha1.params.view(torch.int32), ha2.params.view(torch.int32))
    assert torch.equal(ha1.losses(), ha2.losses())


# Free global interval (Sec. 3.1: beta = G / K1 need not be an integer; Sec. 4's ImageNet
# run uses K1 = 20 and G = 43) with a diminishing step size gamma_n = gamma_0 / (n + 1)
# (Theorem 3.3), two rounds each, against the oracle.
FREE_G = [(SMALL_FP32, 5), (SMALL_BF16, 3), (FUSE_THREE, 7), (SMALL_BF16.replace(K1=3), 7)]


@pytest.mark.parametrize("w,G", FREE_G, ids=lambda v: getattr(v, "name", str(v)))
def test_free_global_interval_against_oracle(w, G):
    ha, X, y = setup(w)
    ha.set_global_steps(G)
    start = oracle_params(ha, ha.params)
    o = make_oracle(w, ha, X, y, start)
    o.G = G
    o_ref = (make_oracle(w, ha, X, y, start, mode="bf16_acc32") if w.precision == "bf16" else None)
    if o_ref is not None:
        o_ref.G = G
    for n in range(2):
        lr = w.lr / (n + 1)
        ha.set_lr(lr)
        for oo in (o, o_ref):
            if oo is not None:
                oo.lr = lr
                oo.round()
        ha.round()
    ha.check()
    compare(ha, o, o_ref=o_ref, end_to_end=True)
    p = ha.params.cpu().numpy().view(np.uint32)
    assert np.all(p == p[0])                      # the round ends with the global average
    assert ha.get_step() == 2 * G


@pytest.mark.parametrize("w,G", [(SMALL_BF16.replace(K1=3), 7), (FUSE_THREE, 6)],
                         ids=lambda v: getattr(v, "name", str(v)))
def test_free_global_interval_literal_sequence(w, G):
    # round() with G steps equals the calls it stands for, bit for bit: a local average
    # after every K1-th step, the global average after the G-th (preceded by a local
    # average exactly when K1 divides G)
    ha1, X, y = setup(w, perturb=(0.01, 0.01))
    ha2, _, _ = setup(w, perturb=(0.01, 0.01))
    ha1.set_global_steps(G)
    ha1.round()
    for r in range(1, G + 1):
        ha2.step()
        if r % w.K1 == 0:
            ha2.local_average()
    ha2.global_average()
    ha1.check()
    ha2.check()
    assert torch.equal(ha1.params.view(torch.int32), ha2.params.view(torch.int32))


# Per-round batch size B_n (Theorem 3.3's growing batches; a shrinking step is included
# to check that rows beyond the batch add nothing), each learner reading its data
# sequentially, with a diminishing step size; against the oracle.
BATCH_SCHED = [(SMALL_FP32, (3, 7, 5)), (SMALL_BF16, (16, 48, 32)), (FUSE_THREE, (8, 32, 24)),
               (RAGGED_BF16, (12, 20, 7))]


@pytest.mark.parametrize("w,sched", BATCH_SCHED, ids=lambda v: getattr(v, "name", str(v)))
def test_batch_schedule_against_oracle(w, sched):
    ha, X, y = setup(w)
    start = oracle_params(ha, ha.params)
    o = make_oracle(w, ha, X, y, start)
    o_ref = (make_oracle(w, ha, X, y, start, mode="bf16_acc32") if w.precision == "bf16" else None)
    for n, Bn in enumerate(sched):
        ha.set_batch(Bn)
        ha.set_lr(w.lr / (n + 1))
        for oo in (o, o_ref):
            if oo is not None:
                oo.B, oo.lr = Bn, w.lr / (n + 1)
                oo.round()
        ha.round()
    ha.check()
    compare(ha, o, o_ref=o_ref, end_to_end=True)
    gl = ha.losses().numpy()
    assert np.allclose(gl, o.problem.last_loss, rtol=2e-3, atol=1e-4)


def test_batch_schedule_literal_sequence():
    w = SMALL_BF16.replace(K1=3)
    ha1, X, y = setup(w, perturb=(0.01, 0.01))
    ha2, _, _ = setup(w, perturb=(0.01, 0.01))
    for Bn in (48, 16, 32):
        ha1.set_batch(Bn)
        ha1.round()
        ha2.set_batch(Bn)
        for b in range(w.K2):
            for k in range(w.K1):
                ha2.step()
            ha2.local_average()
        ha2.global_average()
    ha1.check()
    ha2.check()
    assert torch.equal(ha1.params.view(torch.int32), ha2.params.view(torch.int32))


def _force(ha, *oracles):
    """Load the GPU's current learner state into the oracles (teacher forcing)."""
    state = oracle_params(ha, ha.params)
    for o in oracles:
        o.params = [a.copy() for a in state]
        o.t = ha.get_step()
    return [a.astype(np.float64) for a in state]


@pytest.mark.parametrize("w", [configs.MLP512_P16, SMALL_BF16], ids=lambda w: w.name)
def test_round_teacher_forced(w):
    # Every local step of a round checked from the GPU's own pre-step state
    # (1e-2, and the update itself within 2e-2), every average bit-exact.
    ha, X, y = setup(w)
    o = make_oracle(w, ha, X, y, oracle_params(ha, ha.params))
    worst = 0.0
    stats = {}
    for b in range(w.K2):
        for k in range(w.K1):
            before = _force(ha, o)
            ha.step()
            o.step()
            worst = max(worst, compare(ha, o, before=before, stats=stats))
        _force(ha, o)
        if b + 1 < w.K2:
            ha.local_average()
            o.local_average()
        else:
            ha.local_average()
            ha.global_average()
            o.local_average()
            o.global_average()
        got = oracle_params(ha, ha.params)
        for g, want in zip(got, o.params):
            assert np.array_equal(g.view(np.uint32), want.view(np.uint32))
    ha.check()
    print(f"{w.name}: worst per-step rel err {worst:.3e}; exempt update rows "
          f"{stats['exempt_rows']} {stats.get('exempt', [])}")


def test_mlp512_round_end_to_end():
    # A whole round without teacher forcing: decision flips compound over the
    # K1*K2 steps, so the bound is SPREAD times the oracle-vs-oracle drift.
    w = configs.MLP512_P16
    ha, X, y = setup(w)
    o = make_oracle(w, ha, X, y, oracle_params(ha, ha.params))
    o_ref = make_oracle(w, ha, X, y, oracle_params(ha, ha.params), mode="bf16_acc32")
    ha.round()
    o.round()
    o_ref.round()
    ha.check()
    report = []
    compare(ha, o, o_ref=o_ref, end_to_end=True, report=report)
    print(w.name, "end-to-end:", [(k, f"{e:.2e}", f"{lim:.2e}") for k, _, e, lim in report])


@pytest.mark.parametrize("w", [configs.MLP2048_P64, configs.MLP4096_P32], ids=lambda w: w.name)
def test_full_size_step_sampled(w):
    # Full-size model, P and B (the launch configuration the bench times); the
    # oracle recomputes the first and the last learner one by one.
    w = w.replace(N=4 * w.B)
    ha, X, y = setup(w, data_device="cuda", perturb=(0.002, 0.05))
    learners = [0, w.P - 1]
    start = oracle_params(ha, ha.params, learners)
    o = make_oracle(w, ha, X, y, start, learners)
    ha.step()
    ha.check()
    o.step()
    report, stats = [], {}
    compare(ha, o, learners, before=[a.astype(np.float64) for a in start], report=report,
            stats=stats)
    print(w.name, [(k, kind, f"{e:.2e}", f"{lim:.2e}") for k, kind, e, lim in report])
    # parameters within 1e-2 outright; update rows beyond 2e-2 only where a ReLU flip is
    # provable, at most one row in a thousand
    print(w.name, "exempt update rows:", stats["exempt_rows"], stats.get("exempt", []))
    rows = sum(ha.dims[1:-1]) * len(learners)
    assert stats["exempt_rows"] <= rows // 1000, stats.get("exempt")


# The full-size workloads in the launch configuration the bench times: a round (compact
# averages, quad- or pair-sum block-end updates, grouped forwards of each block's first
# step, fused update+forwards, tail pieces) gives the bits of the literal step / local /
# global sequence, and every learner holds the same parameters after it.
@pytest.mark.parametrize("w", [configs.MLP2048_P64, configs.MLP4096_P32], ids=lambda w: w.name)
def test_full_size_round_equals_literal_sequence(w):
    w = w.replace(N=2 * w.B * w.K1)
    ha1, X, y = setup(w, data_device="cuda", perturb=(0.002, 0.05))
    ha2, _, _ = setup(w, data_device="cuda", perturb=(0.002, 0.05))
    ha1.round()
    for b in range(w.K2):
        for k in range(w.K1):
            ha2.step()
        ha2.local_average()
    ha2.global_average()
    ha1.check()
    ha2.check()
    assert torch.equal(ha1.params.view(torch.int32), ha2.params.view(torch.int32))
    assert torch.equal(ha1.losses(), ha2.losses())
    p = ha1.params.view(torch.int32)
    assert torch.equal(p, p[:1].expand_as(p))


# A parameter row of 4.2M values and 512 KB of rows per learner and step: spans of at
# least 64 rows go learner by learner; the chunk of steps 2-3 wraps around N = 160 and
# leaves a 32-row span, which goes as one pitched copy.
HOST_ROWS = configs.Workload("mlp_bf16_host_rows", P=4, S=2, K1=2, K2=2, rounds=1,
                             dims=(4096, 1024, 10), precision="bf16", N=160, B=64, lr=0.05,
                             sigma_mu=0.1, init="he")


# bf16 path: the rows are copied beside the kernels in chunks of steps that double in
# length; SMALL_BF16's round reads more rows than each learner has (the chunks wrap
# around N), FUSE_PIECES has 6 steps (chunks 0 | 1 | 2-3 | 4-5), a free global interval
# of 7 steps ends on a short chunk.  fp32 path: the rows are copied ahead of the round.
@pytest.mark.parametrize("w,G", [(SMALL_BF16, 0), (FUSE_THREE, 0), (FUSE_PIECES, 0),
                                 (SMALL_BF16.replace(K1=3), 7), (SMALL_FP32, 0), (HOST_ROWS, 0)],
                         ids=lambda v: getattr(v, "name", str(v)))
def test_round_host_matches_device_round(w, G):
    ha1, X, y = setup(w)
    ha2, _, _ = setup(w)
    for h in (ha1, ha2):
        h.set_global_steps(G)
    Xh, yh = X.pin_memory(), y.pin_memory()
    for _ in range(2):                  # the second round starts mid data set
        ha1.round()
        loss = ha2.round_host(Xh, yh)
        torch.cuda.synchronize()
        assert torch.equal(ha1.params, ha2.params)
        assert torch.allclose(loss, ha1.losses())


# The bound device data set starts empty, so every row that a step reads has to be copied
# by the round itself: chunk boundaries, the wrap around N, and a second round that
# starts mid data set.
@pytest.mark.parametrize("w,G", [(FUSE_THREE, 0), (FUSE_PIECES, 0), (SMALL_BF16.replace(K1=3, N=700), 11),
                                 (SMALL_BF16.replace(K1=3), 7), (SMALL_FP32, 0), (HOST_ROWS, 0)],
                         ids=lambda v: getattr(v, "name", str(v)))
def test_round_host_copies_every_row_it_reads(w, G):
    ha1, X, y = setup(w)
    ha2 = HierAvg(w.P, w.S, w.K1, w.K2, w.lr, w.B, w.dims, w.precision)
    ha2.bind(ha1.params.clone(), torch.zeros_like(X, device="cuda"), torch.zeros_like(y, device="cuda"))
    for h in (ha1, ha2):
        h.set_global_steps(G)
    Xh, yh = X.pin_memory(), y.pin_memory()
    for _ in range(2):
        ha1.round()
        loss = ha2.round_host(Xh, yh)
        torch.cuda.synchronize()
        assert torch.equal(ha1.params, ha2.params)
        assert torch.allclose(loss, ha1.losses())


def test_resume_from_saved_step():
    w = SMALL_BF16
    ha1, X, y = setup(w)
    ha1.round()
    saved = ha1.params.clone()
    ha1.round()
    ha2, _, _ = setup(w)
    ha2.params.copy_(saved)
    ha2.set_step(w.K1 * w.K2)
    ha2.round()
    torch.cuda.synchronize()
    assert torch.equal(ha1.params, ha2.params)


# fp32 kernels at the edges of their tiles: tiles of 8, 16, 32 and 64 samples with one
# sample missing or too many; widths that are no multiple of 4 (4-byte copies) or end inside
# a 64-wide chunk; a reduction split over a cluster of 8 (one learner, 2048 inputs); the
# small last layer at its limits (16 classes, 64 samples, slices of 64 features, one odd
# slice) and just past them (17 classes, 65 samples, more than 8 x 1024 features).  (The smaller
# of these nets run whole steps in one launch; the last three are past that.)
def _fp32(dims, P, S, B, **kw):
    return configs.Workload("fp32_" + "-".join(map(str, dims)) + f"_P{P}_B{B}", P=P, S=S, K1=kw.get("K1", 2),
                            K2=2, rounds=1, dims=dims, precision="fp32", N=kw.get("N", 3 * B + 1), B=B,
                            lr=0.05, sigma_mu=0.1, init="he")


FP32_CASES = [_fp32((64, 64, 17), 4, 2, 8), _fp32((130, 65, 40), 3, 1, 9), _fp32((260, 132, 128, 300), 2, 2, 33),
              _fp32((100, 36, 10), 2, 1, 65), _fp32((2048, 64, 10), 1, 1, 32), _fp32((96, 72, 40), 2, 1, 130),
              _fp32((3072, 10), 2, 2, 64), _fp32((512, 16), 3, 1, 1), _fp32((37, 10), 4, 4, 17),
              _fp32((70, 5), 2, 2, 3), _fp32((8200, 10), 1, 1, 2), _fp32((516, 61, 16), 2, 1, 16),
              _fp32((516, 61, 16), 2, 1, 31), _fp32((2048, 200, 10), 1, 1, 7), _fp32((3000, 61, 16), 2, 1, 16),
              _fp32((2048, 64, 17), 1, 1, 31), _fp32((8200, 10), 1, 1, 32)]


@pytest.mark.parametrize("w", FP32_CASES, ids=lambda w: w.name)
def test_fp32_step_at_tile_edges(w):
    test_one_step_from_distinct_learners(w)


# One-layer fp32 models run the steps between two averages in one launch: the bits of the
# single steps, with batches that wrap around the data set, a last block shorter than K1,
# one batch buffer instead of two (64 samples of 3072 features), and 4-byte copies.
@pytest.mark.parametrize("w,G", [(configs.SOFTMAX_P4, 0), (_fp32((3072, 10), 4, 2, 64), 5),
                                 (_fp32((37, 13), 6, 3, 5, K1=3, N=11), 7)],
                         ids=lambda v: getattr(v, "name", str(v)))
def test_fp32_steps_in_one_launch(w, G):
    ha1, X, y = setup(w, perturb=(0.01, 0.01))
    ha2, _, _ = setup(w, perturb=(0.01, 0.01))
    ha1.set_global_steps(G)
    for _ in range(2):
        ha1.round()
        n = G or w.K1 * w.K2
        for r in range(1, n + 1):
            ha2.step()
            if r % w.K1 == 0:
                ha2.local_average()
        ha2.global_average()
    torch.cuda.synchronize()
    assert ha1.get_step() == ha2.get_step() == 2 * n
    assert torch.equal(ha1.params.view(torch.int32), ha2.params.view(torch.int32))
    assert torch.equal(ha1.losses(), ha2.losses())


# The one-kernel last layer on input widths that are no multiple of 64: the narrowest (8
# features, half an MMA step), a width over 4 and over 8 CTAs whose last slice ends on an
# odd multiple of 8, one class and 16, a one-layer model whose batches wrap, and a wide
# one; over 1024 features behind a hidden layer, or 40 classes, stay with the cross-entropy in
# the forward's epilogue.  The last two have 464 and 512 CTAs, four to an SM.
def _head(dims, P, S, B, N):
    return configs.Workload("head_" + "-".join(map(str, dims)) + f"_P{P}_B{B}", P=P, S=S, K1=2, K2=2, rounds=1,
                            dims=dims, precision="bf16", N=N, B=B, lr=0.05, sigma_mu=0.1, init="he")


HEAD_CASES = [_head((4096, 8, 10), 4, 2, 64, 256), _head((600, 200, 13), 6, 3, 20, 50),
              _head((128, 1000, 16), 24, 4, 33, 132), _head((4096, 520, 1), 2, 1, 1, 4),
              _head((3336, 10), 4, 4, 64, 90), _head((4104, 16), 2, 2, 64, 256), _head((64, 1032, 16), 2, 2, 64, 256),
              _head((264, 200, 40), 6, 3, 20, 50), _head((3072, 10), 58, 2, 16, 40), _head((64, 512, 13), 128, 4, 20, 60)]


@pytest.mark.parametrize("w", HEAD_CASES, ids=lambda w: w.name)
def test_head_widths(w):
    test_one_step_from_distinct_learners(w)
    test_literal_sequence_equals_round(w)


# Whole steps of a small net in one launch, several between two averages: one to four layers,
# widths below the eight slices of a learner and of odd length, 1 to 32 classes, batches of 1
# to 64 that wrap around the data set (more than once in one launch), a last block shorter
# than K1, odd clusters, and 16 learners or more, two CTAs to an SM (1000-120-8 is just too large
# for that and takes the kernels per layer).
def _small(dims, precision, P, S, B, K1, N):
    return configs.Workload(f"small_{precision}_" + "-".join(map(str, dims)) + f"_P{P}_B{B}", P=P, S=S, K1=K1,
                            K2=2, rounds=1, dims=dims, precision=precision, N=N, B=B, lr=0.05, sigma_mu=0.1,
                            init="he")


SMALL_CASES = [_small((100, 37, 10), "fp32", 4, 2, 7, 2, 40), _small((5, 3, 2), "fp32", 3, 3, 1, 3, 2),
               _small((33, 64, 65, 7, 32), "fp32", 6, 2, 33, 2, 50), _small((300, 31), "fp32", 1, 1, 64, 3, 100),
               _small((264, 136, 200, 13), "bf16", 6, 3, 20, 4, 50), _small((8, 8, 1), "bf16", 2, 2, 1, 2, 1),
               _small((784, 40, 10), "bf16", 15, 5, 64, 3, 192), _small((136, 104, 88, 72, 32), "bf16", 5, 5, 17, 2, 20),
               _small((1024, 17), "bf16", 18, 6, 48, 5, 96), _small((1000, 120, 8), "bf16", 16, 4, 16, 2, 64),
               _small((520, 72, 8), "bf16", 16, 4, 16, 2, 64)]


@pytest.mark.parametrize("w", SMALL_CASES, ids=lambda w: w.name)
def test_small_net_steps(w):
    test_one_step_from_distinct_learners(w)
    test_free_global_interval_literal_sequence(w, 2 * w.K1 + 1)
    test_literal_sequence_equals_round(w)
    test_round_host_matches_device_round(w, 0)
    test_round_host_copies_every_row_it_reads(w, 2 * w.K1 + 1)


# The group-sum and head cases above on nets past the one-launch steps' size, so that quads,
# pairs with three group sums per cluster, one cluster of all learners and 4 CTAs of the head
# per learner stay covered.
@pytest.mark.parametrize("w", [GROUP_S8.replace(dims=(512, 384, 10)), GROUP_S6.replace(dims=(392, 264, 13)),
                               GROUP_S12_K1.replace(dims=(512, 512, 10)), GROUP_SP.replace(dims=(512, 384, 10)),
                               HEAD_F128.replace(dims=(512, 320, 10)),
                               RAGGED_BF16.replace(dims=(520, 264, 328, 13))], ids=lambda w: w.name)
def test_group_sums_past_small_nets(w):
    test_one_step_from_distinct_learners(w)
    test_literal_sequence_equals_round(w)


# The backward of few long tiles in pieces of one promotion segment: a last piece of one chunk,
# a ragged layer, 48 chunks in 12 pieces (the last length that is not split in pieces of 48), and
# a class layer whose dX is split.
@pytest.mark.parametrize("w", [_head((128, 512, 1088, 10), 2, 2, 32, 128), _head((64, 200, 1608, 13), 3, 1, 20, 50),
                               _head((64, 256, 3072, 10), 2, 1, 64, 256), _head((64, 264, 1500), 4, 2, 16, 64)],
                         ids=lambda w: w.name)
def test_backward_in_segment_pieces(w):
    test_one_step_from_distinct_learners(w)
    test_literal_sequence_equals_round(w)


# The pieces' partials are the sums that a whole tile adds in the same order.  12 learners of this
# net have room for a static step's scratch only without them (a plan of whole tiles), 11 with
# them; learners are independent until they are averaged and nothing else of the plan depends on
# their number here, so the steps of the first 11 have to give the same bits.
def test_backward_in_segment_pieces_gives_the_bits_of_whole_tiles():
    dims = (13056, 128, 3072, 10)
    whole = _head(dims, 12, 1, 64, 128)
    partials = 12 * 128 * 64 * 4                                  # of one learner: 12 pieces
    ha = {}
    X, y = learner_data(whole)
    layers = perturbed_layers(whole, 0.01, seed=7)
    for P in (11, 12):
        w = whole.replace(P=P)
        ha[P] = HierAvg(P, 1, w.K1, w.K2, w.lr, w.B, dims, w.precision)
        ha[P].bind(ha[P].pack(layers[:P]), X[:P].contiguous().cuda(), y[:P].contiguous().cuda())
        for _ in range(2):
            ha[P].step()
        ha[P].check()
    assert ha[12].workspace_bytes <= 32 << 20 < ha[12].workspace_bytes + 12 * partials
    per_learner = ha[12].workspace_bytes / 12
    assert ha[11].workspace_bytes > 11 * (per_learner + 0.9 * partials)
    assert torch.equal(ha[11].params.view(torch.int32), ha[12].params[:11].view(torch.int32))
    assert torch.equal(ha[11].losses(), ha[12].losses()[:11])


# An fp32 data set may start anywhere (bind asks for 16 bytes in bf16 only): where the widths are
# multiples of four, 4-byte copies of its rows meet 16-byte copies of the weights.  Which copies
# move the operands changes no sum: the bits of the aligned data set.  A small net, one layer
# (several steps per launch), and tiles with a last layer's kernel of their own and without.
@pytest.mark.parametrize("w", [_fp32((100, 37, 10), 4, 2, 7), _fp32((3072, 10), 2, 2, 20),
                               _fp32((784, 512, 10), 2, 1, 33), _fp32((260, 132, 300), 2, 2, 65)],
                         ids=lambda w: w.name)
@pytest.mark.parametrize("offset", [1, 2])
def test_fp32_rows_off_16_bytes(w, offset):
    X, y = learner_data(w)
    layers = perturbed_layers(w, 0.01, seed=5)
    buf = torch.empty(X.numel() + offset, dtype=torch.float32, device="cuda")
    shifted = buf[offset:].view(X.shape)
    shifted.copy_(X)
    assert shifted.data_ptr() % 16 != 0
    runs = []
    for rows in (X.cuda(), shifted):
        ha = HierAvg(w.P, w.S, w.K1, w.K2, w.lr, w.B, w.dims, w.precision)
        ha.bind(ha.pack(layers), rows, y.cuda())
        ha.round()
        ha.step()
        ha.check()
        runs.append(ha)
    assert torch.equal(runs[0].params.view(torch.int32), runs[1].params.view(torch.int32))
    assert torch.equal(runs[0].losses(), runs[1].losses())


# The cross-entropy over a cluster: fewer samples than its CTAs, a last CTA with fewer than
# the others, more samples than threads, just past and just below the logits from which on it is
# spread (12288), class slices of one partial tile and of more than one tile of 128 with an odd rest.
# In bf16 with one wave of the other kernel's CTAs up to 48 classes per sample, both sides of that;
# few samples where those CTAs are more than a wave.
# (300 samples: the mean gradient is small, and the update's bound of 1e-5 has to hold over half
# an ulp of a weight of 0.6, 3e-8: at lr = 0.05 that is 1.2e-5 of the update, at 1 6e-7.)
XENT_CASES = [_fp32((40, 36, 1500), 2, 1, 9), _fp32((64, 65), 2, 1, 300).replace(lr=1.0),
              _fp32((40, 33), 3, 1, 373).replace(lr=1.0), _fp32((40, 33), 3, 1, 372).replace(lr=1.0),
              _small((64, 72, 2459), "bf16", 2, 2, 5, 2, 20), _small((64, 72, 1100), "bf16", 3, 1, 64, 2, 130),
              _small((72, 2056), "bf16", 2, 1, 33, 1, 50), _small((64, 136, 193), "bf16", 2, 2, 64, 2, 130),
              _small((64, 136, 191), "bf16", 2, 2, 64, 2, 130), _small((64, 64, 3073), "bf16", 64, 8, 4, 2, 16),
              _small((64, 64, 1025), "bf16", 100, 4, 13, 2, 40), _small((64, 72, 1537), "bf16", 2, 2, 32, 2, 70),
              _small((64, 72, 1536), "bf16", 2, 2, 32, 2, 70)]


@pytest.mark.parametrize("w", XENT_CASES, ids=lambda w: w.name)
def test_cross_entropy_over_a_cluster(w):
    test_one_step_from_distinct_learners(w)
