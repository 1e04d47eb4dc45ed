"""The bounded wait of the bounded-row engine's cluster exchange: with the test
hook CTA 1 of every cluster keeps its second step's delta from the others, so
their waits run out (about a second).  The call reports FV_ETIMEOUT, the
context stays usable, and ordinary calls after it are exact.  The engines with
backpointer rows, which ordinary calls reach through a smaller workspace, have
the same check there."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def run_case(K, lengths, how, compact=False):
    import paper_2510_19301_gb300 as fv
    from paper_2510_19301_gb300 import _lib as L
    L.load(build_if_missing=True)
    rng = np.random.default_rng(77 + K)
    log_pi, logA = W.random_model(K, rng)
    E = [W.gaussian_emissions(t, K, rng) for t in lengths]
    m = fv.Model(log_pi, logA)
    b = fv.Batch(lengths, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m])

    def decoder(flags):
        ws = torch.empty(fv.workspace_min_size([m], b, **how), dtype=torch.uint8, device="cuda") if compact else None
        return fv.Decoder([m], b, flags=flags, workspace=ws, **how)

    dec = decoder(L.FV_TEST_WITHHOLD_STEP)
    dec.launch()
    torch.cuda.synchronize()
    assert dec.device_status() == L.FV_ETIMEOUT
    hmm = oracle.HMM(log_pi, logA)
    pick = list(range(0, len(lengths), max(1, len(lengths) // 12)))
    if how.get("mode") == "beam":
        ref = [oracle.beam(hmm, E[i], how["B"])[:2] for i in pick]
    else:
        ref = [oracle.viterbi(hmm, E[i]) for i in pick]
    off = np.concatenate([[0], np.cumsum(lengths)])
    for _ in range(2):
        paths, scores = decoder(0)()
        paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
        for i, (p, s) in zip(pick, ref):
            assert np.array_equal(paths[off[i]:off[i + 1]], p)
            assert np.float32(scores[i]).view(np.int32) == np.float32(s).view(np.int32)


# clusters of 2, 8, 2, 4 and 8 CTAs
@pytest.mark.parametrize("K,lengths", [(200, [5, 9, 3]), (300, [5, 9, 3]), (1000, [5, 9, 3]), (1100, [5, 9, 3]),
                                       (2100, [2, 40, 33])])
def test_withheld_step(K, lengths):
    run_case(K, lengths, {})


# several jobs side by side in a cluster, some of them over before the others
# wait: two-step sequences, and one-step ones that never wait for the hook
@pytest.mark.parametrize("K,n", [(256, 1500), (256, 500), (512, 120)])
def test_withheld_step_with_many_jobs_per_cluster(K, n):
    lengths = [1 + (i * 7) % 12 for i in range(n)]
    run_case(K, lengths, {})


@pytest.mark.parametrize("K", [900, 1100])
def test_withheld_step_of_a_cluster_beam(K):
    run_case(K, [5, 9, 3], dict(mode="beam", B=60, P=0))


@pytest.mark.parametrize("K", [300, 1000, 1100, 2100])
def test_withheld_step_of_the_backpointer_engines(K):
    run_case(K, [5, 9, 3], {}, compact=True)
