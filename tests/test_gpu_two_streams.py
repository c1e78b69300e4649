"""Two sessions on two streams of one device, each driven by its own thread: their launches share the SMs in any mixture, and
what a session computes must not depend on it."""
import threading

import pytest
import torch

import synthetic_inputs as si

pytestmark = pytest.mark.gpu

# wide enough that the last tiles of most maps of a prompt pass are done in pieces
SHAPE = si.ModelShape("pieces", 2, 1536, 12, 4, 128, 4224, 2003, "bf16", 1e-5, 10000.0)
LENGTHS = (77, 300, 17, 129, 500, 64, 256, 411)


@pytest.fixture(scope="module")
def kb():
    from paper_2505_16162_b200 import build
    build.build()
    from paper_2505_16162_b200 import binding
    return binding


def _prompts(sess, seed, rounds):
    """Prompts of all lengths, several times over: first token and pooled state of each."""
    return [sess.prefill(si.uniform_tokens(seed, r, n, SHAPE.vocab).numpy(), want_pooled=True) for r in range(rounds) for n in LENGTHS]


def _after(sess, seed):
    """What the last prompt left in the K/V cache, as the logits of one pass."""
    return sess.verify(si.uniform_tokens(seed, 100, 3, SHAPE.vocab).numpy(), want_logits=True)["logits"]


def test_prompts_of_two_sessions_at_once_equal_the_serial_ones(kb):
    w = si.make_model_weights(SHAPE, 4, device="cuda", gain_spread=0.1)
    streams = [torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-1)]
    torch.cuda.synchronize()
    sess = [kb.Session.from_shape(SHAPE, w, 600, max_draft=4, stream=s) for s in streams]
    rounds = 6
    want = [(_prompts(sess[i], i, rounds), _after(sess[i], i)) for i in range(2)]
    got, errors = [None, None], []

    def work(i):
        try:
            with torch.cuda.stream(streams[i]):
                got[i] = _prompts(sess[i], i, rounds)
        except Exception as e:                                   # reported by the thread that started this one
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(2):
        assert all(f0 == f1 and torch.equal(p0, p1) for (f0, p0), (f1, p1) in zip(want[i][0], got[i], strict=True))
        assert torch.equal(want[i][1], _after(sess[i], i))


def test_an_error_is_reported_to_the_session_that_met_it(kb):
    """One session's logits hold no finite value, another's are sound: every call of the first says so, none of the second does."""
    shape = si.SHAPES["tiny"]
    sound = si.make_model_weights(shape, 0, device="cuda")
    bad = dict(sound, final_norm=torch.full_like(sound["final_norm"], float("nan")))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    sess = [kb.Session.from_shape(shape, w, 96, max_draft=4, stream=s) for w, s in zip((bad, sound), streams)]
    prompt = si.uniform_tokens(0, 0, 20, shape.vocab).numpy()
    first = sess[1].prefill(prompt)
    seen, errors = [], []

    def sick():
        for _ in range(150):
            try:
                sess[0].prefill(prompt)
                seen.append(0)
            except kb.KnnssdError as e:
                seen.append(e.status)

    def well():
        for _ in range(150):
            try:
                if sess[1].prefill(prompt) != first:
                    errors.append("another token")
            except kb.KnnssdError as e:
                errors.append(str(e))

    threads = [threading.Thread(target=f) for f in (sick, well)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
    assert seen == [5] * 150


def test_stand_alone_operators_from_several_threads(kb):
    """Scratch from the shared pool, words of pinned memory per thread: what a call returns must not depend on the others'."""
    g = torch.Generator(device="cuda").manual_seed(3)
    def rand(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    jobs = []
    for i in range(4):
        logits = 1.4 * rand(5, 3000 + 517 * i)
        p = kb.knnssd_filtered_probs(logits, 1.0, 0.95)
        q = kb.knnssd_filtered_probs(logits[:4] + 0.3 * rand(4, logits.shape[1]), 1.0, 0.95)
        x = rand(200 + 40 * i, 96)
        jobs.append({"p": p, "q": q, "drafts": q.argmax(dim=1).cpu().numpy(), "anchors": rand(30 + i, 256), "query": rand(256), "x": x, "start": x[:3].contiguous(),
                     "W": rand(640, 2048).bfloat16(), "rows": rand(40 + 30 * i, 2048)})

    def once(j, r):
        u = [((7 * r + e) % 31) / 31 for e in range(5)]
        a = kb.knnssd_build_anchors(j["x"], j["start"], 20, 4)
        return (kb.knnssd_sample_token(j["p"][0], u[0]), kb.knnssd_spec_accept(j["p"], j["q"], j["drafts"], u[:4], u[4]), kb.knnssd_cosine_top1(j["query"], j["anchors"]),
                a["labels"].tolist(), a["anchors"].tolist(), a["centroids"], kb.knnssd_gemm_split(j["W"], j["rows"]))

    rounds = 12
    want = [[once(j, r) for r in range(rounds)] for j in jobs]
    got, errors = [None] * len(jobs), []
    torch.cuda.synchronize()

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                got[i] = [once(jobs[i], r) for r in range(rounds)]
                torch.cuda.current_stream().synchronize()
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for w, h in zip(want, got):
        for a, b in zip(w, h, strict=True):
            assert a[:5] == b[:5] and torch.equal(a[5], b[5]) and torch.equal(a[6], b[6])


def test_anchors_of_different_point_counts_from_several_threads(kb):
    """5 clusters of 700 .. 2600 points: the assignment takes blocks of four to eight warps with 48 to 72 KB of shared memory, by one kernel."""
    g = torch.Generator(device="cuda").manual_seed(5)
    xs = [torch.randn(n, 260, generator=g, device="cuda") for n in (700, 1000, 1500, 2000, 2300, 2600)]

    def once(x):
        a = kb.knnssd_build_anchors(x, x[:5].contiguous(), 12, 4)
        return a["labels"].tolist(), a["anchors"].tolist(), a["centroids"], a["rounds"]

    want, got, errors = [once(x) for x in xs], [[] for _ in xs], []
    torch.cuda.synchronize()

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(40):
                    got[i].append(once(xs[i]))
                torch.cuda.current_stream().synchronize()
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(xs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:2]
    for w, hs in zip(want, got):
        for h in hs:
            assert w[:2] == h[:2] and torch.equal(w[2], h[2]) and w[3] == h[3]
