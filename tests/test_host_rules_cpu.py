"""Host-side decisions of the entry points (csrc/spa_host_rules.h), compiled with the host compiler
alone: no GPU, and none of the calls that they guard."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1106_0322_gb300", "csrc")


def _run(tmp_path, body):
    """Compile and run a C++ main() of CHECK(condition) lines; a failed one is reported."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text('#include "spa_host_rules.h"\n#include <cstdio>\n#include <cstdlib>\n#include <thread>\nstatic int bad = 0;\n'
                   '#define CHECK(x) do { if (!(x)) { std::printf("%s\\n", #x); ++bad; } } while (0)\n'
                   "using namespace spa;\nint main() {\n" + body + "\nreturn bad != 0; }\n")
    subprocess.run([cxx, "-std=c++17", "-Wall", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_particles_are_read_in_place_only_inside_an_allocation_of_the_contexts_device(tmp_path):
    """Device 0 holds [4096, 4096 + 6400): 100 particles of 16 coordinates fit it exactly."""
    _run(tmp_path, """
    MemoryFacts m; m.device = true; m.ordinal = 0; m.begin = 4096; m.bytes = 6400;
    MemoryFacts other = m; other.ordinal = 1;
    MemoryFacts host = m; host.device = false;
    const MemoryFacts unknown;
    CHECK(particles_in_place(m, 0, 4096, 100, 16, 0, 0));
    CHECK(!particles_in_place(other, 0, 4096, 100, 16, 0, 0));
    CHECK(particles_in_place(other, 1, 4096, 100, 16, 0, 0));
    CHECK(!particles_in_place(host, 0, 4096, 100, 16, 0, 0));
    CHECK(!particles_in_place(unknown, 0, 4096, 100, 16, 0, 0));
    // past either end of the allocation
    CHECK(!particles_in_place(m, 0, 4096, 101, 16, 0, 0));
    CHECK(!particles_in_place(m, 0, 4112, 100, 16, 0, 0));
    CHECK(particles_in_place(m, 0, 4112, 99, 16, 0, 0));
    CHECK(!particles_in_place(m, 0, 4080, 10, 16, 0, 0));
    // 16-byte rows for p % 4 == 0, 4-byte elements otherwise
    CHECK(!particles_in_place(m, 0, 4100, 10, 16, 0, 0));
    CHECK(particles_in_place(m, 0, 4100, 10, 15, 0, 0));
    CHECK(!particles_in_place(m, 0, 4098, 10, 15, 0, 0));
    // outputs that overlap: before, across, inside, behind
    CHECK(particles_in_place(m, 0, 4896, 10, 16, 4096, 800));
    CHECK(!particles_in_place(m, 0, 4896, 10, 16, 4096, 801));
    CHECK(!particles_in_place(m, 0, 4896, 10, 16, 4900, 8));
    CHECK(!particles_in_place(m, 0, 4896, 10, 16, 5535, 8));
    CHECK(particles_in_place(m, 0, 4896, 10, 16, 5536, 8));
    """)


def test_own_stream_is_waited_for_until_the_host_has_waited_for_that_very_stream(tmp_path):
    """Handles 1 (the context's own), 2 (a configured one), 3 (a caller's)."""
    _run(tmp_path, """
    const void *own = (void*)1, *conf = (void*)2, *user = (void*)3;
    OwnStream s; s.handle = own;
    CHECK(s.holds_up(user) && !s.holds_up(own));  // nothing has waited for it yet
    s.waited_for(own);
    CHECK(!s.holds_up(user));
    // a sweep enqueued on the own stream, then a call on a configured stream that waits for that one only
    s.handed_out(own);
    s.handed_out(conf);
    s.waited_for(conf);
    CHECK(s.holds_up(user) && s.holds_up(conf));
    s.waited_for(user);
    CHECK(s.holds_up(user));
    s.waited_for(own);
    CHECK(!s.holds_up(user) && !s.holds_up(conf));
    // a call that took the stream and returned early: nobody has waited
    s.handed_out(own);
    CHECK(s.holds_up(user));
    """)


def test_every_use_of_the_contexts_stream_hands_it_out():
    """No code of the runtime reads own_stream past stream(), except to create, wait for or destroy it."""
    import re

    src = open(os.path.join(CSRC, "spa_capi.cu")).read()
    lines = [ln for ln in src.splitlines() if "own_stream" in re.sub(r"//.*", "", ln)]
    allowed = (r"cudaStream_t own_stream = nullptr", r": own_stream;", r"cudaStreamCreateWithFlags\(&c->own_stream",
               r"own\.handle = c->own_stream", r"cudaStreamSynchronize\(c->own_stream\)", r"waited_for\(c->own_stream\)",
               r"cudaStreamDestroy\(c->own_stream\)", r"launch_step_constants\(.*c->own_stream\)")
    for ln in lines:
        assert any(re.search(a, ln) for a in allowed), ln


def test_pinned_words_are_shared_by_page_given_back_and_kept_to_their_cuda_context(tmp_path):
    _run(tmp_path, """
    PinnedWords pool;
    std::vector<void*> made, freed;
    auto alloc = [&](size_t n) { made.push_back(std::aligned_alloc(4096, n)); return made.back(); };
    auto release = [&](void* p) { freed.push_back(p); };
    std::vector<uint32_t*> w;
    for (int k = 0; k < 130; ++k) w.push_back(pool.take(7, alloc));
    CHECK(made.size() == 3);  // 64 to a page
    for (size_t a = 0; a < w.size(); ++a)
        for (size_t b = 0; b < a; ++b) CHECK((w[a] > w[b] ? w[a] - w[b] : w[b] - w[a]) >= 16);
    pool.give(w[3], 7, 7, release);
    CHECK(pool.take(7, alloc) == w[3] && made.size() == 3);
    // another CUDA context never gets words of this one's pages
    uint32_t* other = pool.take(8, alloc);
    CHECK(made.size() == 4 && other == made[3]);
    // empty pages are freed, the last one kept for the next context
    for (uint32_t* x : w) pool.give(x, 7, 7, release);
    CHECK(freed.size() == 2 && pool.pages() == 2);
    CHECK(pool.take(7, alloc) && made.size() == 4);
    // given back from a thread in another CUDA context, or after a reset: nothing is freed there
    uint32_t* one = pool.take(9, alloc);
    std::vector<uint32_t*> nine;
    for (int k = 0; k < 64; ++k) nine.push_back(pool.take(9, alloc));
    for (uint32_t* x : nine) pool.give(x, 9, 8, release);
    pool.give(one, 9, 0, release);
    CHECK(freed.size() == 2);
    // no memory: no word, and nothing is kept of the attempt
    const size_t before = pool.pages();
    CHECK(pool.take(10, [](size_t) { return (void*)nullptr; }) == nullptr && pool.pages() == before);
    // two threads take and give words of one CUDA context
    auto work = [&] {
        for (int k = 0; k < 2000; ++k) {
            uint32_t* x = pool.take(11, [](size_t n) { return std::aligned_alloc(4096, n); });
            *x = (uint32_t)k;
            if (*x != (uint32_t)k) ++bad;
            pool.give(x, 11, 11, [](void* p) { std::free(p); });
        }
    };
    std::thread t1(work), t2(work);
    t1.join();
    t2.join();
    CHECK(pool.pages() == before + 1);
    """)


def test_set_config_waits_before_the_stream_changes():
    """Read from the source: the wait stands before the new configuration is taken over, and a sweep
    that is left running on a configured stream is marked by an event."""
    import re

    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "spa_capi.cu")).read())
    body = src[src.index("int spa_set_config("):src.index("int spa_get_config(")]
    assert re.search(r"if \(k->stream != c->cfg\.stream\) rc = change_stream\(c\);", body[:body.index("c->cfg = *k")])
    run = src[src.index("int spa_run_device("):src.index("int spa_sync(")]
    assert "return leave_running(" in run


def test_device_entry_points_follow_the_default_stream_when_given_its_handle():
    """Read from the source: the legacy default stream's handle is NULL, which the entry points take
    as the context's own (non-blocking) stream; each orders that behind the default stream."""
    import re

    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "spa_capi.cu")).read())
    loglik = src[src.index("static int loglik_impl("):src.index("int spa_loglik_repeat(")]
    grad = src[src.index("static int grad_impl("):src.index("int spa_grad(")]
    for body, dev in ((loglik, "B_dev"), (grad, "dev")):
        settled = body.count("rc = settle_stream(c, st);")
        assert settled >= 1
        assert len(re.findall(r"if \(rc == SPA_OK && %s && !st_user\) rc = follow_default_stream\(c, st\);" % dev,
                              body)) == settled
    run = src[src.index("static int run_common("):src.index("int spa_run(")]
    assert re.search(r"if \(sched_on_device && !c->cfg\.stream\) \{\s*rc = follow_default_stream\(c, st\);", run)
