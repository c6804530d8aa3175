"""Index arithmetic and dispatch rules of the kernels, evaluated on the host."""
from host_rules import evaluate


def test_production_histogram_entries_beyond_32_bits(tmp_path):
    """accepted calls have windows of more than 2^31 entries (bin, class)"""
    cases = [(80000, 36001, 36000),   # q = 10, L = 200, one window
             (26886, 80340, 80339),   # q = 255, L = 284, 6 windows that do not overlap
             (1, 7, 3)]
    assert evaluate(tmp_path, ["heo_index(%d, %d, %d)" % c for c in cases]) == [b * n + c for b, n, c in cases]


def test_leading_words_are_shifted_by_less_than_their_width(tmp_path):
    ks = range(-200, 300)
    taken = [k for k, ok in zip(ks, evaluate(tmp_path, ["leading_words(%d)" % k for k in ks])) if ok]
    assert taken and all(0 < 58 - k < 32 for k in taken)


def test_faulting_in_a_result_buffer_keeps_what_it_holds(tmp_path):
    """a read that fails later leaves the caller's buffer as it was; every page is
    looked at once, whatever the alignment"""
    assert evaluate(tmp_path, [r"""([] {
        std::vector<unsigned char> v(9000003);
        for (size_t i = 0; i < v.size(); ++i) v[i] = (unsigned char)(i * 7 + 1);
        rewl::host::fault_in(v.data() + 1, v.size() - 1);
        rewl::host::fault_in(v.data(), 0);
        rewl::host::fault_in(v.data() + 5, 1);
        for (size_t i = 0; i < v.size(); ++i)
            if (v[i] != (unsigned char)(i * 7 + 1)) return 0;
        return 1;
    })()"""]) == [1]


def test_production_form_is_the_faster_one(tmp_path):
    """(q, L, h, W, m, walkers a CTA, CTAs per SM): the form that was measured the
    faster by a fifth or more"""
    groups = [(10, 80, 64, 766, 16, 7, 1), (10, 80, 64, 766, 256, 8, 1), (10, 300, 717, 1000, 3, 8, 1),
              (255, 80, 64, 766, 32, 8, 1), (255, 200, 200, 1578, 32, 8, 1), (80, 80, 200, 253, 64, 8, 1),
              (255, 40, 64, 191, 64, 8, 3), (30, 40, 256, 50, 256, 8, 3), (10, 40, 512, 25, 256, 8, 3),
              (255, 80, 8, 4655, 128, 4, 1), (10, 16, 100, 20, 256, 8, 3), (80, 80, 2, 10240, 256, 2, 1)]
    threads = [(255, 80, 64, 766, 256, 8, 1), (255, 80, 8, 4655, 256, 4, 1), (80, 128, 64, 1955, 256, 5, 1),
               (255, 40, 64, 191, 256, 8, 3), (80, 40, 256, 50, 256, 8, 3), (30, 80, 400, 127, 256, 8, 1),
               (255, 200, 200, 1578, 128, 8, 1), (255, 16, 100, 20, 256, 8, 3)]
    rule = ["production_lane_groups(model(%d, %d, %d, %d, %d, %d), kSms, %d, %d)"
            % (q, L, h, W, m, 4 if q <= 16 else 8, P, c) for q, L, h, W, m, P, c in groups + threads]
    assert evaluate(tmp_path, rule) == [1] * len(groups) + [0] * len(threads)


def test_narrow_lane_groups_hold_the_walkers_that_an_sm_is_given(tmp_path):
    """walkers per CTA, against what the bytes that decide which windows fit allow"""
    def granted(L, B, m_per_sm, lanes):
        al = lambda x: -(-x // 16) * 16
        n = L * L
        per = al((B + 48) * 8) + al(n // 2) + al((lanes + 8) * 16) + al((lanes + 8) * 4) + al(2 * (-(-min(n, 8192) // 32)) * 4)
        return min(232448 // per, 256 // lanes, m_per_sm)

    cases = [(L, h, W, m, lanes) for L, h, W, ms in ((80, 64, 764, (16, 32, 64, 128)), (80, 173, 291, (16, 64)),
                                                     (40, 41, 291, (64, 200)), (16, 40, 48, (64, 256)))
             for m in ms for lanes in (2, 4, 8)]
    P = evaluate(tmp_path, ["plan_sweep(model(10, %d, %d, %d, %d, 4), kSms, kShared, SWEEP_FAST, %d).P" % c for c in cases])
    for (L, h, W, m, lanes), p in zip(cases, P):
        assert p >= 0.9 * granted(L, W + 1, -(-h * m // 152), lanes), (L, h, m, lanes, p)


def test_entry_form(tmp_path):
    """(q, L, h, W, m): a thread per walker for many walkers of small lattices"""
    threads = [(10, 8, 32, 14, 256), (10, 12, 64, 17, 256), (10, 16, 96, 20, 256), (10, 24, 128, 35, 256), (10, 32, 256, 31, 256)]
    warps = [(2, 8, 4, 73, 2), (10, 16, 32, 58, 256), (10, 24, 32, 131, 256), (10, 32, 128, 62, 256), (10, 64, 512, 63, 256)]
    rule = ["init_by_threads(model(%d, %d, %d, %d, %d, 4), kSms)" % c for c in threads + warps]
    assert evaluate(tmp_path, rule) == [1] * len(threads) + [0] * len(warps)


def test_conflict_marks_of_wide_windows(tmp_path):
    """512 where ln g shadow and lattice pass 96 KB; else one per site, 8192, or 2048
    beside a lattice in global memory"""
    cases = [(80, 1, 12800, 0, 512), (200, 20, 13914, 1, 512), (78, 1, 12168, 0, 512), (91, 5, 8281, 0, 8192),
             (80, 64, 766, 0, 6400), (200, 40, 7442, 1, 2048)]
    marks = evaluate(tmp_path, ["fast_layout(model(10, %d, %d, %d, 1, 4), 32, %d).marks" % c[:4] for c in cases])
    assert marks == [c[4] for c in cases]
