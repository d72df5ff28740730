// Host rules on how a launch's work is placed.
#pragma once

namespace msf {

struct WorkUnits {
    double cost;
    long long n;
};

// End of n classes of equal units placed longest first, each on the least
// loaded of `slots` places. Places of equal load are kept together, so a call
// takes a few microseconds whatever the number of units. Sorts u.
inline double lpt_end(WorkUnits* u, int n, int slots) {
    for (int i = 0; i < n; ++i)
        for (int k = i + 1; k < n; ++k)
            if (u[k].cost > u[i].cost) {
                const WorkUnits t = u[i];
                u[i] = u[k];
                u[k] = t;
            }
    struct Level {
        double load;
        long long count;
    };
    Level lv[64] = {{0.0, slots}};  // lightest first
    int nl = 1;
    double end = 0;
    for (int i = 0; i < n; ++i) {
        long long left = u[i].n;
        while (left > 0) {
            // many rounds: whole rounds over every place keep their order
            if (left >= 4ll * slots) {
                const long long r = left / slots - 2;
                for (int k = 0; k < nl; ++k) lv[k].load += r * u[i].cost;
                left -= r * slots;
                continue;
            }
            const long long m = left < lv[0].count ? left : lv[0].count;
            const double load = lv[0].load + u[i].cost;
            left -= m;
            lv[0].count -= m;
            if (lv[0].count == 0) {
                for (int k = 1; k < nl; ++k) lv[k - 1] = lv[k];
                --nl;
            }
            int at = 0;
            while (at < nl && lv[at].load < load) ++at;
            if (at < nl && lv[at].load == load) {
                lv[at].count += m;
            } else if (nl < 64) {
                for (int k = nl; k > at; --k) lv[k] = lv[k - 1];
                lv[at] = {load, m};
                ++nl;
            } else {
                lv[at < nl ? at : nl - 1].count += m;
            }
            end = load > end ? load : end;
        }
    }
    for (int k = 0; k < nl; ++k) end = lv[k].load > end ? lv[k].load : end;
    return end;
}

// Pyramid tasks that a thread of the embedding tiles' idle warps takes: `one` on
// tiles of one K chunk, `more` on longer ones (0: the pool CTAs take them all).
struct IdleTasks {
    int one, more;
};

// A launch of `ctas` CTAs (embedding tiles and pool CTAs, two on an SM), `total`
// pool tasks, of which two and four a thread would give `two_four` to the idle
// warps and one and three `one_three`: the larger up to a quarter of all tasks,
// else the smaller up to a third, so that no tile waits for them. Where the pool
// CTAs start early anyway they only cost the tiles: so from nine CTAs an SM on, and
// from five if they take a fifth of the tasks. Over 250 launches against none: there
// 10 % faster at best, 4 % on average and at worst 2 % slower; with fewer CTAs or
// tasks, from three CTAs an SM on, 10 % faster to 19 % (2.9 us) slower.
inline IdleTasks idle_tasks(long long ctas, int sms, long long total, long long two_four, long long one_three) {
    IdleTasks t = {0, 0};
    long long share = 0;
    if (4 * two_four <= total)
        t = {2, 4}, share = two_four;
    else if (3 * one_three <= total)
        t = {1, 3}, share = one_three;
    if (ctas <= 5ll * sms || (5 * share < total && ctas <= 9ll * sms)) t = {0, 0};
    return t;
}

}  // namespace msf
