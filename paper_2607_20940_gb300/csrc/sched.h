// Host estimate of when a launch's work ends.
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

}  // namespace msf
